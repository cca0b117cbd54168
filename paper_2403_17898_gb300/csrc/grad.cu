// Backward of the EWA projection (Sec. 3.1, Eq. 1) and of the neural-Gaussian decoders
// (Sec. 3.2, Eq. offsets and Eq. mlp), plus the L1 photometric loss and a fused Adam update.
//
// project_bwd: one thread per Gaussian; recomputes the forward quantities and chains
//   d(u, v, conic) -> d(mean, scale, unit quaternion).
// decode_bwd (FP32; decode_bwd_tc.cu has the tensor-core rows): a row pass recomputes the three decoders
//   of 64 anchors at a time by register-blocked products and produces d(feature), d(offsets), d(l_v)
//   and the rows z, h, dy, dp; a weight pass forms dY^T H and dP^T Z of the rows (staged in shared
//   memory), a 4 x 8 block of elements per thread, written as per-block partials and summed by a
//   deterministic reduction.
#include "internal.cuh"
#include "decode_bwd.cuh"
#include "tc.cuh"

namespace ogs {
namespace {

using namespace db;

constexpr int kPbThreads = 256;

struct PbArgs {
    ogs_gaussians g;
    const uint32_t* count;
    int64_t n_fixed;
    int rel;
    Cam cam;
    const uint2* rect;
    const float* drec;     // [G][9]: du dv da db dc do dr dg db
    float* dmeans;         // [G][3]
    float* dscales;        // [G][3]
    float* dquats;         // [G][4]
};

__global__ void __launch_bounds__(kPbThreads) project_bwd_kernel(PbArgs a) {
    const Cam& c = a.cam;
    const int64_t n = a.count ? (int64_t)*a.count : a.n_fixed;
    for (int64_t gi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; gi < n;
         gi += (int64_t)gridDim.x * blockDim.x) {
        float gm0 = 0.f, gm1 = 0.f, gm2 = 0.f, gs0 = 0.f, gs1 = 0.f, gs2 = 0.f;
        float gq0 = 0.f, gq1 = 0.f, gq2 = 0.f, gq3 = 0.f;
        const uint2 rc = a.rect[gi];
        const bool vis = (rc.x & 0xFFFFu) < (rc.y & 0xFFFFu);
        if (vis) {
            const float* dr = a.drec + 9 * gi;
            const float du = dr[0], dv = dr[1], dca = dr[2], dcb = dr[3], dcc = dr[4];
            float m0 = a.g.means[3 * gi], m1 = a.g.means[3 * gi + 1], m2 = a.g.means[3 * gi + 2];
            if (!a.rel) { m0 -= c.c[0]; m1 -= c.c[1]; m2 -= c.c[2]; }
            const float px = c.R[0] * m0 + c.R[1] * m1 + c.R[2] * m2;
            const float py = c.R[3] * m0 + c.R[4] * m1 + c.R[5] * m2;
            const float pz = c.R[6] * m0 + c.R[7] * m1 + c.R[8] * m2;
            const float4 q = *reinterpret_cast<const float4*>(a.g.quats + 4 * gi);
            const float s[3] = {a.g.scales[3 * gi], a.g.scales[3 * gi + 1], a.g.scales[3 * gi + 2]};
            const float w = q.x, x = q.y, y = q.z, z = q.w;
            const float Rq[9] = {1.f - 2.f * (y * y + z * z), 2.f * (x * y - w * z), 2.f * (x * z + w * y),
                                 2.f * (x * y + w * z), 1.f - 2.f * (x * x + z * z), 2.f * (y * z - w * x),
                                 2.f * (x * z - w * y), 2.f * (y * z + w * x), 1.f - 2.f * (x * x + y * y)};
            float M[9], S[9];
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int k = 0; k < 3; ++k) M[3 * r + k] = Rq[3 * r + k] * s[k];
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    S[3 * r + k] = M[3 * r] * M[3 * k] + M[3 * r + 1] * M[3 * k + 1] + M[3 * r + 2] * M[3 * k + 2];
            const float iz = 1.0f / pz;
            const float xz = px * iz, yz = py * iz;
            const bool clx = xz < -c.limx || xz > c.limx, cly = yz < -c.limy || yz > c.limy;
            const float tx = fminf(fmaxf(xz, -c.limx), c.limx) * pz;
            const float ty = fminf(fmaxf(yz, -c.limy), c.limy) * pz;
            const float J[6] = {c.fx * iz, 0.f, -c.fx * tx * iz * iz, 0.f, c.fy * iz, -c.fy * ty * iz * iz};
            float T[6];
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    T[3 * r + k] = J[3 * r] * c.R[k] + J[3 * r + 1] * c.R[3 + k] + J[3 * r + 2] * c.R[6 + k];
            float TS[6];
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    TS[3 * r + k] = T[3 * r] * S[k] + T[3 * r + 1] * S[3 + k] + T[3 * r + 2] * S[6 + k];
            const float A = TS[0] * T[0] + TS[1] * T[1] + TS[2] * T[2] + 0.3f;
            const float B = TS[0] * T[3] + TS[1] * T[4] + TS[2] * T[5];
            const float Cc = TS[3] * T[3] + TS[4] * T[4] + TS[5] * T[5] + 0.3f;
            const float id = 1.0f / (A * Cc - B * B);
            const float ka = Cc * id, kb = -B * id, kc = A * id;
            // dL/dM (M = cov2 + 0.3 I) = -K G K with G the symmetric gradient of the conic
            const float g00 = dca, g01 = 0.5f * dcb, g11 = dcc;
            const float t00 = ka * g00 + kb * g01, t01 = ka * g01 + kb * g11;
            const float t10 = kb * g00 + kc * g01, t11 = kb * g01 + kc * g11;
            const float G00 = -(t00 * ka + t01 * kb), G01 = -(t00 * kb + t01 * kc);
            const float G11 = -(t10 * kb + t11 * kc);
            const float Gm[4] = {G00, G01, G01, G11};
            // dL/dSigma = T^T Gm T ; dL/dT = 2 Gm T Sigma
            float gS[9];
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    gS[3 * r + k] = T[r] * (Gm[0] * T[k] + Gm[1] * T[3 + k]) +
                                    T[3 + r] * (Gm[2] * T[k] + Gm[3] * T[3 + k]);
            float gT[6];
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    gT[3 * r + k] = 2.f * (Gm[2 * r] * TS[k] + Gm[2 * r + 1] * TS[3 + k]);
            float gJ[6];
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    gJ[3 * r + k] = gT[3 * r] * c.R[3 * k] + gT[3 * r + 1] * c.R[3 * k + 1] +
                                    gT[3 * r + 2] * c.R[3 * k + 2];
            const float iz2 = iz * iz, iz3 = iz2 * iz;
            float gp0 = 0.f, gp1 = 0.f, gp2 = 0.f;
            gp2 += gJ[0] * (-c.fx * iz2) + gJ[4] * (-c.fy * iz2);
            if (!clx) { gp0 += gJ[2] * (-c.fx * iz2); gp2 += gJ[2] * (2.f * c.fx * px * iz3); }
            else gp2 += gJ[2] * (c.fx * (xz < 0.f ? -c.limx : c.limx) * iz2);
            if (!cly) { gp1 += gJ[5] * (-c.fy * iz2); gp2 += gJ[5] * (2.f * c.fy * py * iz3); }
            else gp2 += gJ[5] * (c.fy * (yz < 0.f ? -c.limy : c.limy) * iz2);
            gp0 += du * c.fx * iz;
            gp2 += du * (-c.fx * px * iz2);
            gp1 += dv * c.fy * iz;
            gp2 += dv * (-c.fy * py * iz2);
            gm0 = c.R[0] * gp0 + c.R[3] * gp1 + c.R[6] * gp2;
            gm1 = c.R[1] * gp0 + c.R[4] * gp1 + c.R[7] * gp2;
            gm2 = c.R[2] * gp0 + c.R[5] * gp1 + c.R[8] * gp2;
            // Sigma = M M^T, M = R(q) S:  dL/dM = 2 gS M
            float gR[9];
            float gsv[3] = {0.f, 0.f, 0.f};
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const float gM = 2.f * (gS[3 * r] * M[k] + gS[3 * r + 1] * M[3 + k] + gS[3 * r + 2] * M[6 + k]);
                    gsv[k] += gM * Rq[3 * r + k];
                    gR[3 * r + k] = gM * s[k];
                }
            gs0 = gsv[0]; gs1 = gsv[1]; gs2 = gsv[2];
            gq0 = 2.f * (-z * gR[1] + y * gR[2] + z * gR[3] - x * gR[5] - y * gR[6] + x * gR[7]);
            gq1 = 2.f * (y * gR[1] + z * gR[2] + y * gR[3] - 2.f * x * gR[4] - w * gR[5] + z * gR[6] +
                         w * gR[7] - 2.f * x * gR[8]);
            gq2 = 2.f * (-2.f * y * gR[0] + x * gR[1] + w * gR[2] + x * gR[3] + z * gR[5] - w * gR[6] +
                         z * gR[7] - 2.f * y * gR[8]);
            gq3 = 2.f * (-2.f * z * gR[0] - w * gR[1] + x * gR[2] + w * gR[3] - 2.f * z * gR[4] +
                         y * gR[5] + x * gR[6] + y * gR[7]);
        }
        a.dmeans[3 * gi] = gm0; a.dmeans[3 * gi + 1] = gm1; a.dmeans[3 * gi + 2] = gm2;
        a.dscales[3 * gi] = gs0; a.dscales[3 * gi + 1] = gs1; a.dscales[3 * gi + 2] = gs2;
        *reinterpret_cast<float4*>(a.dquats + 4 * gi) = make_float4(gq0, gq1, gq2, gq3);
    }
}

// ---------------------------------------------------------------------------------------
// decoder backward
// ---------------------------------------------------------------------------------------

// Row pass: 64 anchors at a time, the decoders recomputed and differentiated by small matrix products
// with both operands in shared memory and register blocks of outputs (as the FP32 decoder's):
//   hidden    a thread owns 4 anchors x 12 hidden units
//   outputs   4 anchors x the 11 outputs of one Gaussian slot; the thread turns them into that
//             Gaussian's dy (its gradients were loaded during the product) and its shares of doffs
//             and dlv
//   dh        4 anchors x 8 covariance or 16 opacity / colour hidden units, masked by the ReLU into dp
//   dfeat     4 anchors x 4 features
// The rows z, h, dy, dp go to scratch for the weight pass.  Each anchor appears once per view, so
// nothing needs atomics.  Products are packed over anchor pairs and summed in input order.  Bound by
// the FP32 pipes, shared-memory loads and the gathers' latency: 31k anchors 81 us, against 125 us with
// two threads per anchor (every weight read once per four products, strided gradient loads).  168
// registers with 144 bytes spilled, two CTAs per SM.
constexpr int kRowAnchors = 64;
constexpr int kRowGroups = kRowAnchors / 4;              // of four anchors
constexpr int kRowThreads = kRowGroups * kK;             // (anchor group, Gaussian slot)
constexpr int kRowHid = 12;                              // hidden units per thread
constexpr int kW2Pitch = kH + 4;                         // conflict-free by slots, 16-byte rows
static_assert(kRowThreads == 160 && kRowGroups * 8 == 128, "thread roles");

struct __align__(16) RowSmem {
    float w1[kDin + kMaxApp][3 * kH];    // transposed; rows kDin .. are the appearance weights
    float w1f[3 * kH][kF];               // W1 restricted to the features
    float w2[kNOut][kW2Pitch];           // stacked second layers
    float b1[3 * kH];
    float b2[kNOut + 2];
    float h[3 * kH][kRowAnchors];        // hidden activations, then dp
    float d[kNOut + 3 * kK][kRowAnchors];    // inputs z, then dy and the shares of dlv
    float rows[kRowAnchors][8];          // anchor index, weight, l_v
};
static_assert(kDin + kMaxApp <= kNOut, "z fits under dy");
static_assert(sizeof(RowSmem) <= 112 * 1024, "two CTAs per SM");

// dh of kN hidden units from h0 (decoder rows row0 .. row0 + nrows of W2 and dy) for anchor group
// ag, through the ReLU; dp replaces h and goes to the rows.
template <int kN>
__device__ __forceinline__ void dh_block(RowSmem& s, const DbArgs& a, int ag, int h0, int row0,
                                         int nrows, uint32_t base, uint32_t M) {
    const int hl = h0 % kH;
    f32x2 acc[kN][2];
#pragma unroll
    for (int o = 0; o < kN; ++o) acc[o][0] = acc[o][1] = 0;
#pragma unroll 2
    for (int k = 0; k < nrows; ++k) {
        const float4 d = *reinterpret_cast<const float4*>(&s.d[row0 + k][4 * ag]);
        const f32x2 d0 = pack2(d.x, d.y), d1 = pack2(d.z, d.w);
#pragma unroll
        for (int q = 0; q < kN / 4; ++q) {
            const float4 w = *reinterpret_cast<const float4*>(&s.w2[row0 + k][hl + 4 * q]);
            const float wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const f32x2 w2 = pack2(wv[u], wv[u]);
                acc[4 * q + u][0] = fma2(w2, d0, acc[4 * q + u][0]);
                acc[4 * q + u][1] = fma2(w2, d1, acc[4 * q + u][1]);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < kN / 4; ++q) {
        float dp[4][4];                                  // [hidden][anchor]
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            float* hp = &s.h[h0 + 4 * q + u][4 * ag];
            const float4 h = *reinterpret_cast<const float4*>(hp);
            dp[u][0] = h.x > 0.f ? lo2(acc[4 * q + u][0]) : 0.f;
            dp[u][1] = h.y > 0.f ? hi2(acc[4 * q + u][0]) : 0.f;
            dp[u][2] = h.z > 0.f ? lo2(acc[4 * q + u][1]) : 0.f;
            dp[u][3] = h.w > 0.f ? hi2(acc[4 * q + u][1]) : 0.f;
            *reinterpret_cast<float4*>(hp) = make_float4(dp[u][0], dp[u][1], dp[u][2], dp[u][3]);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r)
            if (base + 4 * ag + r < M)
                *reinterpret_cast<float4*>(a.rowP + (size_t)(base + 4 * ag + r) * kRowP + h0 + 4 * q) =
                    make_float4(dp[0][r], dp[1][r], dp[2][r], dp[3][r]);
    }
}

template <bool APP>
__global__ void __launch_bounds__(kRowThreads, 2) decode_bwd_rows(DbArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    RowSmem& s = *reinterpret_cast<RowSmem*>(smem_raw);
    const uint32_t M = a.counts->n_selected;
    const uint32_t ntiles = (M + kRowAnchors - 1) / kRowAnchors;
    if (blockIdx.x >= ntiles) return;
    const int t = threadIdx.x, napp = a.mlp.A;
#pragma unroll 8
    for (int e = t; e < kDin * 3 * kH; e += kRowThreads) {
        const int i = e / (3 * kH), o = e % (3 * kH);
        const float v = a.mlp.w1[o * kDin + i];
        s.w1[i][o] = v;
        if (i < kF) s.w1f[o][i] = v;
    }
    if (APP) {
        for (int e = t; e < kMaxApp * kH; e += kRowThreads) {
            const int q = e / kH, o = e % kH;
            s.w1[kDin + q][kH + o] = q < napp ? a.mlp.w1_app[o * napp + q] : 0.f;
        }
    }
#pragma unroll 8
    for (int e = t; e < kNOut * kH; e += kRowThreads)
        s.w2[e / kH][e % kH] = e < kK * kH ? a.mlp.w2_op[e]
                                           : (e < 4 * kK * kH ? a.mlp.w2_col[e - kK * kH]
                                                              : a.mlp.w2_cov[e - 4 * kK * kH]);
    for (int e = t; e < kNB1; e += kRowThreads) s.b1[e] = a.mlp.b1[e];
    for (int e = t; e < kNOut; e += kRowThreads)
        s.b2[e] = e < kK ? a.mlp.b2_op[e] : (e < 4 * kK ? a.mlp.b2_col[e - kK] : a.mlp.b2_cov[e - 4 * kK]);
    const Cam& c = a.cam;
    for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const uint32_t base = tile * kRowAnchors;
        // gather: two threads per anchor, inputs transposed and as rows
        if (t < 2 * kRowAnchors) {
            const int al = t % kRowAnchors, half = t / kRowAnchors;
            const uint32_t r = base + al;
            const bool valid = r < M;
            const uint32_t j = valid ? a.sel_idx[r] : 0u;
            float4 v[4];
            const float4* f4 = reinterpret_cast<const float4*>(a.feat + (size_t)j * kF) + 4 * half;
            float4* zr = reinterpret_cast<float4*>(a.rowZ + (size_t)r * kRowZ);
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = valid ? f4[i] : make_float4(0.f, 0.f, 0.f, 0.f);
            if (half == 0) {
                float dv[3] = {0.f, 0.f, 0.f}, lv[3] = {0.f, 0.f, 0.f}, d = 1.f, w = 0.f;
                if (valid) {
                    w = a.sel_w[r];
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        dv[q] = a.pos[3 * (size_t)j + q] - c.c[q];
                        lv[q] = a.lv[3 * (size_t)j + q];
                    }
                    d = sqrtf(dv[0] * dv[0] + dv[1] * dv[1] + dv[2] * dv[2]);
                    zr[kF / 4] = make_float4(dv[0] / d, dv[1] / d, dv[2] / d, d);
                    zr[kF / 4 + 1] = make_float4(0.f, 0.f, 0.f, 0.f);
                }
#pragma unroll
                for (int q = 0; q < 3; ++q) s.d[kF + q][al] = dv[q] / d;
                s.d[kF + 3][al] = d;
                float* rw = s.rows[al];
                rw[0] = __uint_as_float(j);
                rw[1] = w;
                rw[2] = lv[0]; rw[3] = lv[1]; rw[4] = lv[2];
            } else if (APP) {
#pragma unroll
                for (int q = 0; q < kMaxApp; ++q)
                    s.d[kDin + q][al] = valid && q < napp ? a.mlp.app[(size_t)j * napp + q] : 0.f;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (valid) zr[4 * half + i] = v[i];
                const int k = 16 * half + 4 * i;
                s.d[k][al] = v[i].x;
                s.d[k + 1][al] = v[i].y;
                s.d[k + 2][al] = v[i].z;
                s.d[k + 3][al] = v[i].w;
            }
        }
        __syncthreads();
        if (t < 128) {                                   // hidden units
            const int ag = t % kRowGroups, o0 = t / kRowGroups * kRowHid;
            f32x2 acc[kRowHid][2];
#pragma unroll
            for (int o = 0; o < kRowHid; ++o) acc[o][0] = acc[o][1] = pack2(s.b1[o0 + o], s.b1[o0 + o]);
#pragma unroll 4
            for (int k = 0; k < kDin; ++k) {
                const float4 z = *reinterpret_cast<const float4*>(&s.d[k][4 * ag]);
                const f32x2 z0 = pack2(z.x, z.y), z1 = pack2(z.z, z.w);
#pragma unroll
                for (int q = 0; q < kRowHid / 4; ++q) {
                    const float4 w = *reinterpret_cast<const float4*>(&s.w1[k][o0 + 4 * q]);
                    const float wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const f32x2 w2 = pack2(wv[u], wv[u]);
                        acc[4 * q + u][0] = fma2(w2, z0, acc[4 * q + u][0]);
                        acc[4 * q + u][1] = fma2(w2, z1, acc[4 * q + u][1]);
                    }
                }
            }
            if (APP) {                                   // the colour decoder also sees the code
#pragma unroll 1
                for (int k = kDin; k < kDin + kMaxApp; ++k) {
                    const float4 z = *reinterpret_cast<const float4*>(&s.d[k][4 * ag]);
                    const f32x2 z0 = pack2(z.x, z.y), z1 = pack2(z.z, z.w);
#pragma unroll
                    for (int o = 0; o < kRowHid; ++o) {
                        if (o0 + o < kH || o0 + o >= 2 * kH) continue;
                        const f32x2 w2 = pack2(s.w1[k][o0 + o], s.w1[k][o0 + o]);
                        acc[o][0] = fma2(w2, z0, acc[o][0]);
                        acc[o][1] = fma2(w2, z1, acc[o][1]);
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < kRowHid / 4; ++q) {
                float h[4][4];                           // [hidden][anchor]
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const f32x2* p = acc[4 * q + u];
                    h[u][0] = fmaxf(lo2(p[0]), 0.f); h[u][1] = fmaxf(hi2(p[0]), 0.f);
                    h[u][2] = fmaxf(lo2(p[1]), 0.f); h[u][3] = fmaxf(hi2(p[1]), 0.f);
                    *reinterpret_cast<float4*>(&s.h[o0 + 4 * q + u][4 * ag]) =
                        make_float4(h[u][0], h[u][1], h[u][2], h[u][3]);
                }
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    if (base + 4 * ag + r < M)
                        *reinterpret_cast<float4*>(a.rowH + (size_t)(base + 4 * ag + r) * kRowH + o0 + 4 * q) =
                            make_float4(h[0][r], h[1][r], h[2][r], h[3][r]);
            }
        }
        __syncthreads();
        {                                                // outputs -> dy of one Gaussian slot
            const int i = t % kK, ag = t / kK;
            const int row1 = kK + 3 * i, row2 = 4 * kK + 7 * i;
            GaussGrad gg[4];                             // in flight during the product
            float O[4][3], dO[4][3];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t r = base + 4 * ag + q;
                if (r < M) {
                    gg[q] = load_gauss_grad(a, (size_t)r * kK + i);
                    const size_t o = ((size_t)__float_as_uint(s.rows[4 * ag + q][0]) * kK + i) * 3;
#pragma unroll
                    for (int e = 0; e < 3; ++e) {
                        O[q][e] = a.offs[o + e];
                        dO[q][e] = a.doffs[o + e];
                    }
                }
            }
            f32x2 acc[11][2];
#pragma unroll
            for (int e = 0; e < 11; ++e) {
                const float b = s.b2[e == 0 ? i : (e < 4 ? row1 + e - 1 : row2 + e - 4)];
                acc[e][0] = acc[e][1] = pack2(b, b);
            }
#pragma unroll 2
            for (int o = 0; o < kH; ++o) {
#pragma unroll
                for (int m = 0; m < 3; ++m) {
                    const float4 h = *reinterpret_cast<const float4*>(&s.h[m * kH + o][4 * ag]);
                    const f32x2 h0 = pack2(h.x, h.y), h1 = pack2(h.z, h.w);
#pragma unroll
                    for (int e = m == 0 ? 0 : (m == 1 ? 1 : 4); e < (m == 0 ? 1 : (m == 1 ? 4 : 11)); ++e) {
                        const float w = s.w2[e == 0 ? i : (e < 4 ? row1 + e - 1 : row2 + e - 4)][o];
                        acc[e][0] = fma2(pack2(w, w), h0, acc[e][0]);
                        acc[e][1] = fma2(pack2(w, w), h1, acc[e][1]);
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int al = 4 * ag + q;
                const uint32_t r = base + al;
                float dy[11], dlv[3] = {0.f, 0.f, 0.f};
#pragma unroll
                for (int e = 0; e < 11; ++e) dy[e] = 0.f;
                if (r < M) {
                    float y[11];
#pragma unroll
                    for (int e = 0; e < 11; ++e) y[e] = q & 1 ? hi2(acc[e][q / 2]) : lo2(acc[e][q / 2]);
                    const float* rw = s.rows[al];
                    const float lvv[3] = {rw[2], rw[3], rw[4]};
                    dy_opacity(gg[q], rw[1], y, dy);
                    dy_color(gg[q], y + 1, dy + 1);
                    dy_cov(gg[q], lvv, y + 4, dy + 4, dlv);
                    // positions: mu = x_v + O * l_v
                    float* dof = a.doffs + ((size_t)__float_as_uint(rw[0]) * kK + i) * 3;
#pragma unroll
                    for (int e = 0; e < 3; ++e) {
                        dof[e] = fmaf(gg[q].mean[e], lvv[e], dO[q][e]);
                        dlv[e] = fmaf(gg[q].mean[e], O[q][e], dlv[e]);
                    }
                    float* yr = a.rowY + (size_t)r * kRowY;
                    yr[i] = dy[0];
#pragma unroll
                    for (int e = 0; e < 3; ++e) yr[kRowCol + 3 * i + e] = dy[1 + e];
#pragma unroll
                    for (int e = 0; e < 7; ++e) yr[kRowCov + 7 * i + e] = dy[4 + e];
                    if (i == 0) {
#pragma unroll
                        for (int e = 0; e < kRowY; ++e)
                            if (row_out(e) < 0) yr[e] = 0.f;
                    }
                }
                s.d[i][al] = dy[0];
#pragma unroll
                for (int e = 0; e < 3; ++e) {
                    s.d[row1 + e][al] = dy[1 + e];
                    s.d[kNOut + 3 * i + e][al] = dlv[e];
                }
#pragma unroll
                for (int e = 0; e < 7; ++e) s.d[row2 + e][al] = dy[4 + e];
            }
        }
        __syncthreads();
        // hidden gradients: 64 threads on the covariance decoder, 32 on each other one
        {
            const int ag = t % kRowGroups, hg = t / kRowGroups;
            if (hg < 4) dh_block<8>(s, a, ag, 2 * kH + 8 * hg, 4 * kK, 7 * kK, base, M);
            else if (hg < 6) dh_block<16>(s, a, ag, kH + 16 * (hg - 4), kK, 3 * kK, base, M);
            else if (hg < 8) dh_block<16>(s, a, ag, 16 * (hg - 6), 0, kK, base, M);
            else
                for (int e = t - 128; e < 3 * kRowAnchors; e += kRowThreads - 128) {
                    const int al = e % kRowAnchors, q = e / kRowAnchors;     // l_v gradients
                    if (base + al < M) {
                        float v = 0.f;
#pragma unroll
                        for (int i = 0; i < kK; ++i) v += s.d[kNOut + 3 * i + q][al];
                        a.dlv[3 * (size_t)__float_as_uint(s.rows[al][0]) + q] += v;
                    }
                }
        }
        __syncthreads();
        if (t < 128) {                                   // features: opacity and colour, then covariance
            const int ag = t % kRowGroups, i0 = t / kRowGroups * 4;
            float4 df[4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (base + 4 * ag + q < M)
                    df[q] = *reinterpret_cast<const float4*>(
                        a.dfeat + (size_t)__float_as_uint(s.rows[4 * ag + q][0]) * kF + i0);
            f32x2 acc[2][4][2];
#pragma unroll
            for (int m = 0; m < 2; ++m) {
#pragma unroll
                for (int u = 0; u < 4; ++u) acc[m][u][0] = acc[m][u][1] = 0;
#pragma unroll 4
                for (int o = m ? 2 * kH : 0; o < (m ? 3 * kH : 2 * kH); ++o) {
                    const float4 d = *reinterpret_cast<const float4*>(&s.h[o][4 * ag]);
                    const float4 w = *reinterpret_cast<const float4*>(&s.w1f[o][i0]);
                    const f32x2 d0 = pack2(d.x, d.y), d1 = pack2(d.z, d.w);
                    const float wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        acc[m][u][0] = fma2(pack2(wv[u], wv[u]), d0, acc[m][u][0]);
                        acc[m][u][1] = fma2(pack2(wv[u], wv[u]), d1, acc[m][u][1]);
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (base + 4 * ag + q < M) {
                    float g[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const f32x2 v = add2(acc[0][u][q / 2], acc[1][u][q / 2]);
                        g[u] = q & 1 ? hi2(v) : lo2(v);
                    }
                    *reinterpret_cast<float4*>(
                        a.dfeat + (size_t)__float_as_uint(s.rows[4 * ag + q][0]) * kF + i0) =
                        make_float4(df[q].x + g[0], df[q].y + g[1], df[q].z + g[2], df[q].w + g[3]);
                }
            }
        }
        if (APP) {                                       // code gradient: dapp_c += sum_o Wa[o][c] dp_o
            for (int e = t; e < kRowAnchors * kMaxApp; e += kRowThreads) {
                const int al = e % kRowAnchors, q = e / kRowAnchors;
                if (q < napp && base + al < M) {
                    float v = 0.f;
#pragma unroll
                    for (int o = 0; o < kH; ++o) v = fmaf(s.w1[kDin + q][kH + o], s.h[kH + o][al], v);
                    a.dapp[(size_t)__float_as_uint(s.rows[al][0]) * napp + q] += v;
                }
            }
        }
        __syncthreads();                                 // everything is rewritten by the next tile
    }
}

// Weight pass: dW2 = dY^T H (block-diagonal), dW1 = dP^T Z, db2 = sum dY, db1 = sum dP over
// the selected anchors.  Split over anchors: each CTA stages chunks of kWChunk rows in shared
// memory (double-buffered bulk copies) and accumulates fixed 4 x 8 blocks of outputs in
// registers; its totals go to its partial row, summed across CTAs in a fixed order.
// Bound by the FP32 pipes and the rows' HBM reads (1376 B per anchor).  A thread's block takes
// three 16-byte shared loads for 32 products (packed FP32 pairs), where the earlier 1 x 4 items
// took two loads for four and waited on shared memory three cycles in four: 100k anchors
// 128 -> 49 us; same summation order, same bits.
constexpr int kWThreads = 256;
constexpr int kWChunk = 32;
constexpr int kTilesW2 = kRowY / 4 * (kH / 8);           // 3 + 8 + 18 row groups of 4, 8 columns
constexpr int kTilesW1 = (3 * kH / 8) * (kDin / 4);       // 8 rows, 4 columns
constexpr int kTiles = kTilesW2 + kTilesW1;               // 224: the last warp sums the biases
constexpr int kItems1 = kNOut + kNB1;                     // 206 bias sums
constexpr int kBiasThreads = kWThreads - kTiles;
static_assert(kTiles % 32 == 0 && kBiasThreads > 0, "whole warps per role");
static_assert(kH == 32 && kDin == 36 && kRowCol == 12 && kRowCov == 44 && kRowY == 116,
              "block layout of the weight gradients");

// Block of the weight gradients owned by thread t < kTiles: four values a and eight values b of
// an anchor's rows, out[i][j] = sum a_i b_j.  dW2 blocks: a = dy rows row .. row + 3, b = hidden
// columns col .. col + 7 of its decoder dec (sums over a row's padding are not written).  dW1
// blocks: a = inputs col .. col + 3, b = dp rows row .. row + 7.
struct WBlock {
    bool w2;
    int row, col, dec;
};

__device__ __forceinline__ WBlock weight_block(int t) {
    WBlock b;
    b.w2 = t < kTilesW2;
    if (b.w2) {
        const int rg = t / (kH / 8);
        b.dec = rg < 3 ? 0 : (rg < 11 ? 1 : 2);
        b.row = 4 * rg;
        b.col = 8 * (t % (kH / 8));
    } else {
        const int i = t - kTilesW2;
        b.dec = 0;
        b.row = 8 * (i / (kDin / 4));
        b.col = 4 * (i % (kDin / 4));
    }
    return b;
}

// Shared-memory stage of one chunk: the four row arrays back to back, each [kWChunk][row].
constexpr int kWStageFloats = kWChunk * (kRowY + kRowH + kRowP + kRowZ);
constexpr int kWSmemBytes = 2 * kWStageFloats * (int)sizeof(float);
constexpr uint32_t kWWaitLimit = 1u << 24;

// Bulk copies of chunk ch's rows (the first nv of them; every row is a multiple of 16 bytes and
// the arrays start 256-byte aligned) into stage `st`, completing on mbar.
__device__ __forceinline__ void weights_issue(const DbArgs& a, float* stage, uint32_t ch,
                                              uint32_t M, uint64_t* mbar) {
    const uint32_t r0 = ch * kWChunk;
    const uint32_t nv = min((uint32_t)kWChunk, M - r0);
    tc::mbar_expect_tx(mbar, nv * 4u * (kRowY + kRowH + kRowP + kRowZ));
    tc::bulk_load(stage, a.rowY + (size_t)r0 * kRowY, nv * 4u * kRowY, mbar);
    tc::bulk_load(stage + kWChunk * kRowY, a.rowH + (size_t)r0 * kRowH, nv * 4u * kRowH, mbar);
    tc::bulk_load(stage + kWChunk * (kRowY + kRowH), a.rowP + (size_t)r0 * kRowP,
                  nv * 4u * kRowP, mbar);
    tc::bulk_load(stage + kWChunk * (kRowY + kRowH + kRowP), a.rowZ + (size_t)r0 * kRowZ,
                  nv * 4u * kRowZ, mbar);
}

// The chunks arrive by bulk copies into two shared-memory stages: the copy of a CTA's next
// chunk is issued before its current one is summed (the other stage was released by the
// barrier that ended the previous chunk), so the CTA's loads overlap its arithmetic.
__global__ void __launch_bounds__(kWThreads) decode_bwd_weights(DbArgs a) {
    extern __shared__ __align__(16) float s_w[];
    __shared__ __align__(8) uint64_t mbar[2];
    const uint32_t M = a.counts->n_selected;
    const int t = threadIdx.x;
    const bool tile = t < kTiles;
    const WBlock wb = weight_block(tile ? t : 0);
    // offsets of a and b inside a stage, and their row pitches
    const int pitch_a = wb.w2 ? kRowY : kRowZ, pitch_b = wb.w2 ? kRowH : kRowP;
    const int off_a = wb.w2 ? wb.row : kWChunk * (kRowY + kRowH + kRowP) + wb.col;
    const int off_b = wb.w2 ? kWChunk * kRowY + wb.dec * kH + wb.col
                            : kWChunk * (kRowY + kRowH) + wb.row;
    f32x2 acc[4][4];                          // [a][pairs of b]
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0;
    float acc1[(kItems1 + kBiasThreads - 1) / kBiasThreads] = {};
    const uint32_t nchunks = (M + kWChunk - 1) / kWChunk;
    if (t == 0) {
        tc::mbar_init(&mbar[0], 1);
        tc::mbar_init(&mbar[1], 1);
        if (blockIdx.x < nchunks) weights_issue(a, s_w, blockIdx.x, M, &mbar[0]);
    }
    __syncthreads();
    bool timed_out = false;
    uint32_t i = 0;
    for (uint32_t ch = blockIdx.x; ch < nchunks; ch += gridDim.x, ++i) {
        const uint32_t st = i & 1u;
        float* stage = s_w + st * kWStageFloats;
        if (t == 0 && ch + gridDim.x < nchunks)
            weights_issue(a, s_w + (st ^ 1u) * kWStageFloats, ch + gridDim.x, M, &mbar[st ^ 1u]);
        if (!tc::mbar_wait(&mbar[st], (i >> 1) & 1u, kWWaitLimit)) {
            timed_out = true;
            // the copies may still be landing: wait for them (bounded) before moving on
            tc::mbar_wait(&mbar[st], (i >> 1) & 1u, kWWaitLimit);
        }
        const int nv = (int)min((uint32_t)kWChunk, M - ch * kWChunk);
        float(*sY)[kRowY] = reinterpret_cast<float(*)[kRowY]>(stage);
        float(*sH)[kRowH] = reinterpret_cast<float(*)[kRowH]>(stage + kWChunk * kRowY);
        float(*sP)[kRowP] = reinterpret_cast<float(*)[kRowP]>(stage + kWChunk * (kRowY + kRowH));
        float(*sZ)[kRowZ] =
            reinterpret_cast<float(*)[kRowZ]>(stage + kWChunk * (kRowY + kRowH + kRowP));
        if (nv < kWChunk) {                   // the last, partial chunk: zero the rows past it
            for (int e = t; e < (kWChunk - nv) * kRowY; e += kWThreads) sY[nv + e / kRowY][e % kRowY] = 0.f;
            for (int e = t; e < (kWChunk - nv) * kRowH; e += kWThreads) {
                sH[nv + e / kRowH][e % kRowH] = 0.f;
                sP[nv + e / kRowP][e % kRowP] = 0.f;
            }
            for (int e = t; e < (kWChunk - nv) * kRowZ; e += kWThreads) sZ[nv + e / kRowZ][e % kRowZ] = 0.f;
            __syncthreads();
        }
        if (tile) {
            const float* pa = stage + off_a;
            const float* pb = stage + off_b;
#pragma unroll 8
            for (int k = 0; k < kWChunk; ++k) {
                const float4 a = *reinterpret_cast<const float4*>(pa + k * pitch_a);
                const float4 b0 = *reinterpret_cast<const float4*>(pb + k * pitch_b);
                const float4 b1 = *reinterpret_cast<const float4*>(pb + k * pitch_b + 4);
                const float av[4] = {a.x, a.y, a.z, a.w};
                const f32x2 bv[4] = {pack2(b0.x, b0.y), pack2(b0.z, b0.w), pack2(b1.x, b1.y),
                                     pack2(b1.z, b1.w)};
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        acc[i][j] = fma2(pack2(av[i], av[i]), bv[j], acc[i][j]);
            }
        } else {
#pragma unroll
            for (int q = 0; q < (int)(sizeof(acc1) / sizeof(float)); ++q) {
                const int item = t - kTiles + q * kBiasThreads;
                float s = 0.f;
                if (item < kNOut) {
#pragma unroll 8
                    for (int k = 0; k < kWChunk; ++k) s += sY[k][out_row(item)];
                } else if (item < kItems1) {
#pragma unroll 8
                    for (int k = 0; k < kWChunk; ++k) s += sP[k][item - kNOut];
                }
                acc1[q] += s;
            }
        }
        __syncthreads();                      // this stage is free for the copy after next
    }
    if (timed_out && t == 0) atomicExch(const_cast<uint32_t*>(&a.counts->timeout), 1u);
    // this CTA's totals -> its partial row (flat layout of the decoder gradients)
    float* out = a.partial + (size_t)blockIdx.x * kNWeights;
    if (tile) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float v = j & 1 ? hi2(acc[i][j / 2]) : lo2(acc[i][j / 2]);
                if (wb.w2) {
                    const int row = row_out(wb.row + i);
                    if (row >= 0) out[kOffW2 + row * kH + wb.col + j] = v;
                } else {
                    out[(wb.row + j) * kDin + wb.col + i] = v;
                }
            }
        }
    } else {
#pragma unroll
        for (int q = 0; q < (int)(sizeof(acc1) / sizeof(float)); ++q) {
            const int item = t - kTiles + q * kBiasThreads;
            if (item < kNOut) out[kOffB2 + item] = acc1[q];
            else if (item < kItems1) out[kOffB1 + (item - kNOut)] = acc1[q];
        }
    }
}

// Appearance weight gradients (Sec. 4.4): dWa[o][c] = sum over the selected anchors of the
// colour decoder's pre-activation gradient dp_o (rowP columns 32..63) times the anchor's code
// value c.  Thread (o, c) of each CTA accumulates over chunks of kWChunk rows staged in shared
// memory; its total goes to the CTA's partial row, summed across CTAs by reduce_app in a
// fixed order.
static_assert(kWChunk * kMaxApp == kAppItems, "one code value staged per thread");

__global__ void __launch_bounds__(kAppItems) decode_bwd_app_weights(DbArgs a,
                                                                    float* __restrict__ part) {
    __shared__ float sP[kWChunk][kH + 1];
    __shared__ float sC[kWChunk][kMaxApp];
    const uint32_t M = a.counts->n_selected;
    const int t = threadIdx.x, o = t / kMaxApp, q = t % kMaxApp;
    const int napp = a.mlp.A;
    float acc = 0.f;
    const uint32_t nchunks = (M + kWChunk - 1) / kWChunk;
    for (uint32_t ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
        const uint32_t r0 = ch * kWChunk;
        const int nv = (int)min((uint32_t)kWChunk, M - r0);
        __syncthreads();
        for (int e = t; e < kWChunk * kH; e += kAppItems) {
            const int k = e / kH, h = e % kH;
            sP[k][h] = k < nv ? a.rowP[(size_t)(r0 + k) * kRowP + kH + h] : 0.f;
        }
        {
            const int k = t / kMaxApp, c = t % kMaxApp;
            sC[k][c] = (k < nv && c < napp) ? a.mlp.app[(size_t)a.sel_idx[r0 + k] * napp + c] : 0.f;
        }
        __syncthreads();
#pragma unroll 8
        for (int k = 0; k < kWChunk; ++k) acc = fmaf(sP[k][o], sC[k][q], acc);
    }
    part[(size_t)blockIdx.x * kAppItems + t] = acc;
}

// dw1_app[o][c] += sum over blocks of part[b][o * kMaxApp + c] (fixed order, c < A).
__global__ void __launch_bounds__(kAppItems) reduce_app(const float* __restrict__ part,
                                                        int nblocks, float* dw1_app, int napp) {
    const int t = threadIdx.x, o = t / kMaxApp, q = t % kMaxApp;
    float s = 0.f;
#pragma unroll 8
    for (int b = 0; b < nblocks; ++b) s += part[(size_t)b * kAppItems + t];
    if (q < napp) dw1_app[o * napp + q] += s;
}

// dmlp[e] += sum over blocks of partial[b][e].  A CTA owns 32 consecutive outputs (one per
// lane, coalesced reads); its 8 warps sum interleaved blocks, then warp 0 adds the 8 warp
// sums in a fixed order: deterministic.  Latency-bound (8.7 MB out of L2): a warp's loads are
// issued 19 at a time, 9.3 -> 5.6 us.
constexpr int kRedWarps = 8;
static_assert(kDbBlocks % kRedWarps == 0, "every warp sums as many blocks");

__device__ __forceinline__ float* grad_slot(const ogs_mlp& grads, int e) {
    int i = e;
    if (i < kNW1) return const_cast<float*>(grads.w1) + i;
    if ((i -= kNW1) < kNB1) return const_cast<float*>(grads.b1) + i;
    if ((i -= kNB1) < kK * kH) return const_cast<float*>(grads.w2_op) + i;
    if ((i -= kK * kH) < 3 * kK * kH) return const_cast<float*>(grads.w2_col) + i;
    if ((i -= 3 * kK * kH) < 7 * kK * kH) return const_cast<float*>(grads.w2_cov) + i;
    if ((i -= 7 * kK * kH) < kK) return const_cast<float*>(grads.b2_op) + i;
    if ((i -= kK) < 3 * kK) return const_cast<float*>(grads.b2_col) + i;
    return const_cast<float*>(grads.b2_cov) + (i - 3 * kK);
}

__global__ void __launch_bounds__(32 * kRedWarps) reduce_partials(const float* __restrict__ partial,
                                                                  ogs_mlp grads) {
    __shared__ float s[kRedWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int e = blockIdx.x * 32 + lane;
    float acc = 0.f;
    if (e < kNWeights) {
#pragma unroll 19
        for (int b = 0; b < kDbBlocks / kRedWarps; ++b)
            acc += partial[(size_t)(warp + b * kRedWarps) * kNWeights + e];
    }
    s[warp][lane] = acc;
    __syncthreads();
    if (warp == 0 && e < kNWeights) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < kRedWarps; ++w) t += s[w][lane];
        *grad_slot(grads, e) += t;
    }
}

// ---------------------------------------------------------------------------------------
// loss and optimiser
// ---------------------------------------------------------------------------------------

// L = mean |img - target|; dimg = sign(img - target) / n; loss accumulated into *loss
__global__ void l1_kernel(const float* __restrict__ img, const float* __restrict__ target,
                          int64_t n, float scale, float* __restrict__ dimg,
                          float* __restrict__ loss) {
    float s = 0.f;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const float d = img[i] - target[i];
        s += fabsf(d);
        dimg[i] = d > 0.f ? scale : (d < 0.f ? -scale : 0.f);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane_id() == 0 && loss) atomicAdd(loss, s * scale);
}

// x *= *s (the chain-rule factor that a loss's backward receives)
__global__ void scale_kernel(float* __restrict__ x, int64_t n, const float* __restrict__ s) {
    const float f = *s;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        x[i] *= f;
}

// One parameter: m, v moments; step lr * m_hat / (sqrt(v_hat) + eps) with the bias
// corrections folded into reciprocals (ibc1 = 1/(1 - b1^t), ibc2 = 1/(1 - b2^t)) and one
// fast division, so the update costs a handful of instructions and the kernel stays
// memory-bound.
__device__ __forceinline__ void adam_one(float& p, float& g, float& m, float& v, float lr,
                                         float b1, float b2, float eps, float ibc1, float ibc2,
                                         int zero_grad) {
    m = fmaf(b1, m, (1.f - b1) * g);
    v = fmaf(b2, v, (1.f - b2) * g * g);
    p -= __fdividef(lr * ibc1 * m, __fsqrt_rn(v * ibc2) + eps);
    if (zero_grad) g = 0.f;
}

// Streaming update: 16-byte vectors when all four arrays are 16-byte aligned (n/4 vectors
// plus a scalar tail), scalars otherwise.  HBM-bound: 16 B read + 12 B written per parameter
// (+4 B for the gradients that were nonzero, cleared with zero_grad).
__global__ void __launch_bounds__(256) adam_kernel(float* __restrict__ p, float* __restrict__ grad,
                                                   float* __restrict__ m, float* __restrict__ v,
                                                   int64_t n, float lr, float b1, float b2,
                                                   float eps, float ibc1, float ibc2,
                                                   int zero_grad, int vec) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int64_t first = 0;
    if (vec) {
        const int64_t n4 = n / 4;
        float4* p4 = reinterpret_cast<float4*>(p);
        float4* g4 = reinterpret_cast<float4*>(grad);
        float4* m4 = reinterpret_cast<float4*>(m);
        float4* v4 = reinterpret_cast<float4*>(v);
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
            float4 P = p4[i], G = g4[i], M = m4[i], V = v4[i];
            // most anchors get no gradient in a step: clear only vectors that hold one
            const bool touched = G.x != 0.f || G.y != 0.f || G.z != 0.f || G.w != 0.f;
            adam_one(P.x, G.x, M.x, V.x, lr, b1, b2, eps, ibc1, ibc2, zero_grad);
            adam_one(P.y, G.y, M.y, V.y, lr, b1, b2, eps, ibc1, ibc2, zero_grad);
            adam_one(P.z, G.z, M.z, V.z, lr, b1, b2, eps, ibc1, ibc2, zero_grad);
            adam_one(P.w, G.w, M.w, V.w, lr, b1, b2, eps, ibc1, ibc2, zero_grad);
            p4[i] = P; m4[i] = M; v4[i] = V;
            if (zero_grad && touched) g4[i] = G;
        }
        first = 4 * n4;
    }
    for (int64_t i = first + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        float P = p[i], G = grad[i], M = m[i], V = v[i];
        adam_one(P, G, M, V, lr, b1, b2, eps, ibc1, ibc2, zero_grad);
        p[i] = P; m[i] = M; v[i] = V;
        if (zero_grad) grad[i] = G;
    }
}

}  // namespace

cudaError_t db::launch_weight_pass(const DbArgs& a, const DbScratch& s, const ogs_mlp& dmlp,
                                   cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(decode_bwd_weights,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, kWSmemBytes);
    if (e != cudaSuccess) return e;
    decode_bwd_weights<<<kDbBlocks, kWThreads, kWSmemBytes, st>>>(a);
    reduce_partials<<<(kNWeights + 31) / 32, 32 * kRedWarps, 0, st>>>(s.partial, dmlp);
    if (a.mlp.A > 0) {
        decode_bwd_app_weights<<<kDbBlocks, kAppItems, 0, st>>>(a, s.partial_app);
        reduce_app<<<1, kAppItems, 0, st>>>(s.partial_app, kDbBlocks,
                                            const_cast<float*>(dmlp.w1_app), a.mlp.A);
    }
    return cudaGetLastError();
}

}  // namespace ogs

using namespace ogs;
using namespace ogs::db;

extern "C" ogs_status ogs_project_bwd(const ogs_gaussians* g, int64_t n_gauss, int32_t means_relative,
                                      const ogs_camera* cam, const uint32_t* rect, const float* drec,
                                      float* dmeans, float* dscales, float* dquats,
                                      const ogs_counts* counts, void* stream) {
    if (!g || !cam || !rect || !drec || !dmeans || !dscales || !dquats || n_gauss < 0)
        return OGS_ERR_ARG;
    if (!aligned(g->quats, 16) || !aligned(dquats, 16) || !aligned(rect, 8)) return OGS_ERR_ARG;
    if (n_gauss == 0) return OGS_OK;
    PbArgs a{*g, counts ? &counts->n_gaussians : nullptr, n_gauss, means_relative, make_cam(*cam),
             reinterpret_cast<const uint2*>(rect), drec, dmeans, dscales, dquats};
    project_bwd_kernel<<<stride_grid(n_gauss, kPbThreads, 8), kPbThreads, 0,
                         (cudaStream_t)stream>>>(a);
    return launch_status();
}

extern "C" size_t ogs_decode_bwd_scratch_bytes(int64_t sel_cap) {
    return db_layout(sel_cap < 0 ? 0 : sel_cap, nullptr, nullptr);
}

extern "C" ogs_status ogs_decode_bwd(const float* pos, const float* feat, const float* offs,
                                     const float* lv, int64_t N, const ogs_mlp* mlp,
                                     const ogs_camera* cam, const uint32_t* sel_idx,
                                     const float* sel_w, int64_t sel_cap,
                                     const ogs_counts* counts, const float* dmeans,
                                     const float* dscales, const float* dquats, const float* drec,
                                     float* dfeat, float* doffs, float* dlv, const ogs_mlp* dmlp,
                                     void* scratch, size_t scratch_bytes, void* stream) {
    if (!pos || !feat || !offs || !lv || !mlp || !cam || !sel_idx || !sel_w || !counts ||
        !dmeans || !dscales || !dquats || !drec || !dfeat || !doffs || !dlv || !dmlp || !scratch)
        return OGS_ERR_ARG;
    if (mlp->F != kF || mlp->H != kH || mlp->k != kK || N < 0 || sel_cap < 0 || !app_ok(*mlp))
        return OGS_ERR_ARG;
    if (!dmlp->w1 || !dmlp->b1 || !dmlp->w2_op || !dmlp->b2_op || !dmlp->w2_col ||
        !dmlp->b2_col || !dmlp->w2_cov || !dmlp->b2_cov)
        return OGS_ERR_ARG;
    if (mlp->A > 0 && (!dmlp->w1_app || !dmlp->app)) return OGS_ERR_ARG;
    if (scratch_bytes < ogs_decode_bwd_scratch_bytes(sel_cap) || !aligned(scratch, 16) ||
        !aligned(dquats, 16) || !aligned(feat, 16) || !aligned(dfeat, 16))
        return OGS_ERR_ARG;
    if (sel_cap == 0) return OGS_OK;
    cudaStream_t st = (cudaStream_t)stream;
    DbScratch sc;
    db_layout(sel_cap, scratch, &sc);
    DbArgs a{pos, feat, offs, lv, sel_idx, sel_w, counts, *mlp, make_cam(*cam), dmeans, dscales,
             dquats, drec, dfeat, doffs, dlv, sc.rowY, sc.rowH, sc.rowP, sc.rowZ, sc.partial,
             const_cast<float*>(dmlp->app)};
    const auto rows = mlp->A > 0 ? decode_bwd_rows<true> : decode_bwd_rows<false>;
    if (cudaFuncSetAttribute(rows, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(RowSmem)) != cudaSuccess)
        return OGS_ERR_CUDA;
    const int64_t tiles = (sel_cap + kRowAnchors - 1) / kRowAnchors;
    rows<<<(int)(tiles < 2 * kSmCount ? tiles : 2 * kSmCount), kRowThreads, sizeof(RowSmem), st>>>(a);
    if (launch_weight_pass(a, sc, *dmlp, st) != cudaSuccess) return OGS_ERR_CUDA;
    return launch_status();
}

extern "C" ogs_status ogs_loss_l1(const float* img, const float* target, int64_t n, float* dimg,
                                  float* loss, void* stream) {
    if (!img || !target || !dimg || n <= 0) return OGS_ERR_ARG;
    l1_kernel<<<stride_grid(n, 256, 8), 256, 0, (cudaStream_t)stream>>>(img, target, n,
                                                                         1.0f / (float)n, dimg, loss);
    return launch_status();
}

// Adam over the rows whose stamp equals `value` (the anchors a training step selected).  A
// warp takes kRows rows at a time: their stamps are read in coalesced loads, and the elements of
// the touched rows form one run that the lanes walk together, kAdamFly elements of a lane in flight
// (short rows share a warp's round, and no row waits for the one before); gradients of updated rows
// are cleared.  28 B per element of a touched row, but few rows are touched, so the kernel waits on
// the round trips stamp -> elements: the more rows a warp looks at together, the fewer of them.  2M
// anchors, four 1080p views' rows, row lengths 32, 30 and 3: 26, 33 and 12 us; a row at a time took 33, 38 and
// 29 us, 32 stamps at a time 30, 35 and 24 us.
// With fewer rows, windows of 128 leave too few warps to share the touched rows: 128 from 24 windows
// per SM on (16 for short rows), 32 (64) down to kAdamFew rows, four below.  us for windows of 128 / 64 / 32 / 4
// rows of 32 elements: 500k rows, 2 % touched 6.8 / 8.4 / 7.8 / 14.5, 6 % 12.5 / 12.4 / 10.6 / 18.7; 350k, 2 % 6.4 / 7.2 /
// 6.4 / 12.3, 6 % 10.5 / 10.5 / 9.6 / 14.5; 100k, all touched 48.7 / 28.9 / 18.8 / 16.7; 16k, all touched 47.4 / 26.8 /
// 14.6 / 6.4; 500, all touched 45.3 / 26.9 / 14.5 / 4.4.  Rows of 3: 350k, 2 % touched 4.4 / 6.4 / 6.3 / 12.5; 100k, all
// touched 8.4 / 6.4 / 4.4 / 10.4.
constexpr int64_t kAdamWindow = (int64_t)kSmCount * 128;               // one window of 128 rows per SM
constexpr int64_t kAdamMany = 24 * kAdamWindow, kAdamManyShort = 16 * kAdamWindow, kAdamFew = 32768;
constexpr int kAdamShort = 8;            // elements of a short row
constexpr int kAdamFly = 4;

template <int kRows>
__global__ void __launch_bounds__(256) adam_rows_kernel(float* __restrict__ p,
                                                        float* __restrict__ grad,
                                                        float* __restrict__ m,
                                                        float* __restrict__ v, int64_t rows,
                                                        int row_len,
                                                        const uint32_t* __restrict__ stamp,
                                                        uint32_t value, float lr, float b1,
                                                        float b2, float eps, float ibc1,
                                                        float ibc2, int zero_grad) {
    constexpr int kLoads = (kRows + 31) / 32;
    __shared__ uint8_t s_row[256 / 32][kRows];             // touched rows of the warp, in order
    const int lane = (int)lane_id(), w = threadIdx.x >> 5;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t r0 = warp * kRows; r0 < rows; r0 += nwarps * kRows) {
        bool hit[kLoads];
#pragma unroll
        for (int q = 0; q < kLoads; ++q) {
            const int64_t r = r0 + 32 * q + lane;
            hit[q] = 32 * q + lane < kRows && r < rows && stamp[r] == value;
        }
        int n = 0;
#pragma unroll
        for (int q = 0; q < kLoads; ++q) {
            const uint32_t todo = __ballot_sync(0xffffffffu, hit[q]);
            if (hit[q]) s_row[w][n + __popc(todo & lanemask_lt())] = (uint8_t)(32 * q + lane);
            n += __popc(todo);
        }
        if (!n) continue;
        __syncwarp();
        const int64_t total = (int64_t)n * row_len;
        const bool small = total <= 0x7FFFFFFF;            // 32-bit division
        for (int64_t i0 = lane; i0 < total; i0 += 32 * kAdamFly) {
            int64_t at[kAdamFly];
            float P[kAdamFly], G[kAdamFly], M[kAdamFly], V[kAdamFly];
#pragma unroll
            for (int u = 0; u < kAdamFly; ++u) {
                const int64_t i = i0 + 32 * u;
                if (i < total) {
                    const uint32_t k = small ? (uint32_t)i / (uint32_t)row_len
                                             : (uint32_t)((uint64_t)i / (uint32_t)row_len);
                    at[u] = (r0 + s_row[w][k]) * row_len + (i - (int64_t)k * row_len);
                    P[u] = p[at[u]]; G[u] = grad[at[u]]; M[u] = m[at[u]]; V[u] = v[at[u]];
                }
            }
#pragma unroll
            for (int u = 0; u < kAdamFly; ++u) {
                if (i0 + 32 * u < total) {
                    adam_one(P[u], G[u], M[u], V[u], lr, b1, b2, eps, ibc1, ibc2, zero_grad);
                    p[at[u]] = P[u];
                    m[at[u]] = M[u];
                    v[at[u]] = V[u];
                    if (zero_grad) grad[at[u]] = G[u];
                }
            }
        }
        __syncwarp();                                      // the list is rewritten
    }
}

// The first 9 counts->n_gaussians values of drec to zero (at most 9 g_cap); with `held`, the first
// 9 held[0], and held[0] becomes counts->n_gaussians once every CTA has read it (held[1] counts them; two
// CTAs per SM, since the atomics queue up: views of up to 600k Gaussians as without held, 4.2 to 6.3 us, with eight 5.1
// to 6.3; counted before the clearing, beside the others' reads of held[0], eight took 11.5 to 13.9).
__global__ void __launch_bounds__(256) clear_records_kernel(float* __restrict__ drec, int64_t g_cap,
                                                            const ogs_counts* __restrict__ counts,
                                                            uint32_t* held, int vec) {
    const int64_t g = held ? held[0] : counts->n_gaussians, n = 9 * (g < g_cap ? g : g_cap);
    const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t n4 = vec ? n / 4 : 0;
    for (int64_t i = i0; i < n4; i += stride)
        reinterpret_cast<float4*>(drec)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int64_t i = 4 * n4 + i0; i < n; i += stride) drec[i] = 0.f;
    if (!held) return;
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(held + 1, 1u) == gridDim.x - 1) {
        held[0] = counts->n_gaussians;
        held[1] = 0u;
    }
}

extern "C" ogs_status ogs_clear_records(float* drec, int64_t g_cap, const ogs_counts* counts,
                                        void* stream) {
    if (!drec || !counts || g_cap < 0) return OGS_ERR_ARG;
    if (g_cap == 0) return OGS_OK;
    clear_records_kernel<<<stride_grid(9 * g_cap / 4 + 1, 256, 8), 256, 0, (cudaStream_t)stream>>>(
        drec, g_cap, counts, nullptr, aligned(drec, 16));
    return launch_status();
}

extern "C" ogs_status ogs_renew_records(float* drec, int64_t g_cap, const ogs_counts* counts,
                                        uint32_t* held, void* stream) {
    if (!drec || !counts || !held || g_cap < 0) return OGS_ERR_ARG;
    if (g_cap == 0) return OGS_OK;
    clear_records_kernel<<<stride_grid(9 * g_cap / 4 + 1, 256, 2), 256, 0, (cudaStream_t)stream>>>(
        drec, g_cap, counts, held, aligned(drec, 16));
    return launch_status();
}

// stamp[sel_idx[r]] = value for the r < counts->n_selected selected anchors
__global__ void stamp_rows_kernel(const uint32_t* __restrict__ sel_idx,
                                  const ogs_counts* __restrict__ counts,
                                  uint32_t* __restrict__ stamp, uint32_t value) {
    const uint32_t M = counts->n_selected;
    for (uint32_t r = blockIdx.x * blockDim.x + threadIdx.x; r < M; r += gridDim.x * blockDim.x)
        stamp[sel_idx[r]] = value;
}

extern "C" ogs_status ogs_stamp_selected(const uint32_t* sel_idx, const ogs_counts* counts,
                                         int64_t sel_cap, uint32_t* stamp, uint32_t value,
                                         void* stream) {
    if (!sel_idx || !counts || !stamp || sel_cap < 0) return OGS_ERR_ARG;
    if (sel_cap == 0) return OGS_OK;
    stamp_rows_kernel<<<stride_grid(sel_cap, 256, 8), 256, 0, (cudaStream_t)stream>>>(
        sel_idx, counts, stamp, value);
    return launch_status();
}

extern "C" ogs_status ogs_adam_rows(float* param, float* grad, float* m, float* v, int64_t rows,
                                    int32_t row_len, const uint32_t* stamp, uint32_t value,
                                    float lr, float beta1, float beta2, float eps, int32_t step,
                                    int32_t zero_grad, void* stream) {
    if (!param || !grad || !m || !v || !stamp || rows < 0 || row_len < 1 || step < 1)
        return OGS_ERR_ARG;
    if (rows == 0) return OGS_OK;
    const double bc1 = 1.0 - pow((double)beta1, (double)step);
    const double bc2 = 1.0 - pow((double)beta2, (double)step);
    const bool is_short = row_len <= kAdamShort;
    const int n = rows >= (is_short ? kAdamManyShort : kAdamMany) ? 128
                                                                  : (rows < kAdamFew ? 4 : (is_short ? 64 : 32));
    const auto kernel = n == 128 ? adam_rows_kernel<128>
                                 : (n == 64 ? adam_rows_kernel<64>
                                            : (n == 32 ? adam_rows_kernel<32> : adam_rows_kernel<4>));
    kernel<<<stride_grid((rows + n - 1) / n * 32, 256, 8), 256, 0, (cudaStream_t)stream>>>(
        param, grad, m, v, rows, row_len, stamp, value, lr, beta1, beta2, eps, (float)(1.0 / bc1),
        (float)(1.0 / bc2), zero_grad);
    return launch_status();
}

// flag |= bit if any of x[0..n) is NaN or infinite (one atomic per warp that finds one)
__global__ void nonfinite_kernel(const float* __restrict__ x, int64_t n, uint32_t* flag,
                                 uint32_t bit) {
    bool bad = false;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        bad |= !isfinite(x[i]);
    if (__any_sync(0xffffffffu, bad) && lane_id() == 0) atomicOr(flag, bit);
}

extern "C" ogs_status ogs_scan_nonfinite(const float* x, int64_t n, uint32_t* flag, uint32_t bit,
                                         void* stream) {
    if (!x || !flag || n < 0 || bit == 0) return OGS_ERR_ARG;
    if (n == 0) return OGS_OK;
    nonfinite_kernel<<<stride_grid(n, 256, 8), 256, 0, (cudaStream_t)stream>>>(x, n, flag, bit);
    return launch_status();
}

extern "C" ogs_status ogs_counts_status(const ogs_counts* counts, uint32_t nonfinite) {
    if (!counts) return OGS_ERR_ARG;
    if (nonfinite) return OGS_ERR_NONFINITE;
    if (counts->timeout) return OGS_ERR_TIMEOUT;
    if (counts->overflow) return OGS_ERR_CAPACITY;
    return OGS_OK;
}

extern "C" ogs_status ogs_scale(float* x, int64_t n, const float* s, void* stream) {
    if (!x || !s || n < 0) return OGS_ERR_ARG;
    if (n == 0) return OGS_OK;
    scale_kernel<<<stride_grid(n, 256, 8), 256, 0, (cudaStream_t)stream>>>(x, n, s);
    return launch_status();
}

extern "C" ogs_status ogs_adam(float* param, float* grad, float* m, float* v, int64_t n, float lr,
                               float beta1, float beta2, float eps, int32_t step,
                               int32_t zero_grad, void* stream) {
    if (!param || !grad || !m || !v || n < 0 || step < 1) return OGS_ERR_ARG;
    if (n == 0) return OGS_OK;
    const double bc1 = 1.0 - pow((double)beta1, (double)step);
    const double bc2 = 1.0 - pow((double)beta2, (double)step);
    const int vec = aligned(param, 16) && aligned(grad, 16) && aligned(m, 16) && aligned(v, 16);
    adam_kernel<<<stride_grid(vec ? n / 4 + 1 : n, 256, 8), 256, 0, (cudaStream_t)stream>>>(
        param, grad, m, v, n, lr, beta1, beta2, eps, (float)(1.0 / bc1), (float)(1.0 / bc2),
        zero_grad, vec);
    return launch_status();
}
