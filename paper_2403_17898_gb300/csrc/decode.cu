// Neural-Gaussian decoding (Sec. 3.2): per selected anchor, the three attribute MLPs
// (Eq. mlp) and the offset positions (Eq. offsets), FP32 on the CUDA cores.
//
// A CTA takes 64 anchors at a time through two small matrix products with both operands in shared
// memory and register blocks of outputs.  Layer 1: a thread owns 4 anchors x 12 hidden units.
// Layer 2: a thread owns 4 anchors x the 11 outputs of one Gaussian slot (opacity, colour,
// covariance), so it activates and stores that Gaussian by itself, and consecutive threads store
// consecutive Gaussians.  Products are packed over anchor pairs; each output is one chain of
// fused multiply-adds over its inputs, bias first.  Means are written camera-relative
// (x_v - campos + O_i * l_v) so FP32 keeps them accurate far from the world origin.  With
// appearance codes (Sec. 4.4) the colour decoder's hidden units also see the anchor's code.
//
// Bound by the FP32 pipes and shared-memory loads (44 products per six 16-byte loads).  The earlier
// form, a thread per anchor, read every weight once per four products, kept 12 warps an SM and
// stored with a stride of one anchor: 100k anchors 122 us, now 66 us; 4k anchors 38 -> 17 us.
#include "internal.cuh"

namespace ogs {
namespace {

constexpr int kK = 10;                   // Gaussians per anchor
constexpr int kF = 32;
constexpr int kH = 32;
constexpr int kDin = kF + 4;
constexpr int kHid = 3 * kH;             // hidden units of the three decoders
constexpr int kTileA = 64;               // anchors per tile
constexpr int kGroups = kTileA / 4;      // of four anchors
constexpr int kDecThreads = kGroups * kK;            // layer 2: (anchor group, Gaussian slot)
constexpr int kHidPer = 12;              // layer 1: hidden units per thread
constexpr int kL1Threads = kGroups * (kHid / kHidPer);
constexpr int kOut = 11, kOutPad = 12;   // outputs of one Gaussian: 1 + 3 + 7
static_assert(kL1Threads == 128 && kDecThreads == 160, "thread roles");

struct DecArgs {
    const float* pos;
    const float* feat;
    const float* offs;
    const float* lv;
    const uint32_t* sel_idx;
    const float* sel_w;
    const ogs_counts* counts;
    int64_t sel_cap;
    ogs_mlp mlp;
    ogs_gaussians out;
    Cam cam;
};

struct __align__(16) DecSmem {
    float w1[kDin + kMaxApp][kHid];      // transposed; rows kDin .. are the appearance weights
    float w2[kH][kK][kOutPad];           // per hidden unit and Gaussian: opacity, colour, covariance
    float b1[kHid];
    float b2[kK][kOutPad];
    float z[kDin + kMaxApp][kTileA];     // inputs, then the appearance code
    float h[kHid][kTileA];               // hidden activations
    float rows[kTileA][8];               // anchor index, weight, x_v - campos, l_v
};

__device__ __forceinline__ float sigmoidf_(float x) { return 1.0f / (1.0f + __expf(-x)); }

template <bool APP>
__global__ void __launch_bounds__(kDecThreads, 3) decode_fp32(DecArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    DecSmem& s = *reinterpret_cast<DecSmem*>(smem_raw);
    const uint32_t M = a.counts->n_selected;
    const uint32_t ntiles = (M + kTileA - 1) / kTileA;
    if (blockIdx.x >= ntiles) return;
    const int t = threadIdx.x;
    const ogs_mlp& m = a.mlp;
#pragma unroll 8
    for (int e = t; e < kDin * kHid; e += kDecThreads) s.w1[e / kHid][e % kHid] = m.w1[(e % kHid) * kDin + e / kHid];
    if (APP) {
        for (int e = t; e < kMaxApp * kH; e += kDecThreads) {
            const int q = e / kH, o = e % kH;
            s.w1[kDin + q][kH + o] = q < m.A ? m.w1_app[o * m.A + q] : 0.f;
        }
    }
#pragma unroll 8
    for (int e = t; e < kH * kK * kOutPad; e += kDecThreads) {
        const int o = e / (kK * kOutPad), i = e / kOutPad % kK, c = e % kOutPad;
        const float* w = c == 0 ? m.w2_op + i * kH
                                : (c < 4 ? m.w2_col + (3 * i + c - 1) * kH
                                         : m.w2_cov + (7 * i + (c < kOut ? c - 4 : 0)) * kH);
        s.w2[o][i][c] = w[o];
    }
    for (int e = t; e < kHid; e += kDecThreads) s.b1[e] = m.b1[e];
    for (int e = t; e < kK * kOut; e += kDecThreads) {
        const int i = e / kOut, c = e % kOut;
        s.b2[i][c] = c == 0 ? m.b2_op[i] : (c < 4 ? m.b2_col[3 * i + c - 1] : m.b2_cov[7 * i + c - 4]);
    }
    const Cam& c = a.cam;
    for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const uint32_t base = tile * kTileA;
        // gather: two threads per anchor, inputs transposed
        if (t < 2 * kTileA) {
            const int al = t % kTileA, half = t / kTileA;
            const bool valid = base + al < M;
            const uint32_t j = valid ? a.sel_idx[base + al] : 0u;
            float4 v[4];
            const float4* f4 = reinterpret_cast<const float4*>(a.feat + (size_t)j * kF) + 4 * half;
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = valid ? f4[i] : make_float4(0.f, 0.f, 0.f, 0.f);
            if (half == 0) {
                float dv[3] = {0.f, 0.f, 0.f}, lv[3] = {0.f, 0.f, 0.f}, d = 1.f, w = 0.f;
                if (valid) {
                    w = a.sel_w[base + al];
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        dv[q] = a.pos[3 * (size_t)j + q] - c.c[q];
                        lv[q] = a.lv[3 * (size_t)j + q];
                    }
                    d = sqrtf(dv[0] * dv[0] + dv[1] * dv[1] + dv[2] * dv[2]);
                }
#pragma unroll
                for (int q = 0; q < 3; ++q) s.z[kF + q][al] = dv[q] / d;
                s.z[kF + 3][al] = d;
                float4* r = reinterpret_cast<float4*>(s.rows[al]);
                r[0] = make_float4(__uint_as_float(j), w, dv[0], dv[1]);
                r[1] = make_float4(dv[2], lv[0], lv[1], lv[2]);
            } else if (APP) {
#pragma unroll
                for (int q = 0; q < kMaxApp; ++q)
                    s.z[kDin + q][al] = valid && q < m.A ? m.app[(size_t)j * m.A + q] : 0.f;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int k = 16 * half + 4 * i;
                s.z[k][al] = v[i].x;
                s.z[k + 1][al] = v[i].y;
                s.z[k + 2][al] = v[i].z;
                s.z[k + 3][al] = v[i].w;
            }
        }
        __syncthreads();
        if (t < kL1Threads) {
            const int ag = t % kGroups, o0 = t / kGroups * kHidPer;
            f32x2 acc[kHidPer][2];
#pragma unroll
            for (int o = 0; o < kHidPer; ++o) acc[o][0] = acc[o][1] = pack2(s.b1[o0 + o], s.b1[o0 + o]);
#pragma unroll 4
            for (int k = 0; k < kDin; ++k) {
                const float4 z = *reinterpret_cast<const float4*>(&s.z[k][4 * ag]);
                const f32x2 z0 = pack2(z.x, z.y), z1 = pack2(z.z, z.w);
#pragma unroll
                for (int q = 0; q < kHidPer / 4; ++q) {
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
            if (APP) {                             // the colour decoder also sees the code
#pragma unroll 1
                for (int k = kDin; k < kDin + kMaxApp; ++k) {
                    const float4 z = *reinterpret_cast<const float4*>(&s.z[k][4 * ag]);
                    const f32x2 z0 = pack2(z.x, z.y), z1 = pack2(z.z, z.w);
#pragma unroll
                    for (int o = 0; o < kHidPer; ++o) {
                        if (o0 + o < kH || o0 + o >= 2 * kH) continue;
                        const f32x2 w2 = pack2(s.w1[k][o0 + o], s.w1[k][o0 + o]);
                        acc[o][0] = fma2(w2, z0, acc[o][0]);
                        acc[o][1] = fma2(w2, z1, acc[o][1]);
                    }
                }
            }
#pragma unroll
            for (int o = 0; o < kHidPer; ++o)
                *reinterpret_cast<float4*>(&s.h[o0 + o][4 * ag]) =
                    make_float4(fmaxf(lo2(acc[o][0]), 0.f), fmaxf(hi2(acc[o][0]), 0.f),
                                fmaxf(lo2(acc[o][1]), 0.f), fmaxf(hi2(acc[o][1]), 0.f));
        }
        __syncthreads();
        {
            const int i = t % kK, ag = t / kK;
            float O[4][3];                         // in flight during the product
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (base + 4 * ag + q < M) {
                    const uint32_t j = __float_as_uint(s.rows[4 * ag + q][0]);
#pragma unroll
                    for (int e = 0; e < 3; ++e) O[q][e] = a.offs[((size_t)j * kK + i) * 3 + e];
                }
            }
            f32x2 acc[kOut][2];
#pragma unroll
            for (int e = 0; e < kOut; ++e) acc[e][0] = acc[e][1] = pack2(s.b2[i][e], s.b2[i][e]);
#pragma unroll 2
            for (int o = 0; o < kH; ++o) {
                float w[kOutPad];
#pragma unroll
                for (int q = 0; q < kOutPad / 4; ++q) {
                    const float4 v = *reinterpret_cast<const float4*>(&s.w2[o][i][4 * q]);
                    w[4 * q] = v.x; w[4 * q + 1] = v.y; w[4 * q + 2] = v.z; w[4 * q + 3] = v.w;
                }
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    const float4 h = *reinterpret_cast<const float4*>(&s.h[d * kH + o][4 * ag]);
                    const f32x2 h0 = pack2(h.x, h.y), h1 = pack2(h.z, h.w);
#pragma unroll
                    for (int e = d == 0 ? 0 : (d == 1 ? 1 : 4); e < (d == 0 ? 1 : (d == 1 ? 4 : kOut)); ++e) {
                        const f32x2 w2 = pack2(w[e], w[e]);
                        acc[e][0] = fma2(w2, h0, acc[e][0]);
                        acc[e][1] = fma2(w2, h1, acc[e][1]);
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t r = base + 4 * ag + q;
                if (r >= M) continue;
                float y[kOut];
#pragma unroll
                for (int e = 0; e < kOut; ++e) y[e] = q & 1 ? hi2(acc[e][q / 2]) : lo2(acc[e][q / 2]);
                const float4 r0 = *reinterpret_cast<const float4*>(&s.rows[4 * ag + q][0]);
                const float4 r1 = *reinterpret_cast<const float4*>(&s.rows[4 * ag + q][4]);
                const float w = r0.y, dv[3] = {r0.z, r0.w, r1.x}, lv[3] = {r1.y, r1.z, r1.w};
                const size_t g = (size_t)r * kK + i;
                // opacity: w * tanh (a Gaussian with opacity <= 0 is dropped by the projection)
                a.out.opac[g] = w * tanhf(y[0]);
#pragma unroll
                for (int e = 0; e < 3; ++e) {
                    a.out.colors[3 * g + e] = sigmoidf_(y[1 + e]);
                    a.out.scales[3 * g + e] = lv[e] * sigmoidf_(y[4 + e]);
                    a.out.means[3 * g + e] = dv[e] + O[q][e] * lv[e];
                }
                const float q0 = y[7], q1 = y[8], q2 = y[9], q3 = y[10];
                const float inv = 1.0f / sqrtf(q0 * q0 + q1 * q1 + q2 * q2 + q3 * q3);
                *reinterpret_cast<float4*>(a.out.quats + 4 * g) =
                    make_float4(q0 * inv, q1 * inv, q2 * inv, q3 * inv);
            }
        }
        __syncthreads();                           // inputs and rows are rewritten by the next tile
    }
}

template <bool APP>
ogs_status launch_decode(const DecArgs& a, cudaStream_t st) {
    if (cudaFuncSetAttribute(decode_fp32<APP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(DecSmem)) != cudaSuccess)
        return OGS_ERR_CUDA;
    const int64_t tiles = (a.sel_cap + kTileA - 1) / kTileA;
    const int grid = (int)(tiles < 3 * kSmCount ? tiles : 3 * kSmCount);
    decode_fp32<APP><<<grid, kDecThreads, sizeof(DecSmem), st>>>(a);
    return launch_status();
}

}  // namespace
}  // namespace ogs

using namespace ogs;

extern "C" ogs_status ogs_decode(const float* pos, const float* feat, const float* offs,
                                 const float* lv, int64_t N, const ogs_mlp* mlp,
                                 const ogs_camera* cam, const uint32_t* sel_idx,
                                 const float* sel_w, int64_t sel_cap, const ogs_counts* counts,
                                 const ogs_gaussians* out, void* stream) {
    if (!pos || !feat || !offs || !lv || !mlp || !cam || !sel_idx || !sel_w || !counts || !out)
        return OGS_ERR_ARG;
    if (mlp->F != kF || mlp->H != kH || mlp->k != kK || N < 0 || sel_cap < 0 || !app_ok(*mlp))
        return OGS_ERR_ARG;
    if (!mlp->w1 || !mlp->b1 || !mlp->w2_op || !mlp->b2_op || !mlp->w2_col || !mlp->b2_col ||
        !mlp->w2_cov || !mlp->b2_cov)
        return OGS_ERR_ARG;
    if (!out->means || !out->scales || !out->quats || !out->opac || !out->colors)
        return OGS_ERR_ARG;
    if (!aligned(feat, 16) || !aligned(out->quats, 16) || !aligned(mlp->w1, 16)) return OGS_ERR_ARG;
    if (sel_cap == 0) return OGS_OK;
    DecArgs a{pos, feat, offs, lv, sel_idx, sel_w, counts, sel_cap, *mlp, *out, make_cam(*cam)};
    return mlp->A > 0 ? launch_decode<true>(a, (cudaStream_t)stream)
                      : launch_decode<false>(a, (cudaStream_t)stream);
}
