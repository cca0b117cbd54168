// Backward of the front-to-back blending (Sec. 3.1, Eq. 2).
//
// With C = sum_i c_i a_i T_i + T_{n+1} bg:  dC/dc_i = a_i T_i and dC/da_i = T_i (c_i - S_i),
// where S_i is the colour accumulated behind Gaussian i (S_n = bg, S_{i-1} = a_i c_i +
// (1 - a_i) S_i).  Each pixel replays its list back to front from its last blended entry,
// recovering T_i = T_{i+1} / (1 - a_i) from the final transmittance instead of storing
// per-pair values (1 - a_i >= 0.01 because a is clamped to 0.99).  a = min(0.99, o G) has
// zero derivative where clamped.  Same tile/pixel mapping and skip test as the forward (two
// pixels per thread, each warp walking only the records whose alpha >= 1/255 ellipse can
// reach its 8x8 block).
//
// The kernel is bound by instruction issue, so the walk is cut to what a pixel has to do by
// itself: only the scalar S_i . dC is carried (not the three colours), and a (pixel, Gaussian)
// pair leaves two numbers, w = a T (weight of the colour gradient) and s = dL/dpower.  All nine
// record gradients are sums of s and w over pixels: d(u, v, a, b, c) are the moments of s up to
// second order in the pixel's offset, d(o) = sum s / o, d(colour) = sum w dC.  So a warp parks
// (s, w) of kGroup entries in shared memory and then turns round: a lane takes one entry and
// sums its moments over the block's pixels, a column's offset shared by its rows.  That replaces a 16-value shuffle reduction per (warp, entry):
// 1080p with 2.1M list entries (3.9M visits of a warp to an entry, 3.3M with a pixel that
// blended it) 741 -> 411 us, 188 -> 84 instructions per visit; issue slots 69 % busy, shared
// memory 69 %.  Groups of 16 need fewer instructions but 44 KB a CTA (437 us), groups of 32 lost
// more in a first form; evaluating two entries at a time gained 3 % over one, four lost 5 %;
// batches of 64 or 256 records lose 2 to 10 %.
#include <type_traits>

#include "blend_common.cuh"

namespace ogs {
namespace {

using namespace blend;

constexpr int kBwdBatch = 128;           // records staged per shared-memory batch
constexpr int kGroup = 8;                // entries whose (s, w) a warp parks before summing
constexpr int kParts = 32 / kGroup;      // lanes that share one entry's sums
constexpr int kSlots = 32 / kParts;      // pixel pairs summed by one of them
constexpr int kRowPairs = kSlots / 8;    // rows of pixel pairs in those
constexpr int kWalk = 2;                 // entries a warp evaluates at a time
constexpr int kPitch = 33;               // float4 per parked entry: conflict-free both ways
constexpr int kDPitch = 32 + kParts;     // float2 per colour: the parts read different banks
static_assert(kGroup * kPitch * 4 >= 32 * 9, "the sums are laid out over the parked pairs");
static_assert(kBwdBatch * sizeof(StagedRec) < 65536, "record offsets fit 16 bits");

struct __align__(16) BwdSmem {
    StagedRec rec[kBwdBatch];
    float4 park[kThreads / 32][kGroup * kPitch];   // s0, s1, w0, w1 of entry e, pixel pair l
    float2 d[kThreads / 32][3][kDPitch];           // image gradient of the pairs, by colour
    uint32_t g[kBwdBatch];
    uint32_t gid[kThreads / 32][kGroup];           // Gaussians of the group being added
    uint16_t list[kThreads / 32][kBwdBatch];       // byte offsets of the warp's records
    uint8_t m[kBwdBatch];
};

__device__ __forceinline__ f32x2 as2(float2 v) { return pack2(v.x, v.y); }

// Sums the ng parked entries of this warp over its block and adds them to drec.  Lane
// (part, e) takes entry e, whose record lies at offset `at`, and pixel pairs [part kSlots, ...);
// (bx, by) is the block's first pixel.
// The map from moments to gradients is linear, so every part applies it to its own share and
// the shares meet where they are added to drec.  kCareful: some image gradient of the block is
// not finite; pixels that skipped an entry (w = 0) then keep out of its sums by selection.
template <bool kCareful>
__device__ __forceinline__ void flush_group(BwdSmem& sm, int w, int ng, int at, float bx, float by,
                                            float* __restrict__ drec) {
    const int lane = (int)lane_id(), e = lane % kGroup, part = lane / kGroup;
    __syncwarp();
    const float4* park = sm.park[w] + e * kPitch + part * kSlots;
    const float2* dc = sm.d[w][0] + part * (kSlots + 1);
    const StagedRec& rc = *reinterpret_cast<const StagedRec*>(
        reinterpret_cast<const unsigned char*>(sm.rec) + (e < ng ? at : 0));
    const float4 A = rc.A;
    const float2 B = *reinterpret_cast<const float2*>(&rc.B);
    const uint32_t gid = sm.g[&rc - sm.rec];
    // per row pair, packed over its two rows: sums of s, s dx, s dx^2; colours packed alike
    f32x2 m0[kRowPairs], m1[kRowPairs], xx2 = 0;
    f32x2 col[3] = {0, 0, 0};
#pragma unroll
    for (int r = 0; r < kRowPairs; ++r) m0[r] = m1[r] = 0;
    float dx = A.x - bx;                  // of column 0
#pragma unroll
    for (int c = 0; c < 8; ++c, dx -= 1.0f) {
        const f32x2 dx2 = pack2(dx, dx);
#pragma unroll
        for (int r = 0; r < kRowPairs; ++r) {
            const float4 v = park[8 * r + c];
            const f32x2 s = pack2(v.x, v.y), wv = pack2(v.z, v.w);
            const f32x2 sx = mul2(s, dx2);
            m0[r] = add2(m0[r], s);
            m1[r] = add2(m1[r], sx);
            xx2 = fma2(sx, dx2, xx2);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                float2 d = dc[k * kDPitch + 8 * r + c];
                if (kCareful) {
                    d.x = v.z != 0.f ? d.x : 0.f;
                    d.y = v.w != 0.f ? d.y : 0.f;
                }
                col[k] = fma2(wv, as2(d), col[k]);
            }
        }
    }
    float S = 0.f, X = 0.f, Y = 0.f, XY = 0.f, YY = 0.f;
    const float xx = lo2(xx2) + hi2(xx2);
    float dy = A.y - (by + (float)(2 * part * kRowPairs));
#pragma unroll
    for (int r = 0; r < kRowPairs; ++r) {
#pragma unroll
        for (int h = 0; h < 2; ++h, dy -= 1.0f) {
            const float a0 = h ? hi2(m0[r]) : lo2(m0[r]), a1 = h ? hi2(m1[r]) : lo2(m1[r]);
            const float sy = a0 * dy;
            S += a0;
            X += a1;
            Y += sy;
            XY = fmaf(a1, dy, XY);
            YY = fmaf(sy, dy, YY);
        }
    }
    __syncwarp();                        // every lane has read the parked pairs
    float* out = reinterpret_cast<float*>(sm.park[w]);
    if (e < ng) {
        // the record's conic is (a, b, c) with power = -0.5 (a dx^2 + c dy^2) - b dx dy
        constexpr float kA = 1.3862943611198906f;      // 2 / log2(e) = 2 ln 2
        constexpr float kB = 0.6931471805599453f;      // 1 / log2(e) = ln 2
        const float a = A.z * kA, b = A.w * kB, c = B.x * kA;
        float* o = out + 9 * (part * kGroup + e);
        o[0] = -fmaf(a, X, b * Y);
        o[1] = -fmaf(c, Y, b * X);
        o[2] = -0.5f * xx;
        o[3] = -XY;
        o[4] = -0.5f * YY;
        o[5] = S * rcp(B.y);
#pragma unroll
        for (int k = 0; k < 3; ++k) o[6 + k] = lo2(col[k]) + hi2(col[k]);
        if (part == 0) sm.gid[w][e] = gid;
    }
    __syncwarp();
    // consecutive lanes add consecutive components of three entries at a time: whole sectors
    // per atomic instruction
    const int ee = lane / 9, c = lane % 9;
    if (ee < 3) {
        for (int i = ee; i < ng; i += 3) {
            float v = out[9 * i + c];
#pragma unroll
            for (int p = 1; p < kParts; ++p) v += out[9 * (p * kGroup + i) + c];
            atomicAdd(drec + 9 * (size_t)sm.gid[w][i] + c, v);
        }
    }
    __syncwarp();                        // the buffer may be parked in again
}

// A thread's two pixels: the first one's coordinates, and what the walk carries (packed).
struct PairState {
    float fx, fy;
    f32x2 T, Q;              // transmittance behind the entry; colour behind it . image gradient
    float dr[2], dg[2], db[2];
};

// One entry's (s, w) at both pixels and their step towards the front.  A pixel that skipped the
// entry (!ok) has alpha = 0, which leaves its state as it is: the approximate reciprocal of 1 is
// exactly 1 (its bound of an ulp alone would not say so; the blend tests walk past 600 skipped entries).  kCareful: the entry can clamp
// alpha (whose gradient is then zero), or something is not finite (0 x inf): the exact selections.
template <bool kCareful>
__device__ __forceinline__ float4 pair_step(PairState& p, bool ok0, bool ok1, float q0, float q1,
                                            const float4& B, float blue) {
    float a0 = ok0 ? __fmul_rn(B.y, ex2(-q0)) : 0.f, a1 = ok1 ? __fmul_rn(B.y, ex2(-q1)) : 0.f;
    if (kCareful) {
        a0 = fminf(0.99f, a0);
        a1 = fminf(0.99f, a1);
    }
    const f32x2 al = pack2(a0, a1);
    const f32x2 om = sub2(pack2(1.f, 1.f), al);
    p.T = mul2(p.T, pack2(rcp(lo2(om)), rcp(hi2(om))));             // T_i, before this entry
    const f32x2 w = mul2(al, p.T);
    const f32x2 cd = pack2(fmaf(B.z, p.dr[0], fmaf(B.w, p.dg[0], blue * p.db[0])),
                           fmaf(B.z, p.dr[1], fmaf(B.w, p.dg[1], blue * p.db[1])));
    f32x2 df = sub2(cd, p.Q);
    if (kCareful) df = pack2(ok0 ? lo2(df) : 0.f, ok1 ? hi2(df) : 0.f);
    p.Q = fma2(al, df, p.Q);
    f32x2 s = mul2(w, df);                                          // alpha dL/dalpha
    if (kCareful) s = pack2(a0 < 0.99f ? lo2(s) : 0.f, a1 < 0.99f ? hi2(s) : 0.f);
    return make_float4(lo2(s), hi2(s), lo2(w), hi2(w));
}

// Walks a warp's list of a staged batch back to front.  lo: list position of the batch's first
// record; a pixel takes part from its last blended entry on.
template <bool kCareful>
__device__ __forceinline__ void walk_list(BwdSmem& sm, int w, int nw, PairState& ps, int last0,
                                          int last1, float bx, float by, float* __restrict__ drec) {
    const int lane = (int)lane_id();
    const uint16_t* list = sm.list[w];
    const unsigned char* recs = reinterpret_cast<const unsigned char*>(sm.rec);
    int ng = 0, my_at = 0;             // parked entries; record of the one this lane will sum
    // kN entries, list[it], list[it - 1], ...: independent up to the transmittance chain
    auto step = [&](int it, auto n_) {
        constexpr int kN = decltype(n_)::value;
        int at[kN];
        float q0[kN], q1[kN];
        float4 B[kN];
        float2 C[kN];
        bool ok0[kN], ok1[kN], any[kN];
#pragma unroll
        for (int u = 0; u < kN; ++u) {
            at[u] = list[it - u];
            const StagedRec& r = *reinterpret_cast<const StagedRec*>(recs + at[u]);
            const float4 A = r.A;
            B[u] = r.B;
            C[u] = *reinterpret_cast<const float2*>(&r.C);
            const float dx = A.x - ps.fx, dy = A.y - ps.fy, ax = __fmul_rn(A.z, dx);
            q0[u] = power2(ax, dx, dy, A.w, B[u].x);
            q1[u] = power2(ax, dx, dy - 1.0f, A.w, B[u].x);
            ok0[u] = at[u] < last0 && passes(q0[u], C[u].y);
            ok1[u] = at[u] < last1 && passes(q1[u], C[u].y);
            any[u] = __any_sync(0xffffffffu, ok0[u] || ok1[u]);
        }
#pragma unroll
        for (int u = 0; u < kN; ++u) {
            if (!any[u]) continue;
            sm.park[w][ng * kPitch + lane] =
                pair_step<kCareful>(ps, ok0[u], ok1[u], q0[u], q1[u], B[u], C[u].x);
            my_at = lane % kGroup == ng ? at[u] : my_at;
            ++ng;
        }
        if (ng > kGroup - kWalk) {
            flush_group<kCareful>(sm, w, ng, my_at, bx, by, drec);
            ng = 0;
        }
    };
    int it = nw - 1;
    for (; it >= kWalk - 1; it -= kWalk) step(it, std::integral_constant<int, kWalk>());
    for (; it >= 0; --it) step(it, std::integral_constant<int, 1>());
    if (ng) flush_group<kCareful>(sm, w, ng, my_at, bx, by, drec);
}

// 72 registers (a few spilled outside the walk): 411 us; 80 and six CTAs: 422; 64 and eight: 435
constexpr int kMinCtas = 7;

__global__ void __launch_bounds__(kThreads, kMinCtas) blend_bwd_kernel(
    const float4* __restrict__ rec, const uint32_t* __restrict__ pair_gauss,
    const uint2* __restrict__ tile_range, int W, int H, int gx, float bg0, float bg1, float bg2,
    const float* __restrict__ T_final, const uint32_t* __restrict__ n_last,
    const float* __restrict__ dimg, float* __restrict__ drec) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    BwdSmem& sm = *reinterpret_cast<BwdSmem*>(smem_raw);
    __shared__ int s_maxlast;
    const int tile = blockIdx.x;
    int lx, ly;
    pixels_of(threadIdx.x, lx, ly);
    const int tx0 = (tile % gx) * kTile, ty0 = (tile / gx) * kTile;
    const int px = tx0 + lx;
    const int py = ty0 + ly;
    const int w = threadIdx.x >> 5;
    const int lane = (int)lane_id();
    const uint2 range = tile_range[tile];
    if (range.x == range.y) return;    // nothing was blended: no pixel state to read
    const size_t plane = (size_t)W * H;
    float T[2] = {1.f, 1.f}, d[3][2] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
    int last[2] = {0, 0};
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        if (px < W && py + i < H) {
            const size_t pix = (size_t)(py + i) * W + px;
            last[i] = (int)n_last[pix];
            T[i] = T_final[pix];
#pragma unroll
            for (int k = 0; k < 3; ++k) d[k][i] = dimg[k * plane + pix];
        }
    }
    PairState ps;
    ps.fx = (float)px;
    ps.fy = (float)py;
    ps.T = pack2(T[0], T[1]);
    float q[2];
    bool bad = false;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        ps.dr[i] = d[0][i];
        ps.dg[i] = d[1][i];
        ps.db[i] = d[2][i];
        q[i] = fmaf(bg0, d[0][i], fmaf(bg1, d[1][i], bg2 * d[2][i]));
        bad = bad || !isfinite(q[i]) || !isfinite(d[0][i]) || !isfinite(d[1][i]) || !isfinite(d[2][i]);
    }
    ps.Q = pack2(q[0], q[1]);
    if (threadIdx.x == 0) s_maxlast = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) sm.d[w][k][lane + lane / kSlots] = make_float2(d[k][0], d[k][1]);
    __syncthreads();
    const int wlast = (int)__reduce_max_sync(0xffffffffu, (unsigned)max(last[0], last[1]));
    if (lane == 0) atomicMax(&s_maxlast, wlast);
    bad = __any_sync(0xffffffffu, bad);
    __syncthreads();
    const int n = s_maxlast;           // entries beyond every pixel's last blend are unused
    const float bx = (float)(tx0 + 8 * (w & 1)), by = (float)(ty0 + 8 * (w >> 1));
    for (int top = n; top > 0; top -= kBwdBatch) {
        const int lo = max(top - kBwdBatch, 0);
        bool careful = false;
        __syncthreads();
        for (int e = threadIdx.x; lo + e < top; e += kThreads) {
            const uint32_t g = pair_gauss[range.x + lo + e];
            sm.g[e] = g;
            const uint32_t m = stage_rec(rec, g, (float)tx0, (float)ty0, sm.rec[e]);
            sm.m[e] = (uint8_t)m;
            careful = careful || (m & 16u);
        }
        careful = __syncthreads_or(careful) || bad;
        const int nw = warp_list<(int)sizeof(StagedRec)>(sm.m, min(top - lo, wlast - lo), sm.list[w]);
        // list positions as record offsets: entry lo + j lies at j sizeof(StagedRec)
        const int last0 = min(max(last[0] - lo, 0), kBwdBatch) * (int)sizeof(StagedRec);
        const int last1 = min(max(last[1] - lo, 0), kBwdBatch) * (int)sizeof(StagedRec);
        if (careful) walk_list<true>(sm, w, nw, ps, last0, last1, bx, by, drec);
        else walk_list<false>(sm, w, nw, ps, last0, last1, bx, by, drec);
    }
}

}  // namespace
}  // namespace ogs

using namespace ogs;

extern "C" ogs_status ogs_blend_bwd(const ogs_rec2d* rec, const uint32_t* pair_gauss,
                                    const uint32_t* tile_range, int32_t width, int32_t height,
                                    const float* bg, const float* T_final, const uint32_t* n_last,
                                    const float* dimg, float* drec, void* stream) {
    if (!rec || !pair_gauss || !tile_range || !bg || !T_final || !n_last || !dimg || !drec)
        return OGS_ERR_ARG;
    if (width <= 0 || height <= 0 || !aligned(rec, 16) || !aligned(tile_range, 8)) return OGS_ERR_ARG;
    const int gx = (width + kTile - 1) / kTile, gy = (height + kTile - 1) / kTile;
    if (cudaFuncSetAttribute(blend_bwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(BwdSmem)) != cudaSuccess)
        return OGS_ERR_CUDA;
    blend_bwd_kernel<<<gx * gy, blend::kThreads, sizeof(BwdSmem), (cudaStream_t)stream>>>(
        reinterpret_cast<const float4*>(rec), pair_gauss,
        reinterpret_cast<const uint2*>(tile_range), width, height, gx, bg[0], bg[1], bg[2],
        T_final, n_last, dimg, drec);
    return launch_status();
}
