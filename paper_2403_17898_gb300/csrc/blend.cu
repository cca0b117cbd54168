// Front-to-back alpha blending per 16x16 tile (Sec. 3.1, Eq. 2).
//
// One CTA of 4 warps per tile; each thread blends two vertically adjacent pixels (warps cover
// compact 8x8 blocks, so pixels that saturate together share a warp).  The tile's list is
// consumed in batches of 256 records gathered into shared memory, converted once per batch to
// pre-scaled coefficients and to a mask of the 8x8 blocks that the record's alpha >= 1/255
// ellipse can reach; each warp then walks, in list order, only the records whose mask holds
// its block.  One (pixel, Gaussian) evaluation is: offset, a 5-operation quadratic form, the
// exponent-bound skip test, one ex2 and the compositing update, done branch-free: a pixel that
// skips the Gaussian (or saturates on it) adds a zero weight and keeps its transmittance, which
// leaves its sums bit-for-bit as a skipped update would.  Lanes of a warp therefore never
// diverge inside the walk.  A warp stops walking once all its pixels have saturated (checked
// every 128 records) and the CTA stops loading batches once all of its pixels have.
//
// The kernel is bound by instruction issue (FP32, comparisons and selections), not by memory:
// about 50 instructions a visit of a warp to an entry, 83 % of the issue slots.  The skip test is
// one unsigned comparison on the negated exponent, saturation is the sign of T instead of a
// flag per pixel, and the 0.99 clamp is compiled in only for batches with an opacity that can
// reach it.  1080p, 2.1M list entries, with n_last: 230 -> 200 us; the 2M-anchor city frame's
// blend 165 -> 146 us.  (Packed FP32 pairs for T and the weights cost latency on the one chain
// that is serial, 208 us; list bytes read four at a time cost their unpacking, 233 us.)  Four
// entries are evaluated at a time for small images, whose few warps wait on latency.
// The optional n_eval
// output counts, per pixel, the (pixel, Gaussian) tests the kernel made while the pixel still
// needed them: the entries of its warp block's list up to the one it saturated on.
#include <type_traits>

#include "blend_common.cuh"

namespace ogs {
namespace {

using namespace blend;

constexpr int kExitEvery = 128;  // records walked between two warp-wide saturation checks
constexpr int kWalk = 4;         // entries evaluated at a time
static_assert(kBatch <= 256, "entries are listed as bytes");

// A thread's two vertically adjacent pixels.  T is the transmittance, negative once the pixel
// has saturated (or lies outside the image): T (1 - alpha) then falls below every bound by
// itself, so the walk needs no flag beside it.
struct Pixels {
    float fx, fy;                       // the upper one's coordinates
    float T[2], C[2][3];
    int last[2], tests[2];
    __device__ __forceinline__ bool done() const { return T[0] < 0.f && T[1] < 0.f; }
};

// One compositing step of both pixels with the list's entry number idx - 1, branch-free.
// wgt receives the weights alpha T added (0 where the pixel skipped the Gaussian or saturated on
// it).  kClamp: the entry's alpha can exceed 0.99.  Only T is carried from entry to entry:
// two products, a comparison and a selection.
template <bool kEval, bool kLast, bool kClamp>
__device__ __forceinline__ void composite(Pixels& p, const float (&q)[2], const float4& B,
                                          const float2& C, int idx, float (&wgt)[2]) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        if (kEval) p.tests[i] += p.T[i] < 0.f ? 0 : 1;          // a test this pixel still needed
        const bool pass = passes(q[i], C.y);                    // power <= 0 and alpha >= 1/255
        float alpha = __fmul_rn(B.y, ex2(-q[i]));
        if (kClamp) alpha = fminf(0.99f, alpha);
        const float w = __fmul_rn(alpha, p.T[i]);
        const float Tn = __fsub_rn(p.T[i], w);                  // T (1 - alpha)
        const bool apply = pass && Tn >= 1e-4f;                 // else it would saturate the pixel
        const float stay = pass ? -fabsf(p.T[i]) : p.T[i];
        wgt[i] = apply ? w : 0.0f;
        p.T[i] = apply ? Tn : stay;
        if (kLast) p.last[i] = apply ? idx : p.last[i];
        p.C[i][0] = fmaf(B.z, wgt[i], p.C[i][0]);
        p.C[i][1] = fmaf(B.w, wgt[i], p.C[i][1]);
        p.C[i][2] = fmaf(C.x, wgt[i], p.C[i][2]);
    }
}

// Walks the warp's list of nw staged entries front to back, kWalk of them evaluated at a time
// (independent up to the transmittance chain).
template <bool kMaxC, bool kEval, bool kLast, bool kClamp>
__device__ __forceinline__ void walk_list(Pixels& p, const StagedRec* s_rec, const uint8_t* list,
                                          int nw, int b0, const uint32_t* s_anchor,
                                          uint32_t* __restrict__ maxc) {
    auto step = [&](int i, auto n_) {
        constexpr int kN = decltype(n_)::value;
        float q[kN][2];
        float4 B[kN];
        float2 C[kN];
        int j[kN];
#pragma unroll
        for (int u = 0; u < kN; ++u) {
            j[u] = list[i + u];
            const StagedRec& r = s_rec[j[u]];
            const float4 A = r.A;
            B[u] = r.B;
            C[u] = *reinterpret_cast<const float2*>(&r.C);
            const float dx = A.x - p.fx, dy = A.y - p.fy, ax = __fmul_rn(A.z, dx);
            q[u][0] = power2(ax, dx, dy, A.w, B[u].x);
            q[u][1] = power2(ax, dx, dy - 1.0f, A.w, B[u].x);
        }
#pragma unroll
        for (int u = 0; u < kN; ++u) {
            float wgt[2];
            composite<kEval, kLast, kClamp>(p, q[u], B[u], C[u], b0 + j[u] + 1, wgt);
            if (kMaxC) {
                // contributions are >= 0, so their float bits order like unsigned ints
                const uint32_t m = __reduce_max_sync(0xffffffffu,
                                                     __float_as_uint(fmaxf(wgt[0], wgt[1])));
                if (lane_id() == 0 && m) atomicMax(&maxc[s_anchor[j[u]]], m);
            }
        }
    };
    for (int q0 = 0; q0 < nw; q0 += kExitEvery) {
        if (__all_sync(0xffffffffu, p.done())) break;
        const int q1 = min(q0 + kExitEvery, nw);
        int i = q0;
        for (; i + kWalk <= q1; i += kWalk)
            step(i, std::integral_constant<int, kWalk>());
        for (; i < q1; ++i) step(i, std::integral_constant<int, 1>());
    }
}

template <bool kMaxC, bool kEval, bool kLast>
__global__ void __launch_bounds__(kThreads) blend_fwd_kernel(
    const float4* __restrict__ rec, const uint32_t* __restrict__ pair_gauss,
    const uint2* __restrict__ tile_range, int W, int H, int gx, float bg0, float bg1, float bg2,
    float* __restrict__ img, float* __restrict__ T_final, uint32_t* __restrict__ n_last,
    uint32_t* __restrict__ n_eval, const uint32_t* __restrict__ sel_idx, int k,
    uint32_t* __restrict__ maxc) {
    pdl_wait();
    pdl_trigger();
    __shared__ StagedRec s_rec[kBatch];
    __shared__ uint8_t s_m[kBatch];
    __shared__ uint8_t s_list[kThreads / 32][kBatch];
    __shared__ uint32_t s_anchor[kMaxC ? kBatch : 1];
    const int tile = blockIdx.x;
    int lx, ly;
    pixels_of(threadIdx.x, lx, ly);
    const int tx0 = (tile % gx) * kTile, ty0 = (tile / gx) * kTile;
    const int px = tx0 + lx;
    const int py = ty0 + ly;
    const bool in0 = px < W && py < H, in1 = px < W && py + 1 < H;
    const uint2 range = tile_range[tile];
    const int n = (int)(range.y - range.x);
    uint8_t* list = s_list[threadIdx.x >> 5];
    Pixels p{(float)px, (float)py, {in0 ? 1.f : -1.f, in1 ? 1.f : -1.f},
             {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}}, {0, 0}, {0, 0}};
    for (int b0 = 0; b0 < n; b0 += kBatch) {
        if (__syncthreads_and(p.done())) break;
        bool clamp = false;
        for (int e = threadIdx.x; e < kBatch && b0 + e < n; e += kThreads) {
            const uint32_t g = pair_gauss[range.x + b0 + e];
            const uint32_t m = stage_rec(rec, g, (float)tx0, (float)ty0, s_rec[e]);
            s_m[e] = (uint8_t)m;
            clamp = clamp || (m & 16u);
            if (kMaxC) s_anchor[e] = sel_idx[g / (uint32_t)k];
        }
        clamp = __syncthreads_or(clamp);
        const int nw = warp_list<1>(s_m, min(kBatch, n - b0), list);
        if (clamp) walk_list<kMaxC, kEval, kLast, true>(p, s_rec, list, nw, b0, s_anchor, maxc);
        else walk_list<kMaxC, kEval, kLast, false>(p, s_rec, list, nw, b0, s_anchor, maxc);
    }
    const float T0 = fabsf(p.T[0]), T1 = fabsf(p.T[1]);
    const size_t plane = (size_t)W * H;
    if (in0) {
        const size_t pix = (size_t)py * W + px;
        img[pix] = p.C[0][0] + T0 * bg0;
        img[plane + pix] = p.C[0][1] + T0 * bg1;
        img[2 * plane + pix] = p.C[0][2] + T0 * bg2;
        T_final[pix] = T0;
        if (kLast) n_last[pix] = (uint32_t)p.last[0];
        if (kEval) n_eval[pix] = (uint32_t)p.tests[0];
    }
    if (in1) {
        const size_t pix = (size_t)(py + 1) * W + px;
        img[pix] = p.C[1][0] + T1 * bg0;
        img[plane + pix] = p.C[1][1] + T1 * bg1;
        img[2 * plane + pix] = p.C[1][2] + T1 * bg2;
        T_final[pix] = T1;
        if (kLast) n_last[pix] = (uint32_t)p.last[1];
        if (kEval) n_eval[pix] = (uint32_t)p.tests[1];
    }
}

}  // namespace
}  // namespace ogs

using namespace ogs;

extern "C" ogs_status ogs_blend_fwd(const ogs_rec2d* rec, const uint32_t* pair_gauss,
                                    const uint32_t* tile_range, int32_t width, int32_t height,
                                    const float* bg, float* img, float* T_final,
                                    uint32_t* n_last, uint32_t* n_eval, const uint32_t* sel_idx,
                                    int32_t k, uint32_t* maxc, void* stream) {
    if (!rec || !pair_gauss || !tile_range || !bg || !img || !T_final) return OGS_ERR_ARG;
    if (width <= 0 || height <= 0 || !aligned(rec, 16) || !aligned(tile_range, 8)) return OGS_ERR_ARG;
    if (maxc && (!sel_idx || k <= 0)) return OGS_ERR_ARG;
    const int gx = (width + kTile - 1) / kTile, gy = (height + kTile - 1) / kTile;
    cudaStream_t st = (cudaStream_t)stream;
    const float4* r = reinterpret_cast<const float4*>(rec);
    const uint2* tr = reinterpret_cast<const uint2*>(tile_range);
    const dim3 grid(gx * gy), block(blend::kThreads);
    const int variant = (maxc ? 4 : 0) | (n_eval ? 2 : 0) | (n_last ? 1 : 0);
#define OGS_BLEND(M, E, L)                                                                     \
    launch_pdl(blend_fwd_kernel<M, E, L>, grid, block, 0, st, r, pair_gauss, tr, width, height, \
               gx, bg[0], bg[1], bg[2], img, T_final, n_last, n_eval, sel_idx, k, maxc)
    switch (variant) {
        case 0: OGS_BLEND(false, false, false); break;
        case 1: OGS_BLEND(false, false, true); break;
        case 2: OGS_BLEND(false, true, false); break;
        case 3: OGS_BLEND(false, true, true); break;
        case 4: OGS_BLEND(true, false, false); break;
        case 5: OGS_BLEND(true, false, true); break;
        case 6: OGS_BLEND(true, true, false); break;
        default: OGS_BLEND(true, true, true); break;
    }
#undef OGS_BLEND
    return launch_status();
}
