// EWA projection of one 3D Gaussian to its screen-space record and 16x16 tile extent (Sec. 3.1,
// Eq. 1: Sigma = R S S^T R^T, projected with the local affine Jacobian), and the per-tile pair
// counting.  Shared by ogs_project_bin and the fused decode + projection, so both produce the
// same bits.
#pragma once

#include "internal.cuh"

namespace ogs {

struct ProjOut {
    float4 r0, r1, r2;   // the 48-byte record (zeros when the Gaussian is culled)
    uint32_t dkey;       // depth key (float bits of the camera-space depth), ~0 when culled
    uint32_t ntiles;     // tiles of its rectangle (0 when culled)
    uint2 rc;            // (x0 | y0 << 16, x1 | y1 << 16): tiles [x0, x1) x [y0, y1)
};

// Every product and sum below is an explicit round-to-nearest intrinsic, so the compiler cannot
// contract them differently in the kernels that inline this function.
__device__ __forceinline__ float pm(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float pa(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float pf(float a, float b, float c) { return __fmaf_rn(a, b, c); }
// a0 b0 + a1 b1 + a2 b2
__device__ __forceinline__ float dot3(float a0, float a1, float a2, float b0, float b1, float b2) {
    return pf(a2, b2, pf(a1, b1, pm(a0, b0)));
}

// m: camera-relative mean (world axes); q = (w, x, y, z) unit quaternion; s: scales; o: opacity
// (culled when o <= 0); col: colour.
__device__ __forceinline__ ProjOut project_one(const Cam& c, float m0, float m1, float m2,
                                               float4 q, float s0, float s1, float s2, float o,
                                               float col0, float col1, float col2) {
    ProjOut out;
    out.r0 = make_float4(0.f, 0.f, 0.f, 0.f);
    out.r1 = out.r0;
    out.r2 = out.r0;
    out.dkey = 0xFFFFFFFFu;
    out.ntiles = 0;
    out.rc = make_uint2(0, 0);
    if (!(o > 0.0f)) return out;
    const float px = dot3(c.R[0], c.R[1], c.R[2], m0, m1, m2);
    const float py = dot3(c.R[3], c.R[4], c.R[5], m0, m1, m2);
    const float pz = dot3(c.R[6], c.R[7], c.R[8], m0, m1, m2);
    if (!(pz > c.znear)) return out;
    const float w = q.x, x = q.y, y = q.z, z = q.w;
    const float xx = pm(x, x), yy = pm(y, y), zz = pm(z, z);
    const float xy = pm(x, y), xz = pm(x, z), yz = pm(y, z);
    const float wx = pm(w, x), wy = pm(w, y), wz = pm(w, z);
    // M = R(q) S
    const float M00 = pm(pf(-2.f, pa(yy, zz), 1.f), s0), M01 = pm(pm(2.f, pa(xy, -wz)), s1),
                M02 = pm(pm(2.f, pa(xz, wy)), s2);
    const float M10 = pm(pm(2.f, pa(xy, wz)), s0), M11 = pm(pf(-2.f, pa(xx, zz), 1.f), s1),
                M12 = pm(pm(2.f, pa(yz, -wx)), s2);
    const float M20 = pm(pm(2.f, pa(xz, -wy)), s0), M21 = pm(pm(2.f, pa(yz, wx)), s1),
                M22 = pm(pf(-2.f, pa(xx, yy), 1.f), s2);
    // Sigma = M M^T (symmetric)
    const float S00 = dot3(M00, M01, M02, M00, M01, M02);
    const float S01 = dot3(M00, M01, M02, M10, M11, M12);
    const float S02 = dot3(M00, M01, M02, M20, M21, M22);
    const float S11 = dot3(M10, M11, M12, M10, M11, M12);
    const float S12 = dot3(M10, M11, M12, M20, M21, M22);
    const float S22 = dot3(M20, M21, M22, M20, M21, M22);
    // Jacobian of the perspective map at the (frustum-clamped) centre
    const float iz = __frcp_rn(pz);
    const float tx = pm(fminf(fmaxf(pm(px, iz), -c.limx), c.limx), pz);
    const float ty = pm(fminf(fmaxf(pm(py, iz), -c.limy), c.limy), pz);
    const float iz2 = pm(iz, iz);
    const float j00 = pm(c.fx, iz), j02 = -pm(pm(c.fx, tx), iz2);
    const float j11 = pm(c.fy, iz), j12 = -pm(pm(c.fy, ty), iz2);
    // T = J W (2x3)
    const float T00 = pf(j02, c.R[6], pm(j00, c.R[0])), T01 = pf(j02, c.R[7], pm(j00, c.R[1])),
                T02 = pf(j02, c.R[8], pm(j00, c.R[2]));
    const float T10 = pf(j12, c.R[6], pm(j11, c.R[3])), T11 = pf(j12, c.R[7], pm(j11, c.R[4])),
                T12 = pf(j12, c.R[8], pm(j11, c.R[5]));
    // cov2 = T Sigma T^T
    const float U0 = dot3(S00, S01, S02, T00, T01, T02);
    const float U1 = dot3(S01, S11, S12, T00, T01, T02);
    const float U2 = dot3(S02, S12, S22, T00, T01, T02);
    const float V0 = dot3(S00, S01, S02, T10, T11, T12);
    const float V1 = dot3(S01, S11, S12, T10, T11, T12);
    const float V2 = dot3(S02, S12, S22, T10, T11, T12);
    const float ca = pa(dot3(T00, T01, T02, U0, U1, U2), 0.3f);
    const float cb = dot3(T10, T11, T12, U0, U1, U2);
    const float cc = pa(dot3(T10, T11, T12, V0, V1, V2), 0.3f);
    const float det = pf(ca, cc, -pm(cb, cb));
    if (!(det > 0.0f)) return out;
    const float mid = pm(0.5f, pa(ca, cc));
    const float lam = pa(mid, __fsqrt_rn(fmaxf(0.1f, pf(mid, mid, -det))));
    const float r = pm(3.0f, __fsqrt_rn(lam));
    const float u = pf(pm(c.fx, px), iz, c.cx);
    const float v = pf(pm(c.fy, py), iz, c.cy);
    // tiles holding a pixel centre inside [u-r, u+r] x [v-r, v+r]
    const float lo = -64.f, hix = 16.f * c.gx + 64.f, hiy = 16.f * c.gy + 64.f;
    const float ex0 = fminf(fmaxf(ceilf(pa(u, -r)), lo), hix);
    const float ex1 = fminf(fmaxf(floorf(pa(u, r)), lo), hix);
    const float ey0 = fminf(fmaxf(ceilf(pa(v, -r)), lo), hiy);
    const float ey1 = fminf(fmaxf(floorf(pa(v, r)), lo), hiy);
    const int tx0 = max((int)floorf(ex0 * 0.0625f), 0);
    const int tx1 = min((int)floorf(ex1 * 0.0625f) + 1, c.gx);
    const int ty0 = max((int)floorf(ey0 * 0.0625f), 0);
    const int ty1 = min((int)floorf(ey1 * 0.0625f) + 1, c.gy);
    if (!(tx0 < tx1 && ty0 < ty1)) return out;
    const float id = __frcp_rn(det);
    out.r0 = make_float4(u, v, pm(cc, id), -pm(cb, id));
    out.r1 = make_float4(pm(ca, id), o, col0, col1);
    // alpha = o G < 1/255  <=>  power < -ln(255 o): the blend tests the exponent against this
    // bound before evaluating exp
    out.r2 = make_float4(col2, pz, r, -logf(pm(255.0f, o)));
    out.dkey = __float_as_uint(pz);
    out.ntiles = (uint32_t)((tx1 - tx0) * (ty1 - ty0));
    out.rc = make_uint2((uint32_t)tx0 | ((uint32_t)ty0 << 16), (uint32_t)tx1 | ((uint32_t)ty1 << 16));
    return out;
}

// Adds every lane's rectangle to the per-tile counts.  All 32 lanes call it.  The first tile
// of each lane is added with one atomic per distinct tile of the warp (the k Gaussians of an
// anchor sit in consecutive lanes and mostly share it); the rest of a small rectangle by its
// lane, and rectangles of more than kOwnTiles tiles by the whole warp.
constexpr uint32_t kOwnTiles = 8;

// Row and column of tile i of a rectangle of width w and n tiles (row-major), without an integer
// division per tile: i / w by a product with 1 / w.  With n <= 2^20 the quotient (i + 1/2) / w lies
// at least 1 / (2 w) from a whole number and below n / w, so its relative error of 2^-22 cannot
// cross one; larger rectangles divide.  (1M Gaussians with 3.7 tiles each: projection with tile
// counts 67 -> 58 us; the small rectangles walk their rows instead of dividing.)
struct RectRows {
    uint32_t w;
    float inv;
    bool fast;
    __device__ __forceinline__ RectRows(uint32_t w_, uint32_t n) {
        w = w_;
        inv = __frcp_rn((float)w_);
        fast = n <= (1u << 20);
    }
    __device__ __forceinline__ uint32_t row(uint32_t i) const {
        return fast ? (uint32_t)(((float)i + 0.5f) * inv) : i / w;
    }
};

// Calls f(tile, k) for the tiles of a small rectangle (ntiles <= kOwnTiles) after its first, in
// order: k = 1 .. ntiles - 1, walked row by row.
template <class F>
__device__ __forceinline__ void for_own_tiles(uint32_t t0, uint32_t w, uint32_t ntiles, int gx, F f) {
    uint32_t kx = 0, t = t0;
#pragma unroll
    for (uint32_t i = 1; i < kOwnTiles; ++i) {
        if (++kx == w) {
            kx = 0;
            t += (uint32_t)gx - w + 1;
        } else {
            ++t;
        }
        if (i < ntiles) f(t, i);
    }
}

__device__ __forceinline__ void count_tiles(uint32_t* tc, int gx, uint2 rc, uint32_t ntiles) {
    const uint32_t x0 = rc.x & 0xFFFFu, y0 = rc.x >> 16, x1 = rc.y & 0xFFFFu;
    const uint32_t w = x1 - x0;
    const bool own = ntiles > 0 && ntiles <= kOwnTiles;
    const uint32_t t0 = own ? y0 * (uint32_t)gx + x0 : 0xFFFFFFFFu;
    const uint32_t peers = __match_any_sync(0xffffffffu, t0);
    if (own && lane_id() == (uint32_t)(__ffs(peers) - 1)) atomicAdd(tc + t0, (uint32_t)__popc(peers));
    if (own) for_own_tiles(t0, w, ntiles, gx, [&](uint32_t t, uint32_t) { atomicAdd(tc + t, 1u); });
    uint32_t big = __ballot_sync(0xffffffffu, ntiles > kOwnTiles);
    while (big) {
        const int src = __ffs(big) - 1;
        big &= big - 1;
        const uint2 r = make_uint2(__shfl_sync(0xffffffffu, rc.x, src),
                                   __shfl_sync(0xffffffffu, rc.y, src));
        const uint32_t bx0 = r.x & 0xFFFFu, by0 = r.x >> 16, bw = (r.y & 0xFFFFu) - bx0;
        const uint32_t bn = bw * ((r.y >> 16) - by0);
        const RectRows rr(bw, bn);
        for (uint32_t i = lane_id(); i < bn; i += 32) {
            const uint32_t row = rr.row(i);
            atomicAdd(tc + (by0 + row) * (uint32_t)gx + bx0 + (i - row * bw), 1u);
        }
    }
}

// Per-tile counts of many Gaussians: a CTA adds each rectangle's four corners (+1, -1, -1, +1) to a
// (gx + 1) x (gy + 1) table in shared memory and turns the table into counts by sums along the rows and
// then the columns, one coalesced atomic per tile that it met.  Four shared atomics whatever the
// rectangle's size, against one scattered atomic per pair in the L2, where the pairs of crowded tiles queue
// up and large rectangles hold their warp.  The rule: tables within the plain shared memory of a CTA
// and at most 256 tiles a side (the sums walk a side serially), and room for enough Gaussians to pay for
// clearing and summing: 16 per tile, where both took 10 us (4200 Gaussians on 256 tiles).  The room is
// the caller's capacity, since the view's count is on the device.  Projection, an atomic per pair ->
// corners: 41k Gaussians on 64 tiles 24 -> 10 us; 131k on 8160 tiles, 28 tiles each, 36 -> 20, and 1M
// of these 172 -> 40; 1M at 1080p with 6 tiles each 57 -> 30.  A sparse view in large buffers, kernel alone:
// 1080p, 500 Gaussians 6.7 -> 8.8 us, 8k 7.5 -> 9.5, 12k 16.5 -> 9.8, 24k 9.7 -> 9.5, 40k 16.5 -> 9.9; 128 x 128, 500
// 5.1 -> 5.9, 8k 5.7 -> 5.9, 12k 6.6 -> 6.0.  (Taking the atomic route in the kernel below 12k by the view's
// count gave those back and cost the dense views 4 %: 250k at 1080p 15.6 -> 16.2.)
constexpr int kCornerEntries = 12288, kCornerSide = 256;
constexpr int kCornerMinPerTile = 16;
inline int corner_entries(int gx, int gy) { return (gx + 1) * (gy + 1); }
inline bool use_corners(int64_t n_gauss, int gx, int gy) {
    return gx <= kCornerSide && gy <= kCornerSide && corner_entries(gx, gy) <= kCornerEntries &&
           n_gauss >= (int64_t)kCornerMinPerTile * gx * gy;
}
// All threads of the CTA call corner_clear and corner_flush, with a __syncthreads between them and
// the additions.
__device__ __forceinline__ void corner_clear(uint32_t* d, int gx, int gy) {
    for (int e = threadIdx.x; e < (gx + 1) * (gy + 1); e += blockDim.x) d[e] = 0u;
}
__device__ __forceinline__ void corner_add(uint32_t* d, int gx, uint2 rc) {
    const uint32_t p = (uint32_t)gx + 1;
    const uint32_t x0 = rc.x & 0xFFFFu, y0 = rc.x >> 16, x1 = rc.y & 0xFFFFu, y1 = rc.y >> 16;
    atomicAdd(d + y0 * p + x0, 1u);
    atomicAdd(d + y0 * p + x1, 0xFFFFFFFFu);
    atomicAdd(d + y1 * p + x0, 0xFFFFFFFFu);
    atomicAdd(d + y1 * p + x1, 1u);
}
__device__ __forceinline__ void corner_flush(uint32_t* d, int gx, int gy, uint32_t* tile_count) {
    const int p = gx + 1, lane = (int)lane_id();
    for (int y = threadIdx.x >> 5; y < gy; y += (int)blockDim.x >> 5) {     // a warp per row
        uint32_t carry = 0;
        for (int xb = 0; xb < gx; xb += 32) {
            const int x = xb + lane;
            uint32_t v = x < gx ? d[y * p + x] : 0u;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t u = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += u;
            }
            v += carry;
            if (x < gx) d[y * p + x] = v;
            carry = __shfl_sync(0xffffffffu, v, 31);
        }
    }
    __syncthreads();
    for (int x = threadIdx.x; x < gx; x += blockDim.x) {                    // a thread per column
        uint32_t s = 0;
        for (int yb = 0; yb < gy; yb += 8) {
            uint32_t v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = yb + i < gy ? d[(yb + i) * p + x] : 0u;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                s += v[i];
                if (yb + i < gy && s != 0u) atomicAdd(tile_count + (size_t)(yb + i) * gx + x, s);
            }
        }
    }
}

// Rectangles of more than kOwnTiles tiles go through the whole warp in chunks of kChunkTiles
// tiles.  bin_tiles hands each chunk to a list of deferred (Gaussian, chunk) entries that a
// second pass spreads over the whole grid, so that a warp holding many large near-camera
// Gaussians does not walk all their tiles alone; chunks that find the list full stay with
// the warp.
constexpr uint32_t kChunkTiles = 1024;

// Places tiles [lo, hi) of rectangle r (row-major inside it) for Gaussian g with key k: every
// lane of the warp takes one tile in 32, kFly atomics in flight before the stores.  All 32
// lanes call it with the same arguments.
template <uint32_t kFly>
__device__ __forceinline__ void bin_rect_range(uint32_t* tc, int gx, uint2 r, uint32_t lo,
                                               uint32_t hi, uint32_t g, uint32_t k,
                                               uint32_t cap, uint32_t* __restrict__ pair_key,
                                               uint32_t* __restrict__ pair_gauss) {
    const uint32_t bx0 = r.x & 0xFFFFu, by0 = r.x >> 16, bw = (r.y & 0xFFFFu) - bx0;
    const RectRows rr(bw, hi);
    for (uint32_t i0 = lo; i0 < hi; i0 += 32 * kFly) {
        uint32_t tt[kFly], sl[kFly];
#pragma unroll
        for (uint32_t j = 0; j < kFly; ++j) {
            const uint32_t i = i0 + j * 32 + lane_id();
            if (i < hi) {
                const uint32_t row = rr.row(i);
                tt[j] = (by0 + row) * (uint32_t)gx + bx0 + (i - row * bw);
                sl[j] = atomicAdd(tc + tt[j], 1u);
            }
        }
#pragma unroll
        for (uint32_t j = 0; j < kFly; ++j) {
            const uint32_t i = i0 + j * 32 + lane_id();
            if (i < hi && sl[j] < cap) {
                const size_t o = (size_t)tt[j] * cap + sl[j];
                pair_gauss[o] = g;
                pair_key[o] = k;
            }
        }
    }
}

// count_tiles, and each pair placed at once: the atomic that counts a (Gaussian, tile) pair
// returns its slot in the tile's region of cap entries, where the Gaussian's id and depth key
// go (pair_gauss[t * cap + slot], pair_key[...]); slots at or past cap are counted, not
// written (the caller sees the overflow in the counts).  g and dkey are the lane's Gaussian.
// A lane issues all its atomics (up to kOwnTiles at a time) before the first store that needs
// a slot, so their round trips overlap instead of adding up.  A larger rectangle is cut into
// chunks of kChunkTiles tiles, appended as (g, chunk) to `defer` (defer_cap entries, the
// 64-bit counter n_defer counts every chunk offered); chunks past defer_cap are placed here.
__device__ __forceinline__ void bin_tiles(uint32_t* tc, int gx, uint2 rc, uint32_t ntiles,
                                          uint32_t g, uint32_t dkey, uint32_t cap,
                                          uint32_t* __restrict__ pair_key,
                                          uint32_t* __restrict__ pair_gauss,
                                          uint2* __restrict__ defer,
                                          unsigned long long* n_defer, uint32_t defer_cap) {
    const uint32_t x0 = rc.x & 0xFFFFu, y0 = rc.x >> 16, x1 = rc.y & 0xFFFFu;
    const uint32_t w = x1 - x0;
    const uint32_t lane = lane_id();
    // large rectangles first (their list state is dead before the small ones' slots are live)
    const bool is_big = ntiles > kOwnTiles;
    if (__any_sync(0xffffffffu, is_big)) {
        // chunks of the lane's rectangle, numbered across the warp by an inclusive scan
        const uint32_t bn = is_big ? w * ((rc.y >> 16) - y0) : 0;
        const uint32_t nch = (bn + kChunkTiles - 1) / kChunkTiles;
        uint32_t incl = nch;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
            if ((int)lane >= o) incl += v;
        }
        const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
        unsigned long long first = 0;
        if (lane == 0) first = atomicAdd(n_defer, (unsigned long long)total);
        first = __shfl_sync(0xffffffffu, first, 0);
        const unsigned long long mine = first + (incl - nch);    // this lane's first entry
        uint32_t kept = 0;                                       // chunks the list took
        if (mine < (unsigned long long)defer_cap) {
            const unsigned long long room = (unsigned long long)defer_cap - mine;
            kept = room < nch ? (uint32_t)room : nch;
        }
        for (uint32_t c = 0; c < kept; ++c) defer[mine + c] = make_uint2(g, c);
        // what the list could not take stays with the warp, one rectangle at a time (four
        // atomics in flight per lane: this path is rare and keeps the kernel's registers low)
        const uint32_t lo = kept * kChunkTiles;
        uint32_t left = __ballot_sync(0xffffffffu, lo < bn);
        while (left) {
            const int src = __ffs(left) - 1;
            left &= left - 1;
            const uint2 r = make_uint2(__shfl_sync(0xffffffffu, rc.x, src),
                                       __shfl_sync(0xffffffffu, rc.y, src));
            bin_rect_range<4>(tc, gx, r, __shfl_sync(0xffffffffu, lo, src),
                           __shfl_sync(0xffffffffu, bn, src), __shfl_sync(0xffffffffu, g, src),
                           __shfl_sync(0xffffffffu, dkey, src), cap, pair_key, pair_gauss);
        }
    }
    auto put = [&](uint32_t t, uint32_t slot) {
        if (slot < cap) {
            const size_t o = (size_t)t * cap + slot;
            pair_gauss[o] = g;
            pair_key[o] = dkey;
        }
    };
    const bool own = ntiles > 0 && ntiles <= kOwnTiles;
    const uint32_t t0 = own ? y0 * (uint32_t)gx + x0 : 0xFFFFFFFFu;
    const uint32_t peers = __match_any_sync(0xffffffffu, t0);
    const uint32_t leader = __ffs(peers) - 1;
    uint32_t base = 0;
    if (own && lane == leader) base = atomicAdd(tc + t0, (uint32_t)__popc(peers));
    if (own) {
        uint32_t tt[kOwnTiles], sl[kOwnTiles];
        for_own_tiles(t0, w, ntiles, gx, [&](uint32_t t, uint32_t i) {
            tt[i] = t;
            sl[i] = atomicAdd(tc + t, 1u);
        });
#pragma unroll
        for (uint32_t i = 1; i < kOwnTiles; ++i)
            if (i < ntiles) put(tt[i], sl[i]);
    }
    base = __shfl_sync(0xffffffffu, base, leader);
    if (own) put(t0, base + __popc(peers & lanemask_lt()));
}

}  // namespace ogs
