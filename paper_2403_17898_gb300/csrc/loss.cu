// Photometric loss of Sec. 5.1.5: (1 - lambda) L1 + lambda (1 - SSIM), lambda = 0.2, SSIM with
// an 11x11 Gaussian window (sigma 1.5, separable, zero padded) and the usual C1 = 0.01^2,
// C2 = 0.03^2 (Wang et al. 2004), and its gradient with respect to the rendered image.
//
// With m1 = G*x, m2 = G*x^2, m3 = G*(x y) and the SSIM map S = A1 A2 / (B1 B2) (A1 = 2 m1 my
// + C1, A2 = 2 (m3 - m1 my) + C2, B1 = m1^2 + my^2 + C1, B2 = m2 - m1^2 + sy^2 + C2):
//   dS/dm1 = 2 my (A2 - A1)/(B1 B2) + 2 S m1 (1/B2 - 1/B1),  dS/dm2 = -S/B2,  dS/dm3 = 2 A1/(B1 B2),
// and for the mean SSIM:  d/dx = G*g1 + 2 x (G*g2) + y (G*g3), g_i = dS/dm_i / n.
// Two passes (moments -> SSIM map and partial maps; blur of the partial maps -> gradient).  A
// training loop that renders against fixed targets can compute the target's two moments once
// (ogs_ssim_target_stats) and pass them in, so that the forward pass blurs three moments instead
// of five.
//
// All but large images go by 32 x 32 tiles (ssim_tile below), large ones by column strips: both passes
// are then the same walk, a warp owns a strip of 64 columns (two per lane) and marches
// down its rows.  A row pair of the inputs (with a kRad halo; zero outside the image: the
// zero-padded window) passes through a warp-private shared buffer, is blurred horizontally with
// its two rows packed in one register pair, and enters the vertical blur at once: ten partial
// sums per moment live in registers and each row adds its tap to all of them while shifting them
// by one (the shift is the destination of the fused multiply-add), packed over the lane's two
// columns.  Nothing blurred goes through memory, and no warp waits for another.  Bound by the FP32
// pipes (66 packed operations per row, two columns and three moments) and the partial maps'
// traffic.  1080p: forward 57 -> 44 us, backward 54 -> 41 us against tiles as they then were, which
// spent 250 instructions on a pixel (strips 142 and 121); the blurs of both forms sum in the same
// order.  The next row pair is copied asynchronously while the current one is blurred
// (loads into registers were sunk to their use: 71 and 48 us).  The last strip (or tile) of the
// gradient adds the loss, which was a launch of its own.
#include <cmath>

#include "internal.cuh"

namespace ogs {
namespace {

constexpr int kWin = 11;
constexpr int kRad = kWin / 2;
constexpr float kC1 = 0.01f * 0.01f;
constexpr float kC2 = 0.03f * 0.03f;

struct Win {
    float w[kWin];
};

Win make_window() {
    Win g;
    double s = 0.0, t[kWin];
    for (int i = 0; i < kWin; ++i) {
        const double x = i - kRad;
        t[i] = std::exp(-x * x / (2.0 * 1.5 * 1.5));
        s += t[i];
    }
    for (int i = 0; i < kWin; ++i) g.w[i] = (float)(t[i] / s);
    return g;
}

constexpr int kCols = 64;                  // columns of a strip, two per lane
constexpr int kStripWarps = 2;             // strips (one below the other) per CTA
constexpr int kSpan = kCols + 2 * kRad;    // 74 input columns
constexpr int kBufCols = 76;

enum Pass { kMoments3, kMoments5, kGradient, kTargetStats };
__host__ __device__ constexpr int pass_inputs(Pass p) { return p == kGradient ? 3 : (p == kTargetStats ? 1 : 2); }
__host__ __device__ constexpr int pass_moments(Pass p) { return p == kMoments5 ? 5 : (p == kTargetStats ? 2 : 3); }

// Sums over the image, zeroed by the call.  In 64 bits: a thousand strips add to each.
struct LossSums {
    double ssim, l1;
    unsigned int done;      // strips or tiles whose gradient is finished
};

struct StripArgs {
    const float* in[3];     // planes [C][H][W] that are blurred (or whose products are)
    const float* x;         // kGradient: image and target
    const float* y;
    const float* ystat;     // kMoments3: the target's moments [2][C][H][W]
    float* out;             // partial maps [3][C][H][W] / gradient [C][H][W] / moments [2][C][H][W]
    LossSums* sums;
    float* loss;            // kGradient: the loss is added here (may be null)
    Win g;
    int H, W, rows;         // rows of a strip
    int64_t n;              // C H W
    float inv_n, lam;
    unsigned int parts;     // strips or tiles of the launch
    int vec;                // W even and every plane 8-byte aligned: a lane's columns as one vector
};

// Asynchronous 4- and 8-byte copies global -> shared; bytes = 0 reads nothing and writes zeros.
__device__ __forceinline__ void copy4(float* dst, const float* src, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;"
                 :: "r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void copy8(float* dst, const float* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;"
                 :: "r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ f32x2 shared2(const float* p) {
    const float2 v = *reinterpret_cast<const float2*>(p);
    return pack2(v.x, v.y);
}

// the lane's two columns of a row, packed (in1: the second lies in the image)
__device__ __forceinline__ void store2(float* p, f32x2 v, bool in1, int vec) {
    if (vec) {
        *reinterpret_cast<float2*>(p) = make_float2(lo2(v), hi2(v));
    } else {
        p[0] = lo2(v);
        if (in1) p[1] = hi2(v);
    }
}
__device__ __forceinline__ f32x2 both(float v) { return pack2(v, v); }
// reciprocals, a few ulp: two of them in place of seven divisions per pixel
__device__ __forceinline__ f32x2 rcp2(f32x2 v) { return pack2(rcp(lo2(v)), rcp(hi2(v))); }

// The lane's two pixels of the forward pass from their moments: the SSIM values and the partial
// maps gp_i = dS/dm_i / n.  With q = 1 / (B1 B2), S/A1 = A2 q and S/A2 = A1 q, so nothing is divided by
// A1 or A2: where the covariance passes -C2 / 2, A2 now and then rounds to exactly 0 (about one 1080p
// image pair in a hundred has such a pixel), and S times its reciprocal would be 0 x inf there.
__device__ __forceinline__ f32x2 ssim_pixels(f32x2 mx, f32x2 my, f32x2 exx, f32x2 eyy, f32x2 exy,
                                             float inv_n, f32x2& g0, f32x2& g1, f32x2& g2) {
    const f32x2 nx = mul2(mx, both(-1.f)), ny = mul2(my, both(-1.f));
    const f32x2 vx = fma2(nx, mx, exx), vy = fma2(ny, my, eyy), vxy = fma2(nx, my, exy);
    const f32x2 A1 = fma2(add2(mx, mx), my, both(kC1)), A2 = add2(add2(vxy, vxy), both(kC2));
    const f32x2 B1 = add2(fma2(mx, mx, mul2(my, my)), both(kC1));
    const f32x2 B2 = add2(add2(vx, vy), both(kC2));
    const f32x2 iB1 = rcp2(B1), iB2 = rcp2(B2), q = mul2(iB1, iB2);
    const f32x2 S = mul2(mul2(A1, A2), q);
    const f32x2 sn = mul2(S, both(inv_n)), qn = mul2(q, both(2.f * inv_n));
    g0 = fma2(mul2(my, sub2(A2, A1)), qn, mul2(mul2(add2(sn, sn), mx), sub2(iB2, iB1)));
    g1 = mul2(mul2(sn, both(-1.f)), iB2);
    g2 = mul2(A1, qn);
    return S;
}

// Adds one part's sum of the SSIM map (kMoments) or of |x - y| (kGradient) to the image's.  The last
// part of the gradient: loss = (1 - lam) * mean |x - y| + lam * (1 - mean SSIM).
template <Pass kPass>
__device__ __forceinline__ void add_sum(const StripArgs& a, float local) {
    atomicAdd(kPass == kGradient ? &a.sums->l1 : &a.sums->ssim, (double)local);
    if (kPass == kGradient && a.loss) {
        __threadfence();
        if (atomicAdd(&a.sums->done, 1u) == a.parts - 1) {
            __threadfence();
            const double l1 = *(volatile double*)&a.sums->l1;
            const double ssim = *(volatile double*)&a.sums->ssim, n = (double)a.n;
            *a.loss += (float)((1.0 - a.lam) * l1 / n + a.lam * (1.0 - ssim / n));
        }
    }
}

// kMoments: moments -> SSIM map (summed) and the three partial maps.  The five moments are G*x,
// G*y, G*x^2, G*y^2, G*xy; kMoments3 takes the target's two from ystat.
// kGradient: blur of the partial maps -> dSSIM/dx = G*gp0 + 2 x (G*gp1) + y (G*gp2);
// out = (1 - lam) sign(x - y) / n - lam dSSIM/dx, and the L1 sum.
// kTargetStats: G*y and G*y^2.
// CTAs per SM that the registers allow: 144 for kMoments3, 156 for kGradient, 166 for kMoments5.  More CTAs at 128 registers recompute what they cannot keep: 8 CTAs 50 and 48 us.
constexpr int kCtas = 6;
template <Pass kPass>
__global__ void __launch_bounds__(32 * kStripWarps, kCtas) ssim_strip(StripArgs a) {
    constexpr int kIn = pass_inputs(kPass), kM = pass_moments(kPass);
    constexpr bool kExtra = kPass == kMoments3 || kPass == kGradient;
    // a row pair of the inputs, the two rows of a column together; what its epilogue reads
    __shared__ __align__(16) float2 s_buf[kStripWarps][2][kIn][kBufCols];
    __shared__ __align__(16) float s_ext[kStripWarps][2][kExtra ? 4 * kCols : 1];
    pdl_wait();
    pdl_trigger();
    const int lane = (int)lane_id(), w = threadIdx.x >> 5;
    const int y0 = (int)(blockIdx.y * kStripWarps + w) * a.rows;
    if (y0 >= a.H) return;                                 // whole warps; no block barrier below
    const int y1 = min(y0 + a.rows, a.H);
    const int xs = (int)blockIdx.x * kCols;
    const int64_t plane = (int64_t)blockIdx.z * a.H * a.W;
    const int gx = xs + 2 * lane;                          // this lane's output columns gx, gx + 1
    const bool in0 = gx < a.W, in1 = gx + 1 < a.W;
    f32x2 wt[kWin];                                        // the window is symmetric: six pairs
#pragma unroll
    for (int k = 0; k < kWin; ++k) wt[k] = pack2(a.g.w[k < kRad ? k : kWin - 1 - k],
                                                 a.g.w[k < kRad ? k : kWin - 1 - k]);
    int cin[3];                                            // bytes of input column lane + 32 q
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int col = lane + 32 * q, cx = xs - kRad + col;
        cin[q] = col < kSpan && cx >= 0 && cx < a.W ? 4 : 0;
    }
    const int nr = y1 - y0 + 2 * kRad;                     // input rows of the strip
    // the lane's first input column in the next row to be copied, and its output columns in the
    // epilogue's operands of the output row that the copied row completes
    const int64_t at = plane + (int64_t)(y0 - kRad) * a.W + xs - kRad + lane;
    const float* pin[kIn];
#pragma unroll
    for (int j = 0; j < kIn; ++j) pin[j] = a.in[j] + at;
    const int64_t o = plane + (int64_t)(y0 - 2 * kRad) * a.W + gx;
    const float* ext[2] = {(kPass == kGradient ? a.x : a.ystat) + o,
                           (kPass == kGradient ? a.y : a.ystat + a.n) + o};
    // copies input rows r, r + 1 of the strip into buffer b, zero outside the image, with the
    // epilogue's operands of output rows r - 2 kRad, r + 1 - 2 kRad
    auto fetch = [&](int r, int b) {
        float* buf = reinterpret_cast<float*>(&s_buf[w][b][0][lane]);
        float* eb = &s_ext[w][b][kExtra ? 2 * lane : 0];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const bool rin = (unsigned)(y0 - kRad + r + h) < (unsigned)a.H;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int bytes = rin ? cin[q] : 0;
                if (q < 2 || lane < kBufCols - 64)
#pragma unroll
                    for (int j = 0; j < kIn; ++j)
                        copy4(buf + 2 * (kBufCols * j + 32 * q) + h, pin[j] + 32 * q, bytes);
            }
#pragma unroll
            for (int j = 0; j < kIn; ++j) pin[j] += a.W;
            if (kExtra) {
                if (r >= 2 * kRad && r + h < nr && in0) {
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        float* d = eb + (2 * j + h) * kCols;
                        if (a.vec) {
                            copy8(d, ext[j]);
                        } else {
                            copy4(d, ext[j], 4);
                            copy4(d + 1, ext[j] + 1, in1 ? 4 : 0);
                        }
                    }
                }
#pragma unroll
                for (int j = 0; j < 2; ++j) ext[j] += a.W;
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    f32x2 acc[kM][kWin - 1];
#pragma unroll
    for (int j = 0; j < kM; ++j)
#pragma unroll
        for (int k = 0; k < kWin - 1; ++k) acc[j][k] = 0;
    float local = 0.f;
    fetch(0, 0);
    float* out[3] = {a.out + o, a.out + a.n + o, a.out + 2 * a.n + o};
    for (int r = 0; r < nr; r += 2) {
        const int b = (r >> 1) & 1;
        __syncwarp();                                      // the other buffer has been read
        if (r + 2 < nr) fetch(r + 2, b ^ 1);
        else asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();                                      // every lane's copies have landed
        const float2(*buf)[kBufCols] = s_buf[w][b];
        // horizontal blur of both rows (packed) for the lane's two columns
        f32x2 hb[kM][2];
#pragma unroll
        for (int j = 0; j < kM; ++j) hb[j][0] = hb[j][1] = 0;
#pragma unroll
        for (int k2 = 0; k2 < kWin + 1; k2 += 2) {
            float4 v4[kIn];
#pragma unroll
            for (int j = 0; j < kIn; ++j)
                v4[j] = *reinterpret_cast<const float4*>(&buf[j][2 * lane + k2]);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int k = k2 + u;
                f32x2 in[kIn], ch[kM];
#pragma unroll
                for (int j = 0; j < kIn; ++j)
                    in[j] = u ? pack2(v4[j].z, v4[j].w) : pack2(v4[j].x, v4[j].y);
                if (kPass == kMoments3) {
                    ch[0] = in[0]; ch[1] = mul2(in[0], in[0]); ch[2] = mul2(in[0], in[1]);
                } else if (kPass == kMoments5) {
                    ch[0] = in[0]; ch[1] = in[1]; ch[2] = mul2(in[0], in[0]);
                    ch[kM - 2] = mul2(in[1], in[1]); ch[kM - 1] = mul2(in[0], in[1]);
                } else if (kPass == kTargetStats) {
                    ch[0] = in[0]; ch[1] = mul2(in[0], in[0]);
                } else {
#pragma unroll
                    for (int j = 0; j < kM; ++j) ch[j] = in[j < kIn ? j : 0];
                }
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    const int tap = k - t;
                    if (tap < 0 || tap >= kWin) continue;
#pragma unroll
                    for (int j = 0; j < kM; ++j) hb[j][t] = fma2(wt[tap], ch[j], hb[j][t]);
                }
            }
        }
        // vertical blur, one row at a time, both columns packed
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            f32x2 m[kM];
#pragma unroll
            for (int j = 0; j < kM; ++j) {
                const f32x2 v = h ? pack2(hi2(hb[j][0]), hi2(hb[j][1]))
                                  : pack2(lo2(hb[j][0]), lo2(hb[j][1]));
                m[j] = fma2(wt[kWin - 1], v, acc[j][0]);
#pragma unroll
                for (int k = 0; k < kWin - 2; ++k) acc[j][k] = fma2(wt[kWin - 2 - k], v, acc[j][k + 1]);
                acc[j][kWin - 2] = fma2(wt[0], v, 0);
            }
            const bool write = r >= 2 * kRad && r + h < nr && in0;
            f32x2 e0 = 0, e1 = 0;
            if (kExtra && write) {
                e0 = shared2(&s_ext[w][b][kExtra ? h * kCols + 2 * lane : 0]);
                e1 = shared2(&s_ext[w][b][kExtra ? (2 + h) * kCols + 2 * lane : 0]);
            }
            if (!write) {
            } else if (kPass == kTargetStats) {
                store2(out[0], m[0], in1, a.vec);
                store2(out[1], m[1], in1, a.vec);
            } else if (kPass == kGradient) {
                const f32x2 df = sub2(e0, e1);
                const float d0 = lo2(df), d1 = hi2(df);
                local += fabsf(d0) + (in1 ? fabsf(d1) : 0.f);
                const f32x2 sgn = pack2(d0 > 0.f ? a.inv_n : (d0 < 0.f ? -a.inv_n : 0.f),
                                        d1 > 0.f ? a.inv_n : (d1 < 0.f ? -a.inv_n : 0.f));
                const f32x2 dssim = fma2(e1, m[kM - 1], fma2(add2(e0, e0), m[1], m[0]));
                store2(out[0], fma2(both(-a.lam), dssim, mul2(both(1.f - a.lam), sgn)), in1, a.vec);
            } else {
                const bool c3 = kPass == kMoments3;
                f32x2 g0, g1, g2;
                const f32x2 S = ssim_pixels(m[0], c3 ? e0 : m[1], c3 ? m[1] : m[2 % kM],
                                            c3 ? e1 : m[3 % kM], m[kM - 1], a.inv_n, g0, g1, g2);
                local += lo2(S) + (in1 ? hi2(S) : 0.f);
                store2(out[0], g0, in1, a.vec);
                store2(out[1], g1, in1, a.vec);
                store2(out[2], g2, in1, a.vec);
            }
#pragma unroll
            for (int j = 0; j < 3; ++j) out[j] += a.W;
        }
    }
    if (kPass != kTargetStats) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) local += __shfl_xor_sync(0xffffffffu, local, o);
        if (lane == 0) add_sum<kPass>(a, local);
    }
}

// The same passes by tiles, for all but large images: a CTA owns 32 x 32 outputs of one channel, stages
// them with their halo in shared memory, blurs horizontally into shared memory and vertically into
// registers (four outputs along the blur per thread from fourteen loaded inputs).  A tile blurs 1.3 rows
// for each that it keeps, where a strip of ten rows blurs two.  A large image gives strips of more rows,
// and the tiles' second trip through shared memory loses to them.
constexpr int kTX = 32, kTY = 32;
constexpr int kHX = kTX + 2 * kRad, kHY = kTY + 2 * kRad;   // 42 x 42 staged inputs
constexpr int kTileThreads = 256;
constexpr int kRun = 4;                                    // outputs of a thread along a blur
constexpr int kRunSpan = kRun + kWin - 1;                  // their inputs
static_assert(kTX * (kTY / kRun) == kTileThreads, "a vertical run per thread");

template <Pass kPass>
__global__ void __launch_bounds__(kTileThreads) ssim_tile(StripArgs a) {
    constexpr int kIn = pass_inputs(kPass), kM = pass_moments(kPass);
    static_assert(kPass != kTargetStats, "strips only");
    __shared__ float s_in[kIn][kHY][kHX + 1];
    __shared__ float s_h[kM][kHY][kTX + 1];
    __shared__ float s_red[kTileThreads / 32];
    pdl_wait();
    pdl_trigger();
    const int x0 = blockIdx.x * kTX - kRad, y0 = blockIdx.y * kTY - kRad;
    const int64_t plane = (int64_t)blockIdx.z * a.H * a.W;
    {
        // 6 rows of 42 columns at a time (threads 252 .. 255 idle), every load before any store
        constexpr int kRowsPer = kTileThreads / kHX, kTimes = (kHY + kRowsPer - 1) / kRowsPer;
        const int q = threadIdx.x % kHX, r0 = threadIdx.x / kHX, gx = x0 + q;
        float v[kIn][kTimes];
#pragma unroll
        for (int k = 0; k < kTimes; ++k) {
            const int r = r0 + kRowsPer * k, gy = y0 + r;
            const bool in = r0 < kRowsPer && r < kHY && gx >= 0 && gx < a.W && gy >= 0 && gy < a.H;
            const int64_t i = plane + (int64_t)gy * a.W + gx;
#pragma unroll
            for (int j = 0; j < kIn; ++j) v[j][k] = in ? a.in[j][i] : 0.f;
        }
#pragma unroll
        for (int k = 0; k < kTimes; ++k)
#pragma unroll
            for (int j = 0; j < kIn; ++j)
                if (r0 < kRowsPer && r0 + kRowsPer * k < kHY) s_in[j][r0 + kRowsPer * k][q] = v[j][k];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < kHY * (kTX / kRun); e += kTileThreads) {
        const int r = e / (kTX / kRun), q0 = e % (kTX / kRun) * kRun;
        float acc[kM][kRun];
#pragma unroll
        for (int j = 0; j < kM; ++j)
#pragma unroll
            for (int t = 0; t < kRun; ++t) acc[j][t] = 0.f;
#pragma unroll
        for (int k = 0; k < kRunSpan; ++k) {
            float u[kIn], ch[kM];
#pragma unroll
            for (int j = 0; j < kIn; ++j) u[j] = s_in[j][r][q0 + k];
            if (kPass == kGradient) {
#pragma unroll
                for (int j = 0; j < kM; ++j) ch[j] = u[j < kIn ? j : 0];
            } else {
                ch[0] = u[0];
                ch[kPass == kMoments3 ? 1 : 2] = u[0] * u[0];
                ch[kM - 1] = u[0] * u[1];
                if (kPass == kMoments5) {
                    ch[1] = u[1];
                    ch[kM - 2] = u[1] * u[1];
                }
            }
#pragma unroll
            for (int t = 0; t < kRun; ++t) {
                const int tap = k - t;
                if (tap < 0 || tap >= kWin) continue;
#pragma unroll
                for (int j = 0; j < kM; ++j) acc[j][t] = fmaf(a.g.w[tap], ch[j], acc[j][t]);
            }
        }
#pragma unroll
        for (int t = 0; t < kRun; ++t)
#pragma unroll
            for (int j = 0; j < kM; ++j) s_h[j][r][q0 + t] = acc[j][t];
    }
    __syncthreads();
    const int qc = threadIdx.x % kTX, r0 = threadIdx.x / kTX * kRun;       // one run per thread
    const int gx = x0 + kRad + qc, gy = y0 + kRad + r0;
    const int64_t i0 = plane + (int64_t)gy * a.W + gx;
    // what the epilogue reads, loaded before the blur: the target's moments, or image and target
    float ext[2][kRun];
    if (kPass != kMoments5) {
        const float* src[2] = {kPass == kGradient ? a.x : a.ystat, kPass == kGradient ? a.y : a.ystat + a.n};
#pragma unroll
        for (int t = 0; t < kRun; ++t)
#pragma unroll
            for (int j = 0; j < 2; ++j)
                ext[j][t] = gx < a.W && gy + t < a.H ? src[j][i0 + (int64_t)t * a.W] : 0.f;
    }
    float m[kM][kRun];
#pragma unroll
    for (int j = 0; j < kM; ++j)
#pragma unroll
        for (int t = 0; t < kRun; ++t) m[j][t] = 0.f;
#pragma unroll
    for (int k = 0; k < kRunSpan; ++k) {
        float h[kM];
#pragma unroll
        for (int j = 0; j < kM; ++j) h[j] = s_h[j][r0 + k][qc];
#pragma unroll
        for (int t = 0; t < kRun; ++t) {
            const int tap = k - t;
            if (tap < 0 || tap >= kWin) continue;
#pragma unroll
            for (int j = 0; j < kM; ++j) m[j][t] = fmaf(a.g.w[tap], h[j], m[j][t]);
        }
    }
    float local = 0.f;
#pragma unroll
    for (int t = 0; t < kRun; t += 2) {                                    // two rows, packed
        const bool in0 = gx < a.W && gy + t < a.H, in1 = gx < a.W && gy + t + 1 < a.H;
        const int64_t i[2] = {i0 + (int64_t)t * a.W, i0 + (int64_t)(t + 1) * a.W};
        auto pair = [&](int j) { return pack2(m[j][t], m[j][t + 1]); };
        f32x2 g[3];
        if (kPass == kGradient) {
            const f32x2 x = pack2(ext[0][t], ext[0][t + 1]), y = pack2(ext[1][t], ext[1][t + 1]);
            const f32x2 df = sub2(x, y);
            const float d0 = lo2(df), d1 = hi2(df);
            local += (in0 ? fabsf(d0) : 0.f) + (in1 ? fabsf(d1) : 0.f);
            const f32x2 sgn = pack2(d0 > 0.f ? a.inv_n : (d0 < 0.f ? -a.inv_n : 0.f),
                                    d1 > 0.f ? a.inv_n : (d1 < 0.f ? -a.inv_n : 0.f));
            const f32x2 dssim = fma2(y, pair(kM - 1), fma2(add2(x, x), pair(1), pair(0)));
            g[0] = fma2(both(-a.lam), dssim, mul2(both(1.f - a.lam), sgn));
        } else {
            constexpr bool c3 = kPass == kMoments3;
            const f32x2 S = ssim_pixels(pair(0), c3 ? pack2(ext[0][t], ext[0][t + 1]) : pair(1),
                                        c3 ? pair(1) : pair(2), c3 ? pack2(ext[1][t], ext[1][t + 1]) : pair(kM - 2),
                                        pair(kM - 1), a.inv_n, g[0], g[1], g[2]);
            local += (in0 ? lo2(S) : 0.f) + (in1 ? hi2(S) : 0.f);
        }
#pragma unroll
        for (int j = 0; j < (kPass == kGradient ? 1 : 3); ++j) {
            if (in0) a.out[j * a.n + i[0]] = lo2(g[j]);
            if (in1) a.out[j * a.n + i[1]] = hi2(g[j]);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) local += __shfl_xor_sync(0xffffffffu, local, o);
    if (lane_id() == 0) s_red[threadIdx.x >> 5] = local;
    __syncthreads();
    if (threadIdx.x == 0) {
        float s = 0.f;
        for (int k = 0; k < kTileThreads / 32; ++k) s += s_red[k];
        add_sum<kPass>(a, s);
    }
}

// Tiles below this many values C H W, strips from there on (us of a loss call with the target's moments
// given and without, tiles / strips): 3 x 128 x 128 12.1 / 14.5 and 12.2 / 16.5; 3 x 270 x 480 18.0 / 24.6 and 18.4 /
// 26.8; 3 x 540 x 960 30.9 / 36.5 and 33.3 / 40.5; 3 x 675 x 1200 45.2 / 47 and 48.9 / 52; 3 x 720 x 1280 49.6 / 48.8 and
// 51.7 / 54; 3 x 900 x 1600 75.9 / 65.6 and 79.7 / 73.5; 1080p 102 / 88.6 and 109 / 101.
constexpr int64_t kTileMax = 2600000;

// Rows per strip: as many strips as fit the SMs at once, since the ten halo rows of a strip are
// blurred twice and a second wave of CTAs would double the time (1080p, 12 strips' warps per SM:
// 54 rows; 900 CTAs in one wave).
constexpr int kMinRows = 2;

// The target's moments are strips at every size; they take little work a row, so that fewer and longer
// strips are faster: four CTAs per SM instead of six 480 x 270 6.9 -> 4.8 us, 960 x 540 10.9 -> 8.4, 1080p 27 ->
// 23.4 (three 27, eight 23.1 but 960 x 540 9.5).
template <Pass kPass>
void launch_strips(StripArgs a, int C, cudaStream_t st) {
    const int cols = (a.W + kCols - 1) / kCols;
    const int ctas = kPass == kTargetStats ? 4 : kCtas;
    int64_t ny = (int64_t)kSmCount * ctas / ((int64_t)cols * C);
    if (ny < 1) ny = 1;
    const int64_t rows = (a.H + ny * kStripWarps - 1) / (ny * kStripWarps);
    a.rows = (int)(rows < kMinRows ? kMinRows : (rows + 1) / 2 * 2);
    ny = (a.H + (int64_t)a.rows * kStripWarps - 1) / ((int64_t)a.rows * kStripWarps);
    a.parts = (unsigned)((a.H + a.rows - 1) / a.rows) * (unsigned)cols * (unsigned)C;
    launch_pdl(ssim_strip<kPass>, dim3(cols, (unsigned)ny, C), dim3(32 * kStripWarps), 0, st, a);
}

template <Pass kPass>
void launch_pass(StripArgs a, int C, bool tiles, cudaStream_t st) {
    if (!tiles) return launch_strips<kPass>(a, C, st);
    const dim3 grid((a.W + kTX - 1) / kTX, (a.H + kTY - 1) / kTY, C);
    a.parts = grid.x * grid.y * grid.z;
    launch_pdl(ssim_tile<kPass>, grid, dim3(kTileThreads), 0, st, a);
}

}  // namespace
}  // namespace ogs

using namespace ogs;

extern "C" size_t ogs_loss_l1_ssim_scratch_bytes(int32_t C, int32_t H, int32_t W) {
    return sizeof(float) * ((size_t)3 * C * H * W + 4) + 512;   // maps, sums, alignment
}

extern "C" ogs_status ogs_ssim_target_stats(const float* target, int32_t C, int32_t H,
                                            int32_t W, float* ystat, void* stream) {
    if (!target || !ystat || C <= 0 || H <= 0 || W <= 0) return OGS_ERR_ARG;
    StripArgs a = {};
    a.in[0] = target;
    a.out = ystat;
    a.g = make_window();
    a.H = H; a.W = W;
    a.n = (int64_t)C * H * W;
    a.vec = W % 2 == 0 && aligned(ystat, 8);
    launch_strips<kTargetStats>(a, C, (cudaStream_t)stream);
    return launch_status();
}

extern "C" ogs_status ogs_loss_l1_ssim(const float* img, const float* target, int32_t C,
                                       int32_t H, int32_t W, float lambda, float* dimg,
                                       float* loss, const float* target_stats, void* scratch,
                                       size_t scratch_bytes, void* stream) {
    if (!img || !target || !dimg || !scratch || C <= 0 || H <= 0 || W <= 0) return OGS_ERR_ARG;
    if (!(lambda >= 0.f && lambda <= 1.f)) return OGS_ERR_ARG;
    if (scratch_bytes < ogs_loss_l1_ssim_scratch_bytes(C, H, W) || !aligned(scratch, 16))
        return OGS_ERR_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    const int64_t n = (int64_t)C * H * W;
    Carver cv(scratch);
    float* gp = cv.take<float>(3 * n);
    LossSums* sums = cv.take<LossSums>(1);
    if (cudaMemsetAsync(sums, 0, sizeof(LossSums), st) != cudaSuccess) return OGS_ERR_CUDA;
    StripArgs a = {};
    a.in[0] = img;
    a.in[1] = target;
    a.ystat = target_stats;
    a.out = gp;
    a.sums = sums;
    a.g = make_window();
    a.H = H; a.W = W;
    a.n = n;
    a.inv_n = 1.0f / (float)n;
    a.lam = lambda;
    a.vec = W % 2 == 0 && aligned(img, 8) && aligned(target, 8) && aligned(dimg, 8) &&
            aligned(target_stats, 8);
    const bool tiles = n < kTileMax && (H + kTY - 1) / kTY <= 65535;       // (the grid's limit)
    if (target_stats) launch_pass<kMoments3>(a, C, tiles, st);
    else launch_pass<kMoments5>(a, C, tiles, st);
    for (int j = 0; j < 3; ++j) a.in[j] = gp + j * n;
    a.x = img;
    a.y = target;
    a.out = dimg;
    a.loss = loss;
    launch_pass<kGradient>(a, C, tiles, st);
    return launch_status();
}
