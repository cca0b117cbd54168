// Backward of the neural-Gaussian decoders (Sec. 3.2, Eq. offsets and Eq. mlp) with the
// per-anchor products on the 5th-generation tensor cores (BF16 x BF16 -> FP32 in TMEM), 128
// anchors per tile:
//
//   MMA 1:  D[128 x 96]  = Z[128 x 48]  . W1^T     hidden pre-activations (recomputed)
//   MMA 2:  D[128 x 128] = H[128 x 96]  . W2^T     decoder outputs, each decoder's own blocks
//   MMA 3:  D[128 x 96]  = dY[128 x 112] . W2      hidden gradients, each decoder's own blocks
//   MMA 4:  D[128 x 32]  = dP[128 x 96]  . W1f     feature gradients (W1 restricted to f_v)
//
// Between them the FP32 epilogues apply bias/ReLU, compute the output gradients dy of every
// Gaussian, mask dh by the ReLU and accumulate dfeat, doffs and dlv.  With appearance codes
// (Sec. 4.4) the code fills Z's zero-padded columns 40..47 and the colour rows of W1 carry its
// weights there; the code gradient W_app^T dp is formed on the CUDA cores in epilogue 3.  The f32
// rows z, h, dy, dp go to scratch for the weight pass, which is the FP32 split-over-anchors
// product of grad.cu.
//
// The products are tiny, so the kernel is bound by latency: of the gathers, of the Gaussians'
// gradients and of the chain of four products.  Two CTAs share an SM (110 KB each: the operand
// image is packed once per call by db_pack, without the zero blocks of the block-diagonal W2, and
// dY overlays the consumed Z and H), and the output gradients are formed by one thread per
// Gaussian, consecutive Gaussians on consecutive threads, with all of a thread's loads issued
// first: 64 anchors at a time, their outputs staged in shared memory, dy in place of y, stored as
// whole rows by one bulk copy.  (One CTA per SM and one thread per half an anchor, whose loads
// were strided by ten Gaussians: 100k anchors 248 us; now 145 us.)  128 registers, two CTAs' worth, with 252
// bytes spilled.
// Operands live in shared memory in the no-swizzle K-major core-matrix layout; every mbarrier
// wait is bounded and on expiry the kernel sets ogs_counts.timeout, waits (bounded) for the MMAs
// in flight, releases TMEM and exits.
#include "decode_bwd.cuh"
#include "tc.cuh"

namespace ogs {
namespace {

using namespace db;

constexpr int kTM = 128;
constexpr int kThreads = 256;            // two threads per anchor (TMEM lane): halves 0 and 1
constexpr int kK1 = 48;                  // 36 inputs padded
constexpr int kN1 = 96;                  // hidden units of the three decoders
constexpr int kN2 = 112;                 // 110 outputs padded (the K of MMA 3)
constexpr uint32_t kTmemCols = 128;
constexpr uint32_t kColD4 = 96;          // MMA 4 (32 columns); MMAs 1 to 3 start at column 0
// MMA 2: opacity outputs in columns 0..9, covariance in 16..85, colour in 96..125
constexpr int kColCov = 16, kColCol = 96;
constexpr uint32_t kWaitLimit = 1u << 24;
constexpr int kAppK = 40;                // layer-1 K column of an appearance code's first value

// Operand image: packed by db_pack, fetched by every CTA with one bulk copy.
constexpr int kImgB1 = 0;                                // W1 [96][48]
constexpr int kImgB2a = kImgB1 + kN1 * kK1 * 2;          // [16 opacity + 80 covariance][32 + 32]
constexpr int kNB2a = 96, kKB2a = 64;
constexpr int kImgB2b = kImgB2a + kNB2a * kKB2a * 2;     // colour [32][32]
constexpr int kImgB3 = kImgB2b + 32 * 32 * 2;            // W2^T per decoder [32 hidden][its K chunks]
// K chunks (16 stacked outputs each) that hold a decoder's rows: opacity 0, colour 0..2,
// covariance 2..6
__host__ __device__ constexpr int k3_first(int d) { return d == 2 ? 2 : 0; }
__host__ __device__ constexpr int k3_chunks(int d) { return d == 0 ? 1 : (d == 1 ? 3 : 5); }
__host__ __device__ constexpr int b3_off(int d) {        // bytes from kImgB3
    return d == 0 ? 0 : (d == 1 ? 32 * 16 * 2 : 32 * 16 * 2 * 4);
}
constexpr int kImgB4 = kImgB3 + 32 * 16 * 2 * 9;         // W1f^T [32][96]
constexpr int kImgBias1 = kImgB4 + kF * kN1 * 2;         // b1 f32[96]
constexpr int kImgBias2 = kImgBias1 + kN1 * 4;           // b2 f32[kRowY], laid out as a dy row
constexpr int kImgWa = kImgBias2 + kRowY * 4;            // appearance weights f32[32][8], padded
constexpr int kImgBytes = kImgWa + kH * kMaxApp * 4;
static_assert(kImgBytes % 16 == 0, "bulk copy size");
static_assert(kImgBytes <= (int)sizeof(float) * kDbBlocks * kNWeights, "the image fits the partials");

constexpr int kOffWork = (kImgBytes + 127) / 128 * 128;  // operands of the tile, overlaid:
constexpr int kOffA1 = kOffWork;                         //   Z  128 x 48
constexpr int kOffA2 = kOffA1 + kTM * kK1 * 2;           //   H, later dP  128 x 96
constexpr int kOffA3 = kOffWork;                         //   dY 128 x 112, once MMA 2 is done
constexpr int kOffLv = kOffA3 + kTM * kN2 * 2;           //   dlv shares of a round's Gaussians
constexpr int kWorkBytes = kTM * (kK1 + kN1) * 2;
constexpr int kLvPitch = 3 * kK + 1;
constexpr int kRound = kTM / 2;                          // anchors staged at a time
constexpr int kRoundGauss = kRound * kK;
constexpr int kIters = (kRoundGauss + kThreads - 1) / kThreads;
static_assert(kOffLv + kRound * kLvPitch * 4 <= kOffWork + kWorkBytes, "shares behind dY");
constexpr int kOffY = kOffWork + kWorkBytes;             // y, then dy: [64][kRowY] f32
constexpr int kOffRows = kOffY + kRound * kRowY * 4;     // j, w, l_v[3] of each anchor
constexpr int kRowWords = 5;
constexpr int kSmem = kOffRows + kTM * kRowWords * 4;
static_assert(kOffY % 16 == 0 && kRowY % 4 == 0, "rows are read and copied as 16-byte vectors");
static_assert(kSmem <= 112 * 1024, "two CTAs per SM");

constexpr int kPackThreads = 256;
constexpr int kG1 = kN1 * kK1 / 8, kG2a = kNB2a * kKB2a / 8, kG2b = 32 * 32 / 8,
              kG3 = 32 * 16 * 9 / 8, kG4 = kF * kN1 / 8;
constexpr int kPackGroups = kG1 + kG2a + kG2b + kG3 + kG4;
constexpr int kPackItems = kPackGroups + kN1 + kRowY + kH * kMaxApp;

__device__ __forceinline__ void put8(unsigned char* base, int row, int kc, int Kpad,
                                     const float (&v)[8]) {
    __nv_bfloat162 h[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
    *reinterpret_cast<uint4*>(base + tc::core_offset(row, 8 * kc, Kpad)) =
        *reinterpret_cast<const uint4*>(h);
}

// weight of stacked output n of decoder d for its hidden unit o; 0 for the padding rows
__device__ __forceinline__ float w2_of(const ogs_mlp& w, int d, int n, int o) {
    if (d == 0) return n < kK ? w.w2_op[n * kH + o] : 0.f;
    if (d == 1) return n < 3 * kK ? w.w2_col[n * kH + o] : 0.f;
    return n < 7 * kK ? w.w2_cov[n * kH + o] : 0.f;
}

// One 8-element operand row chunk, bias or appearance weight of the image per thread.
__global__ void __launch_bounds__(kPackThreads) db_pack(ogs_mlp m, unsigned char* img) {
    int e = blockIdx.x * kPackThreads + threadIdx.x;
    if (e >= kPackItems) return;
    float v[8];
    if (e < kG1) {                                         // W1 [o][k]
        const int n = e / (kK1 / 8), kc = e % (kK1 / 8);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int k = 8 * kc + i, ca = k - kAppK;
            // columns 40..47: the colour decoder's appearance weights (Sec. 4.4), else zero
            v[i] = k < kDin ? m.w1[n * kDin + k]
                            : (ca >= 0 && ca < m.A && n >= kH && n < 2 * kH
                                   ? m.w1_app[(n - kH) * m.A + ca] : 0.f);
        }
        put8(img + kImgB1, n, kc, kK1, v);
        return;
    }
    if ((e -= kG1) < kG2a) {                               // opacity and covariance blocks of W2
        const int n = e / (kKB2a / 8), kc = e % (kKB2a / 8);
        const bool op = n < kColCov, mine = op == (kc < kH / 8);
#pragma unroll
        for (int i = 0; i < 8; ++i)
            v[i] = mine ? w2_of(m, op ? 0 : 2, op ? n : n - kColCov, 8 * (kc % (kH / 8)) + i) : 0.f;
        put8(img + kImgB2a, n, kc, kKB2a, v);
        return;
    }
    if ((e -= kG2a) < kG2b) {                              // colour block of W2
        const int n = e / (kH / 8), kc = e % (kH / 8);
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = w2_of(m, 1, n, 8 * kc + i);
        put8(img + kImgB2b, n, kc, kH, v);
        return;
    }
    if ((e -= kG2b) < kG3) {                               // W2^T [o][stacked output]
        const int d = e < 32 * 2 ? 0 : (e < 32 * 2 * 4 ? 1 : 2);
        e -= b3_off(d) / 16;
        const int nk = 2 * k3_chunks(d), o = e / nk, kc = e % nk;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = 16 * k3_first(d) + 8 * kc + i;   // stacked output
            v[i] = r < kNOut && dec_of(r) == d ? w2_of(m, d, r - out_base(d), o) : 0.f;
        }
        put8(img + kImgB3 + b3_off(d), o, kc, 8 * nk, v);
        return;
    }
    if ((e -= kG3) < kG4) {                                // W1 restricted to f_v, [i][o]
        const int i = e / (kN1 / 8), kc = e % (kN1 / 8);
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = m.w1[(8 * kc + u) * kDin + i];
        put8(img + kImgB4, i, kc, kN1, v);
        return;
    }
    if ((e -= kG4) < kN1) {
        reinterpret_cast<float*>(img + kImgBias1)[e] = m.b1[e];
    } else if ((e -= kN1) < kRowY) {
        const int n = row_out(e);
        reinterpret_cast<float*>(img + kImgBias2)[e] =
            n < 0 ? 0.f : (n < kK ? m.b2_op[n] : (n < 4 * kK ? m.b2_col[n - kK] : m.b2_cov[n - 4 * kK]));
    } else {
        e -= kRowY;
        const int o = e / kMaxApp, ca = e % kMaxApp;
        reinterpret_cast<float*>(img + kImgWa)[e] = ca < m.A ? m.w1_app[o * m.A + ca] : 0.f;
    }
}

// D[., d ..] (+)= A chunks ca, ca + 1, ... (nk of them, 16 columns each) . B chunks 0, 1, ...
__device__ __forceinline__ void mma_chunks(uint32_t d, const unsigned char* a, int ca, int Ka,
                                           const unsigned char* b, int cb, int Kb, int nk,
                                           uint32_t idesc, bool accumulate) {
    for (int kk = 0; kk < nk; ++kk)
        tc::mma_bf16(d, tc::smem_desc(tc::smem_u32(a + (ca + kk) * 256), 128, 16 * Ka),
                     tc::smem_desc(tc::smem_u32(b + (cb + kk) * 256), 128, 16 * Kb), idesc,
                     accumulate || kk > 0);
}

// The 32 TMEM columns from c0 of this lane's row -> its staged y row (the columns of MMA 2 in
// the order of a dy row; padding columns dropped or kept as the row's padding).
template <int c0>
__device__ __forceinline__ void stage_cols(uint32_t lane_addr, float* y) {
    float v[32];
    tc::tmem_ld32(lane_addr + c0, v);
#pragma unroll
    for (int i = 0; i < 32; i += 4) {
        const int c = c0 + i;
        const int at = c < kRowCol ? c : (c >= kColCol ? c - kColCol + kRowCol
                                                       : (c >= kColCov ? c - kColCov + kRowCov : -1));
        const bool keep = c < kRowCol || (c >= kColCol && at < kRowCov) ||
                          (c >= kColCov && c < kColCol && at < kRowY);
        if (keep) *reinterpret_cast<float4*>(y + at) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
    }
}

struct TcBwdArgs {
    DbArgs a;
    const unsigned char* img;
    uint32_t* timeout;
};

__global__ void __launch_bounds__(kThreads, 2) decode_bwd_rows_tc(TcBwdArgs args) {
    extern __shared__ __align__(1024) unsigned char sm[];
    __shared__ __align__(8) uint64_t mbar;
    __shared__ __align__(8) uint64_t wbar;
    __shared__ uint32_t tmem_base;
    const DbArgs& a = args.a;
    unsigned char* sA1 = sm + kOffA1;
    unsigned char* sA2 = sm + kOffA2;
    unsigned char* sA3 = sm + kOffA3;
    const float* sb1 = reinterpret_cast<const float*>(sm + kImgBias1);
    const float* sb2 = reinterpret_cast<const float*>(sm + kImgBias2);
    const float* sWa = reinterpret_cast<const float*>(sm + kImgWa);
    float* sY = reinterpret_cast<float*>(sm + kOffY);
    float* sLv = reinterpret_cast<float*>(sm + kOffLv);
    float* rows = reinterpret_cast<float*>(sm + kOffRows);
    const int t = threadIdx.x, w = t >> 5;
    const int half = w >> 2;                     // warp-uniform
    const int al = t & (kTM - 1);                // anchor (TMEM lane) of this thread
    const uint32_t M = a.counts->n_selected;
    const uint32_t ntiles = (M + kTM - 1) / kTM;
    if (blockIdx.x >= ntiles) return;                      // uniform, before any TMEM use
    const int napp = a.mlp.A;                              // appearance code width (0: none)

    if (t == 0) {
        tc::mbar_init(&mbar, 1);
        tc::mbar_init(&wbar, 1);
        tc::mbar_expect_tx(&wbar, kImgBytes);
        tc::bulk_load(sm, args.img, kImgBytes, &wbar);     // lands while the inputs are gathered
    }
    if (w == 0) {
        tc::tmem_alloc(&tmem_base, kTmemCols);
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tbase = tmem_base;
    const uint32_t lane_addr = tbase + ((uint32_t)(32 * (w & 3)) << 16);
    const uint32_t id96 = tc::idesc_bf16(kTM, 96), id32 = tc::idesc_bf16(kTM, 32);
    const Cam& c = a.cam;
    uint32_t phase = 0;
    bool aborted = false, have_img = false;

    // issue (thread 0), then all threads wait on the MMA group; false if the wait expired
    auto run = [&](auto issue) -> bool {
        tc::fence_smem_to_async();
        tc::fence_before_sync();
        __syncthreads();
        tc::fence_after_sync();
        if (t == 0) {
            issue();
            tc::commit(&mbar);
        }
        const bool ok = tc::mbar_wait(&mbar, phase, kWaitLimit);
        if (__syncthreads_or(!ok)) return false;
        phase ^= 1;
        tc::fence_after_sync();
        return true;
    };
    // columns [32 q0, 32 q1) of a 96-column accumulator belong to this half
    const int q0 = half == 0 ? 0 : 2, q1 = half == 0 ? 2 : 3;

    for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const uint32_t r = tile * kTM + al;
        const bool valid = r < M;
        uint32_t j = 0;
        if (valid) j = a.sel_idx[r];
        // gather: half 0 features 0..15 and the direction, half 1 features 16..31 and the code
        {
            float x[16], zc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int i = 0; i < 16; ++i) x[i] = 0.f;
            if (valid) {
                const float4* f4 = reinterpret_cast<const float4*>(a.feat + (size_t)j * kF) + 4 * half;
                const float4 u[4] = {f4[0], f4[1], f4[2], f4[3]};
                float4* zr = reinterpret_cast<float4*>(a.rowZ + (size_t)r * kRowZ);
                if (half == 0) {
                    float dv[3], lvv[3];
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        dv[q] = a.pos[3 * (size_t)j + q] - c.c[q];
                        lvv[q] = a.lv[3 * (size_t)j + q];
                    }
                    const float wgt = a.sel_w[r];
                    const float d = sqrtf(dv[0] * dv[0] + dv[1] * dv[1] + dv[2] * dv[2]);
                    zc[0] = dv[0] / d; zc[1] = dv[1] / d; zc[2] = dv[2] / d; zc[3] = d;
                    zr[kF / 4] = make_float4(zc[0], zc[1], zc[2], zc[3]);
                    zr[kF / 4 + 1] = make_float4(0.f, 0.f, 0.f, 0.f);
                    float* rw = rows + al * kRowWords;
                    rw[0] = __uint_as_float(j);
                    rw[1] = wgt;
#pragma unroll
                    for (int q = 0; q < 3; ++q) rw[2 + q] = lvv[q];
                } else {
#pragma unroll
                    for (int ca = 0; ca < kMaxApp; ++ca)
                        zc[ca] = ca < napp ? a.mlp.app[(size_t)j * napp + ca] : 0.f;
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    zr[4 * half + i] = u[i];
                    x[4 * i] = u[i].x; x[4 * i + 1] = u[i].y; x[4 * i + 2] = u[i].z; x[4 * i + 3] = u[i].w;
                }
            }
#pragma unroll
            for (int kc = 0; kc < 2; ++kc) {
                const float v[8] = {x[8 * kc], x[8 * kc + 1], x[8 * kc + 2], x[8 * kc + 3],
                                    x[8 * kc + 4], x[8 * kc + 5], x[8 * kc + 6], x[8 * kc + 7]};
                put8(sA1, al, 2 * half + kc, kK1, v);
            }
            put8(sA1, al, half == 0 ? kF / 8 : kK1 / 8 - 1, kK1, zc);
        }
        if (!have_img) {                                   // the operand image, once per CTA
            have_img = true;
            if (!tc::mbar_wait(&wbar, 0, kWaitLimit)) {
                if (t == 0) atomicExch(args.timeout, 1u);
                tc::mbar_wait(&wbar, 0, kWaitLimit);       // the copy may still be landing
            }
        }
        if (!run([&] { mma_chunks(tbase, sA1, 0, kK1, sm + kImgB1, 0, kK1, kK1 / 16, id96, false); })) {
            aborted = true;
            break;
        }

        // epilogue 1 (this half's columns): bias, ReLU (mask kept), H -> bf16 operand, f32 row
        uint32_t mask[2] = {0u, 0u};
#pragma unroll
        for (int qq = 0; qq < 2; ++qq) {
            const int q = q0 + qq;
            if (q >= q1) break;
            float v[32];
            tc::tmem_ld32(lane_addr + 32 * q, v);
            uint32_t mk = 0;
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                const float p = v[i] + sb1[32 * q + i];
                mk |= (p > 0.f ? 1u : 0u) << i;
                v[i] = fmaxf(p, 0.f);
            }
            mask[qq] = mk;
#pragma unroll
            for (int cc = 0; cc < 4; ++cc) {
                const float h8[8] = {v[8 * cc], v[8 * cc + 1], v[8 * cc + 2], v[8 * cc + 3],
                                     v[8 * cc + 4], v[8 * cc + 5], v[8 * cc + 6], v[8 * cc + 7]};
                put8(sA2, al, 4 * q + cc, kN1, h8);
            }
            if (valid) {
                float4* hr = reinterpret_cast<float4*>(a.rowH + (size_t)r * kRowH + 32 * q);
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    hr[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
            }
        }
        // hidden units 0..31 and 64..95 against the opacity and covariance blocks, 32..63 against
        // the colour block: every output sums the same 16-wide chunks as a block-diagonal W2 (the
        // dropped ones are zero)
        if (!run([&] {
                mma_chunks(tbase, sA2, 0, kN1, sm + kImgB2a, 0, kKB2a, 2, id96, false);
                mma_chunks(tbase, sA2, 4, kN1, sm + kImgB2a, 2, kKB2a, 2, id96, true);
                mma_chunks(tbase + kColCol, sA2, 2, kN1, sm + kImgB2b, 0, kH, 2, id32, false);
            })) {
            aborted = true;
            break;
        }

        // epilogue 2, 64 anchors at a time (TMEM lane quarters 2 round, 2 round + 1)
        for (int round = 0; round < 2; ++round) {
            if (((w & 3) >> 1) == round) {
                float* y = sY + (al - kRound * round) * kRowY;
                if (half == 0) {
                    stage_cols<0>(lane_addr, y);
                    stage_cols<32>(lane_addr, y);
                } else {
                    stage_cols<64>(lane_addr, y);
                    stage_cols<96>(lane_addr, y);
                }
            }
            const uint32_t base = tile * kTM + kRound * round;        // first anchor of the round
            const int nrow = (int)min((uint32_t)kRound, M > base ? M - base : 0u);
            // every load of the thread's Gaussians first, so that their latencies overlap
            GaussGrad gg[kIters];
            float O[kIters][3], dO[kIters][3];
#pragma unroll
            for (int it = 0; it < kIters; ++it) {
                const int gl = it * kThreads + t, rl = gl / kK, i = gl - rl * kK;
                if (rl < nrow) {
                    gg[it] = load_gauss_grad(a, (size_t)base * kK + gl);
                    const uint32_t jg = __float_as_uint(rows[(kRound * round + rl) * kRowWords]);
                    const size_t o = ((size_t)jg * kK + i) * 3;
#pragma unroll
                    for (int e = 0; e < 3; ++e) {
                        O[it][e] = a.offs[o + e];
                        dO[it][e] = a.doffs[o + e];
                    }
                }
            }
            tc::fence_before_sync();
            __syncthreads();
            tc::fence_after_sync();
#pragma unroll
            for (int it = 0; it < kIters; ++it) {
                const int gl = it * kThreads + t, rl = gl / kK, i = gl - rl * kK;
                if (gl >= kRoundGauss) break;
                float* yr = sY + rl * kRowY;
                float* y0 = yr + i;
                float* y1 = yr + kRowCol + 3 * i;
                float* y2 = yr + kRowCov + 7 * i;
                if (rl < nrow) {
                    const float* rw = rows + (kRound * round + rl) * kRowWords;
                    const uint32_t jg = __float_as_uint(rw[0]);
                    const float lvv[3] = {rw[2], rw[3], rw[4]};
                    float y[7], dy[7], dlv[3] = {0.f, 0.f, 0.f};
                    y[0] = *y0 + sb2[i];
                    dy_opacity(gg[it], rw[1], y, dy);
                    *y0 = dy[0];
#pragma unroll
                    for (int e = 0; e < 3; ++e) y[e] = y1[e] + sb2[kRowCol + 3 * i + e];
                    dy_color(gg[it], y, dy);
#pragma unroll
                    for (int e = 0; e < 3; ++e) y1[e] = dy[e];
#pragma unroll
                    for (int e = 0; e < 7; ++e) y[e] = y2[e] + sb2[kRowCov + 7 * i + e];
                    dy_cov(gg[it], lvv, y, dy, dlv);
#pragma unroll
                    for (int e = 0; e < 7; ++e) y2[e] = dy[e];
                    // positions: mu = x_v + O * l_v
                    float* dof = a.doffs + ((size_t)jg * kK + i) * 3;
#pragma unroll
                    for (int e = 0; e < 3; ++e) {
                        dof[e] = fmaf(gg[it].mean[e], lvv[e], dO[it][e]);
                        sLv[rl * kLvPitch + 3 * i + e] = fmaf(gg[it].mean[e], O[it][e], dlv[e]);
                    }
                } else {
                    *y0 = 0.f;
#pragma unroll
                    for (int e = 0; e < 3; ++e) y1[e] = 0.f;
#pragma unroll
                    for (int e = 0; e < 7; ++e) y2[e] = 0.f;
                }
            }
            tc::fence_smem_to_async();                     // dy rows, read by the bulk copy
            __syncthreads();
            if (t == 0 && nrow > 0) {
                tc::bulk_store(a.rowY + (size_t)base * kRowY, sY, (uint32_t)nrow * kRowY * 4u);
                tc::bulk_commit();
            }
            // dy rows -> bf16 operand (stacked outputs without the rows' padding)
            for (int it = t; it < kRound * (kN2 / 8); it += kThreads) {
                const int rl = it % kRound, cc = it / kRound;
                float d8[8];
#pragma unroll
                for (int u = 0; u < 8; u += 2) {
                    const int k = 8 * cc + u;
                    const float2 v = k < kNOut
                        ? *reinterpret_cast<const float2*>(sY + rl * kRowY + out_row(k))
                        : make_float2(0.f, 0.f);
                    d8[u] = v.x;
                    d8[u + 1] = v.y;
                }
                put8(sA3, kRound * round + rl, cc, kN2, d8);
            }
            if (t < 3 * kRound) {                          // l_v: the shares of an anchor's Gaussians
                const int rl = t / 3, e = t % 3;
                if (rl < nrow) {
                    float s = 0.f;
#pragma unroll
                    for (int i = 0; i < kK; ++i) s += sLv[rl * kLvPitch + 3 * i + e];
                    const uint32_t jg = __float_as_uint(rows[(kRound * round + rl) * kRowWords]);
                    a.dlv[3 * (size_t)jg + e] += s;
                }
            }
            if (t == 0) tc::bulk_wait_read();
            __syncthreads();                               // the staged rows may be overwritten
        }
        if (!run([&] {
#pragma unroll
                for (int d = 0; d < 3; ++d)
                    mma_chunks(tbase + 32 * d, sA3, k3_first(d), kN2, sm + kImgB3 + b3_off(d), 0,
                               16 * k3_chunks(d), k3_chunks(d), id32, false);
            })) {
            aborted = true;
            break;
        }

        // epilogue 3 (this half's columns): through the ReLU -> dP (bf16 operand in the H
        // buffer, f32 row)
#pragma unroll
        for (int qq = 0; qq < 2; ++qq) {
            const int q = q0 + qq;
            if (q >= q1) break;
            float v[32];
            tc::tmem_ld32(lane_addr + 32 * q, v);
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = ((mask[qq] >> i) & 1u) && valid ? v[i] : 0.f;
#pragma unroll
            for (int cc = 0; cc < 4; ++cc) {
                const float p8[8] = {v[8 * cc], v[8 * cc + 1], v[8 * cc + 2], v[8 * cc + 3],
                                     v[8 * cc + 4], v[8 * cc + 5], v[8 * cc + 6], v[8 * cc + 7]};
                put8(sA2, al, 4 * q + cc, kN1, p8);
            }
            if (valid) {
                float4* pr = reinterpret_cast<float4*>(a.rowP + (size_t)r * kRowP + 32 * q);
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    pr[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                if (q == 1 && napp > 0) {   // code gradient: dapp_c += sum_o Wa[o][c] dp_o
                    for (int ca = 0; ca < napp; ++ca) {
                        float g = 0.f;
#pragma unroll
                        for (int o = 0; o < kH; ++o) g = fmaf(sWa[o * kMaxApp + ca], v[o], g);
                        a.dapp[(size_t)j * napp + ca] += g;
                    }
                }
            }
        }
        // feature gradients so far, this half's 16 columns: loaded while the product runs
        float4 df[4];
        float4* dfp = reinterpret_cast<float4*>(a.dfeat + (size_t)j * kF) + 4 * half;
        if (valid) {
#pragma unroll
            for (int i = 0; i < 4; ++i) df[i] = dfp[i];
        }
        if (!run([&] { mma_chunks(tbase + kColD4, sA2, 0, kN1, sm + kImgB4, 0, kN1, kN1 / 16, id32, false); })) {
            aborted = true;
            break;
        }

        // epilogue 4: feature gradients
        {
            float v[32];
            tc::tmem_ld32(lane_addr + kColD4, v);
            if (valid) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float4 u = df[i];
                    u.x += half ? v[16 + 4 * i] : v[4 * i];
                    u.y += half ? v[17 + 4 * i] : v[4 * i + 1];
                    u.z += half ? v[18 + 4 * i] : v[4 * i + 2];
                    u.w += half ? v[19 + 4 * i] : v[4 * i + 3];
                    dfp[i] = u;
                }
            }
        }
        tc::fence_before_sync();
        __syncthreads();
        tc::fence_after_sync();
    }
    if (aborted) {
        if (t == 0) atomicExch(args.timeout, 1u);
        tc::mbar_wait(&mbar, phase, kWaitLimit);           // the group that may be in flight
    }
    if (t == 0) tc::bulk_wait_all();                       // the row copies have left this CTA
    tc::fence_before_sync();
    __syncthreads();
    if (w == 0) tc::tmem_dealloc(tbase, kTmemCols);
}

}  // namespace
}  // namespace ogs

using namespace ogs;
using namespace ogs::db;

extern "C" ogs_status ogs_decode_bwd_bf16(const float* pos, const float* feat, const float* offs,
                                          const float* lv, int64_t N, const ogs_mlp* mlp,
                                          const ogs_camera* cam, const uint32_t* sel_idx,
                                          const float* sel_w, int64_t sel_cap,
                                          ogs_counts* counts, const float* dmeans,
                                          const float* dscales, const float* dquats,
                                          const float* drec, float* dfeat, float* doffs,
                                          float* dlv, const ogs_mlp* dmlp, void* scratch,
                                          size_t scratch_bytes, void* stream) {
    if (!pos || !feat || !offs || !lv || !mlp || !cam || !sel_idx || !sel_w || !counts ||
        !dmeans || !dscales || !dquats || !drec || !dfeat || !doffs || !dlv || !dmlp || !scratch)
        return OGS_ERR_ARG;
    if (mlp->F != kF || mlp->H != kH || mlp->k != kK || N < 0 || sel_cap < 0 || !app_ok(*mlp))
        return OGS_ERR_ARG;
    if (mlp->A > 0 && (!dmlp->w1_app || !dmlp->app)) return OGS_ERR_ARG;
    if (!dmlp->w1 || !dmlp->b1 || !dmlp->w2_op || !dmlp->b2_op || !dmlp->w2_col ||
        !dmlp->b2_col || !dmlp->w2_cov || !dmlp->b2_cov)
        return OGS_ERR_ARG;
    if (scratch_bytes < db_layout(sel_cap, nullptr, nullptr) || !aligned(scratch, 16) ||
        !aligned(dquats, 16) || !aligned(feat, 16) || !aligned(dfeat, 16))
        return OGS_ERR_ARG;
    if (sel_cap == 0) return OGS_OK;
    cudaStream_t st = (cudaStream_t)stream;
    DbScratch sc;
    db_layout(sel_cap, scratch, &sc);
    TcBwdArgs args{{pos, feat, offs, lv, sel_idx, sel_w, counts, *mlp, make_cam(*cam), dmeans,
                    dscales, dquats, drec, dfeat, doffs, dlv, sc.rowY, sc.rowH, sc.rowP, sc.rowZ,
                    sc.partial, const_cast<float*>(dmlp->app)},
                   // the image lies in the weight pass's partial rows, which that pass writes later
                   reinterpret_cast<const unsigned char*>(sc.partial), &counts->timeout};
    if (cudaFuncSetAttribute(decode_bwd_rows_tc, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kSmem) != cudaSuccess)
        return OGS_ERR_CUDA;
    const int64_t tiles = (sel_cap + kTM - 1) / kTM;
    const int grid = (int)(tiles < 2 * kSmCount ? tiles : 2 * kSmCount);
    db_pack<<<(kPackItems + kPackThreads - 1) / kPackThreads, kPackThreads, 0, st>>>(
        *mlp, reinterpret_cast<unsigned char*>(sc.partial));
    decode_bwd_rows_tc<<<grid, kThreads, kSmem, st>>>(args);
    if (launch_weight_pass(args.a, sc, *dmlp, st) != cudaSuccess) return OGS_ERR_CUDA;
    return launch_status();
}
