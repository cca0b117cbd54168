// Decoder backward (Sec. 3.2, Eq. offsets and Eq. mlp): shapes, argument block, scratch
// layout and the per-Gaussian output gradient shared by the FP32 and the tensor-core row
// passes (grad.cu, decode_bwd_tc.cu).
#pragma once

#include "internal.cuh"

namespace ogs {
namespace db {

constexpr int kF = 32;
constexpr int kH = 32;
constexpr int kDin = kF + 4;
constexpr int kK = 10;
constexpr int kNW1 = 3 * kH * kDin;                       // 3456
constexpr int kNB1 = 3 * kH;                              // 96
constexpr int kNOut = 11 * kK;                            // 110 (10 + 30 + 70)
constexpr int kNW2 = kNOut * kH;                          // 3520
constexpr int kNWeights = kNW1 + kNB1 + kNW2 + kNOut;     // 7182

// offsets of the decoder gradients inside one flat partial row:
//   dw1 [3][H][Din] | db1 [3][H] | dw2_op [k][H] | dw2_col [3k][H] | dw2_cov [7k][H] |
//   db2_op [k] | db2_col [3k] | db2_cov [7k]
constexpr int kOffB1 = kNW1;
constexpr int kOffW2 = kOffB1 + kNB1;
constexpr int kOffB2 = kOffW2 + kNW2;

// per-anchor rows handed from the row pass to the weight pass (f32, 16-byte aligned rows)
constexpr int kRowY = 116;    // dL/dy: opacity 0..9, colour 12..41, covariance 44..113 (padding
                              // between them unused)
constexpr int kRowCol = 12, kRowCov = 44;
constexpr int kRowH = 96;     // hidden activations of the three decoders
constexpr int kRowP = 96;     // dL/d(pre-activation) of the three decoders
constexpr int kRowZ = 40;     // decoder input z (36, +4 zero)

struct DbArgs {
    const float* pos;
    const float* feat;
    const float* offs;
    const float* lv;
    const uint32_t* sel_idx;
    const float* sel_w;
    const ogs_counts* counts;
    ogs_mlp mlp;
    Cam cam;
    const float* dmeans;
    const float* dscales;
    const float* dquats;
    const float* drec;
    float* dfeat;
    float* doffs;
    float* dlv;
    float* rowY;         // [sel_cap][kRowY]
    float* rowH;         // [sel_cap][kRowH]
    float* rowP;         // [sel_cap][kRowP]
    float* rowZ;         // [sel_cap][kRowZ]
    float* partial;      // [kDbBlocks][kNWeights]
    float* dapp;         // f32[N][A] appearance code gradients (+=), with codes only
};

__device__ __forceinline__ float sigm(float x) { return 1.0f / (1.0f + __expf(-x)); }

// out rows of decoder m (opacity 0, colour 1, covariance 2) inside the 110 stacked outputs
__device__ __forceinline__ int out_base(int m) { return m == 0 ? 0 : (m == 1 ? kK : 4 * kK); }
__device__ __forceinline__ int dec_of(int row) { return row < kK ? 0 : (row < 4 * kK ? 1 : 2); }
// stacked output n's place in a dy row, and back (-1: padding)
__device__ __forceinline__ int out_row(int n) {
    return n < kK ? n : (n < 4 * kK ? n - kK + kRowCol : n - 4 * kK + kRowCov);
}
__device__ __forceinline__ int row_out(int e) {
    if (e < kRowCol) return e < kK ? e : -1;
    if (e < kRowCov) return e - kRowCol < 3 * kK ? e - kRowCol + kK : -1;
    return e - kRowCov < 7 * kK ? e - kRowCov + 4 * kK : -1;
}

// Gradients of one Gaussian that the decoders' backward starts from.
struct GaussGrad {
    float opac, color[3], scale[3], mean[3];
    float4 quat;
};

__device__ __forceinline__ GaussGrad load_gauss_grad(const DbArgs& a, size_t g) {
    GaussGrad o;
    o.opac = a.drec[9 * g + 5];
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        o.color[e] = a.drec[9 * g + 6 + e];
        o.scale[e] = a.dscales[3 * g + e];
        o.mean[e] = a.dmeans[3 * g + e];
    }
    o.quat = *reinterpret_cast<const float4*>(a.dquats + 4 * g);
    return o;
}

// Gradients of the loss w.r.t. a Gaussian's decoder outputs y: opacity w tanh (zero where the
// opacity was dropped), colour sigmoid, scale l_v sigmoid (its l_v term added to dlv), unit
// quaternion.
__device__ __forceinline__ void dy_opacity(const GaussGrad& g, float w, const float* y, float* dy) {
    const float th = tanhf(y[0]);
    dy[0] = w * th > 0.f ? g.opac * w * (1.f - th * th) : 0.f;
}

__device__ __forceinline__ void dy_color(const GaussGrad& g, const float* y, float* dy) {
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        const float sg = sigm(y[e]);
        dy[e] = g.color[e] * sg * (1.f - sg);
    }
}

__device__ __forceinline__ void dy_cov(const GaussGrad& g, const float (&lvv)[3], const float* y,
                                       float* dy, float (&dlv)[3]) {
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        const float sg = sigm(y[e]);
        const float gsc = g.scale[e];
        dlv[e] += gsc * sg;
        dy[e] = gsc * lvv[e] * sg * (1.f - sg);
    }
    const float n2 = y[3] * y[3] + y[4] * y[4] + y[5] * y[5] + y[6] * y[6];
    const float inv = 1.0f / sqrtf(n2);
    const float qn[4] = {y[3] * inv, y[4] * inv, y[5] * inv, y[6] * inv};
    const float gqa[4] = {g.quat.x, g.quat.y, g.quat.z, g.quat.w};
    const float dot = qn[0] * gqa[0] + qn[1] * gqa[1] + qn[2] * gqa[2] + qn[3] * gqa[3];
#pragma unroll
    for (int e = 0; e < 4; ++e) dy[3 + e] = (gqa[e] - qn[e] * dot) * inv;
}

constexpr int kDbBlocks = 2 * kSmCount;

// partial sums of the appearance weight gradients: one kH x kMaxApp row per block
constexpr int kAppItems = kH * kMaxApp;

struct DbScratch {
    float* partial;
    float *rowY, *rowH, *rowP, *rowZ;
    float* partial_app;  // [kDbBlocks][kAppItems]
};

inline size_t db_layout(int64_t sel_cap, void* base, DbScratch* s) {
    Carver cv(base);
    DbScratch t;
    const size_t n = (size_t)(sel_cap > 0 ? sel_cap : 1);
    t.partial = cv.take<float>((size_t)kDbBlocks * kNWeights);
    t.rowY = cv.take<float>(n * kRowY);
    t.rowH = cv.take<float>(n * kRowH);
    t.rowP = cv.take<float>(n * kRowP);
    t.rowZ = cv.take<float>(n * kRowZ);
    t.partial_app = cv.take<float>((size_t)kDbBlocks * kAppItems);
    if (s) *s = t;
    return cv.off + 256;
}

// Weight pass + fixed-order reduction over the rows written by a row pass (grad.cu); with
// appearance codes (a.mlp.A > 0) also the code weights' gradient dmlp.w1_app.
cudaError_t launch_weight_pass(const DbArgs& a, const DbScratch& s, const ogs_mlp& dmlp,
                               cudaStream_t st);

}  // namespace db
}  // namespace ogs
