// What the tensor-core kNN's kernels share: the candidates they buffer, the
// bound on a key's error, and the norm slices folded into the contraction.
// A key estimates ||y||^2 - 2 x.y, the squared distance less the query's norm.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "common.cuh"
#include "internal.h"

namespace atsne {

struct Cand {
    float key;
    int32_t idx;
};

// Which launch wrote a buffer's metadata (count, threshold bits, overflow, tag).
enum : int { META_FIRST = 1, META_RETRY = 2 };

constexpr int F_PARTS = 4;  // parts of a tile's columns in the fixed-threshold kernel, a buffer each (with radii one)
constexpr int FILTER_MAX_SPLITS = 64;  // its column splits at most

// Bound on |estimated - true| key (= squared distance - ||x_i||^2) for query
// row statistics st = (||x||, residual norm of its BF16 copy, norm of its low
// part) against any corpus point (gmax: the corpus maxima of the same): the
// terms the BF16 copies drop (Cauchy-Schwarz on the residual norms), the FP32
// accumulation of the products, and the FP32 norms.
__device__ __forceinline__ float key_error_bound(float4 st, const unsigned *gmax, float acc_coef,
                                                 float sq_coef) {
    const float amax = __uint_as_float(gmax[0]);
    const float rmax = __uint_as_float(gmax[1]);
    const float lmax = __uint_as_float(gmax[2]);
    const float a = st.x, r = st.y, l = st.z;
    const float drop = l * lmax + r * amax + (a + r) * rmax;
    return 2.f * drop + acc_coef * a * amax + (4e-6f + sq_coef) * amax * amax + 4e-6f * a * a;
}

// The same bound over the corpus points of norm at most amax_cap only (a
// point farther in norm than sqrt(d) from the query is farther than sqrt(d)
// in distance). Their residuals are capped by the BF16 rounding bound, the unit
// roundoff 2^-8 of 8 significand bits rounded to nearest (257 becomes 256):
// ||x - hi|| and ||lo|| are at most 2^-8 ||x||, plus a tiny absolute term for
// subnormal values.
__device__ __forceinline__ float key_error_bound_capped(float4 st, const unsigned *gmax, float acc_coef,
                                                        float sq_coef, float amax_cap) {
    const float amax = fminf(__uint_as_float(gmax[0]), amax_cap);
    const float rmax = fminf(__uint_as_float(gmax[1]), 0x1p-8f * amax + 1e-30f);
    const float lmax = fminf(__uint_as_float(gmax[2]), 0x1p-8f * amax + 1e-30f);
    const float a = st.x, r = st.y, l = st.z;
    const float drop = l * lmax + r * amax + (a + r) * rmax;
    return 2.f * drop + acc_coef * a * amax + (4e-6f + sq_coef) * amax * amax + 4e-6f * a * a;
}

// Lane l's value of a corpus row's norm slice (16 BF16): the FP32 squared norm
// n as three pieces h1 + h2 + h3 (each the rounded remainder of the previous:
// together within 2^-24 of it), then zeros.
__device__ __forceinline__ __nv_bfloat16 norm_piece(float n, int l) {
    const __nv_bfloat16 h1 = __float2bfloat16_rn(n);
    const float r1 = n - __bfloat162float(h1);
    const __nv_bfloat16 h2 = __float2bfloat16_rn(r1);
    const __nv_bfloat16 h3 = __float2bfloat16_rn(r1 - __bfloat162float(h2));
    return l == 0 ? h1 : l == 1 ? h2 : l == 2 ? h3 : __float2bfloat16_rn(0.f);
}

// The constant query slice of the folded norms: -1/2 in its first three
// columns, 128 rows of 16. Called by one block.
__device__ __forceinline__ void fold_query_slice(__nv_bfloat16 *aext) {
    for (int t = threadIdx.x; t < 128 * 16; t += blockDim.x)
        aext[t] = __float2bfloat16_rn((t & 15) < 3 ? -0.5f : 0.f);
}

// The fixed-threshold pass over a plan's workspace (knn_filter.cu).
struct FilterArgs {
    const void *a_hi, *a_lo;  // the query rows' BF16 copies
    int64_t a_rows, Q, N;
    int D;
    const int32_t *qlist;
    bool cross;               // queries from another array
    const float *radius, *hint;
    const unsigned *lo_max;
    float acc_coef, sq_coef;
    const int64_t *qcount;
};
atsne_status knn_filter_launch(const TcPlan &pl, const TcWs &w, const FilterArgs &a, cudaStream_t stream);
// Starting thresholds of the rows it gave up (TcWs::retry_rows, flag_count[1]):
// those marked +inf in TcWs::tau get the plan's second rank, the others keep theirs.
atsne_status knn_retry_tau_launch(const TcPlan &pl, const TcWs &w, cudaStream_t stream);
// Tensor maps of BF16 rows: 64-column boxes of rows of Dp (128-byte swizzle),
// and boxes of whole norm slices (rows of 16, 32-byte swizzle).
atsne_status tc_map_bf16(CUtensorMap *m, const void *base, int64_t rows, int Dp, int box_rows);
atsne_status tc_map_ext(CUtensorMap *m, const void *base, int64_t rows, int box_rows);

}  // namespace atsne
