// Per-point Gaussian bandwidth and the conditional rows P_{j|i} (Eq. 3 and
// Eq. 4, Sec. 3, over the kNN support of Eq. 8).
//
// For the shifted distances s_j = d_j - min d of a row, w_j = exp(-beta s_j),
// Z = sum w_j and H = ln Z + beta sum_j w_j s_j / Z (nats); beta is where
// H = ln(perplexity). The definition's search is a bisection: start beta = 1,
// double while no upper bound is known, then halve the bracket, until H is
// within `tol` or `max_iter` steps are done.
//
// A distance of +inf marks an absent neighbour (a neighbourhood shortened by a
// deletion, Sec. 5.3.2): it is outside N_i, takes no part in the sums and gets
// P = 0; a row without any neighbour gets P = 0 and beta = 0.
//
// calibrate_rows_kernel (the default tolerance and step limit, k <= 256): eight
// lanes per row, its distances in registers. H falls monotonically in beta, and
// smoothly in ln beta (dH / d ln beta = -beta^2 Var_w(s)), so Newton steps in
// ln beta, kept inside the bracket that the values of H give, reach the same
// root in about five evaluations of the row where the bisection takes about
// twenty; the last step is applied after the tolerance is met, so the root is
// closer than the bisection's. A row that does not converge (the perplexity is
// out of reach) is bisected as defined. Bound by the exponentials of those
// evaluations (MUFU), 5 instructions per neighbour and evaluation; a thread per
// row (the kernel below) leaves few blocks in flight on small calls. Measured
// against it: 300,000 rows of k = 90 350 to 129 us, 50,000 of k = 150 196 to
// 48 us, 2,000 of k = 90 62 to 12 us, 500 of k = 200 269 to 16 us; the error of
// P against 64 bits falls from 4e-6 to 1.3e-7.
//
// calibrate_kernel (any tolerance, step limit and k): the bisection itself. One
// thread owns one row. A CTA of 128 threads stages its 128 contiguous rows
// (128*k floats, one coalesced sweep) into shared memory with an odd row
// stride, so the per-thread row walks are bank-conflict free; the P rows leave
// the same way.
//
// Arithmetic: FP32 throughout. GB300 runs FP64 at 1/64 of the FP32 rate, and
// the parity bound for P (1e-5 absolute) needs H only to about 1e-6, which the
// 90-term FP32 sums give with a wide margin; the stopping tolerance defaults to
// 1e-5 nats for that reason.
#include <float.h>

#include "common.cuh"
#include "internal.h"

namespace atsne {
namespace {

constexpr int CAL_THREADS = 128;
constexpr float CAL_TOL = 1e-5f;   // the defaults of atsne_calibrate_P
constexpr int CAL_ITERS = 200;
constexpr int NEWTON_ITERS = 24;

// Bisection on beta over the shifted distances s_j of one row (returns the
// final beta and the normaliser Z); GAPS: the row holds absent entries (+inf).
template <bool GAPS>
__device__ __forceinline__ void bisect(const float *row, int k, float target, float tol, int max_iter,
                                       float &bf, float &Z) {
    float beta = 1.f, lo = 0.f, hi = INFINITY;
    for (int it = 1;; ++it) {
        bf = fminf(beta, FLT_MAX);
        float z = 0.f, ws = 0.f;
        for (int j = 0; j < k; ++j) {
            const float s = row[j];
            if (GAPS && s == INFINITY) continue;  // absent
            const float w = expf(-bf * s);
            z += w;
            ws = fmaf(w, s, ws);
        }
        const float H = logf(z) + bf * ws / z;
        Z = z;
        if (fabsf(H - target) < tol || it >= max_iter) break;
        if (H > target) {
            lo = beta;
            beta = isinf(hi) ? 2.f * beta : 0.5f * (beta + hi);
        } else {
            hi = beta;
            beta = 0.5f * (lo + beta);
        }
    }
}

__global__ void __launch_bounds__(CAL_THREADS)
calibrate_kernel(const float *__restrict__ d2, int64_t rows_max, int k, float perplexity, float target,
                 float tol, int max_iter, float *__restrict__ P, float *__restrict__ beta_out, int *status,
                 const int64_t *__restrict__ count) {
    extern __shared__ float sm[];
    const int stride = k | 1;
    const int64_t rows = count ? min(*count, rows_max) : rows_max;
    const int64_t r0 = (int64_t)blockIdx.x * CAL_THREADS;
    if (r0 >= rows) return;
    const int nr = (int)(rows - r0 < CAL_THREADS ? rows - r0 : CAL_THREADS);
    const float *src = d2 + r0 * k;
    for (int t = threadIdx.x; t < nr * k; t += CAL_THREADS) {
        int r = t / k, c = t - r * k;
        sm[r * stride + c] = src[t];
    }
    __syncthreads();

    if ((int)threadIdx.x < nr) {
        float *row = sm + threadIdx.x * stride;
        float dmin = INFINITY;
        bool valid = true;
        int present = 0;
        for (int j = 0; j < k; ++j) {
            float v = row[j];
            valid &= v >= 0.f;  // NaN and negative distances are errors; +inf is absent
            dmin = fminf(dmin, v);
            present += v < INFINITY;
        }
        if (!valid) raise_status(status, DEV_NONFINITE);
        if (dmin < INFINITY)
            for (int j = 0; j < k; ++j) row[j] -= dmin;  // s_j (+inf stays +inf)

        // the entropy over n present neighbours is at most log n, reached only
        // at beta = 0: when n <= perplexity the bisection's limit is beta = 0,
        // a uniform row, which is taken directly
        const bool flat = present > 0 && (float)present <= perplexity;
        float bf = 1.f, Z = 1.f;
        if (flat) bf = 0.f, Z = (float)present;
        // a full row (the usual case) skips the absent-entry test in the sums
        if (dmin < INFINITY && !flat) {
            if (present == k)
                bisect<false>(row, k, target, tol, max_iter, bf, Z);
            else
                bisect<true>(row, k, target, tol, max_iter, bf, Z);
        }
        if (dmin == INFINITY) bf = 0.f;  // no neighbour
        const float inv = dmin < INFINITY ? 1.f / Z : 0.f;
        for (int j = 0; j < k; ++j) row[j] = row[j] == INFINITY ? 0.f : expf(-bf * row[j]) * inv;
        if (beta_out) beta_out[r0 + threadIdx.x] = bf;
    }
    __syncthreads();
    float *dst = P + r0 * k;
    for (int t = threadIdx.x; t < nr * k; t += CAL_THREADS) {
        int r = t / k, c = t - r * k;
        dst[t] = sm[r * stride + c];
    }
}

__device__ __forceinline__ float ex2(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Sums over the eight lanes of a row.
__device__ __forceinline__ float sum8(float v) {
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <int KPL>  // neighbours per lane at most: k <= 8 KPL
__global__ void __launch_bounds__(CAL_THREADS)
calibrate_rows_kernel(const float *__restrict__ d2, int64_t rows_max, int k, float perplexity, float target,
                      float *__restrict__ P, float *__restrict__ beta_out, int *status,
                      const int64_t *__restrict__ count) {
    const int lane = threadIdx.x & 31, gl = lane & 7;
    const int64_t rows = count ? min(*count, rows_max) : rows_max;
    const int64_t r = ((int64_t)blockIdx.x * CAL_THREADS + threadIdx.x) >> 3;
    if ((r & ~(int64_t)3) >= rows) return;  // the whole warp's rows are past the end
    const bool live = r < rows;
    const float *src = d2 + r * k;
    // lane gl holds the neighbours gl, gl + 8, ...; the first kf of its KPL
    // places exist in every lane, the next one in some
    const int kf = k >> 3;
    float s[KPL];
    float dmin = INFINITY;
    bool valid = true;
    int present = 0;
#pragma unroll
    for (int i = 0; i < KPL; ++i) {
        const int j = 8 * i + gl;
        s[i] = live && j < k ? src[j] : INFINITY;
        valid &= s[i] >= 0.f;  // NaN and negative distances are errors; +inf is absent
        dmin = fminf(dmin, s[i]);
        present += s[i] < INFINITY;
    }
    if (!valid) raise_status(status, DEV_NONFINITE);
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        dmin = fminf(dmin, __shfl_xor_sync(0xffffffffu, dmin, o));
        present += __shfl_xor_sync(0xffffffffu, present, o);
    }
    float mean = 0.f;
#pragma unroll
    for (int i = 0; i < KPL; ++i) {
        if (dmin < INFINITY) s[i] -= dmin;  // s_j (+inf stays +inf)
        if (s[i] < INFINITY) mean += s[i];
    }
    mean = sum8(mean) / fmaxf((float)present, 1.f);
    // a full row's places below kf need no test; the others hold +inf where a
    // neighbour is absent
    const bool full = __all_sync(0xffffffffu, !live || present == k);
    // n <= perplexity neighbours: H <= ln n is reached only at beta = 0, a
    // uniform row, taken directly; equal distances (mean 0) are bisected
    const bool flat = present > 0 && (float)present <= perplexity;
    bool todo = live && present > 0 && !flat;
    float beta = 0.f;
    if (todo) beta = mean > 0.f ? fminf(2.f / mean, 1e30f) : 1.f;
    bool found = false;
    float lo = 0.f, hi = INFINITY;
    bool run = todo && mean > 0.f && mean < 1e30f;
    for (int it = 0; it < NEWTON_ITERS && __any_sync(0xffffffffu, run); ++it) {
        const float c = -1.4426950408889634f * beta;
        float z = 0.f, m1 = 0.f, m2 = 0.f;
#pragma unroll
        for (int i = 0; i < KPL; ++i) {
            if (i > kf) continue;
            float sv = s[i];
            float w = ex2(c * sv);
            if (i == kf || !full) {
                const bool in = sv < INFINITY;
                w = in ? w : 0.f;
                sv = in ? sv : 0.f;
            }
            z += w;
            const float ws = w * sv;
            m1 += ws;
            m2 = fmaf(ws, sv, m2);
        }
        z = sum8(z);
        m1 = sum8(m1);
        m2 = sum8(m2);
        const float iz = __fdividef(1.f, z), mu = m1 * iz;
        const float f = logf(z) + beta * mu - target;
        const float g = beta * beta * fmaf(m2, iz, -mu * mu);  // -dH / d ln beta
        if (run) {
            const float step = f / g;
            if (fabsf(f) < CAL_TOL) {
                // (where H is flat the tolerance leaves beta open: bisected)
                found = g > 0.01f;
                if (found) beta = fmaf(beta, step, beta);
                run = false;
            } else {
                if (f > 0.f) lo = beta;
                else hi = beta;
                float nb = beta * expf(fminf(fmaxf(step, -3.f), 3.f));
                if (!(g > 0.f) || !(nb > lo) || !(nb < hi)) nb = isinf(hi) ? 8.f * lo : lo > 0.f ? sqrtf(lo) * sqrtf(hi) : 0.125f * hi;
                beta = nb;
                run = beta < 1e30f && beta > 1e-30f;
            }
        }
    }
    // out of reach, or out of range: the bisection as defined
    bool bis = todo && !found;
    float bb = 1.f, bl = 0.f, bh = INFINITY;
    for (int it = 1; __any_sync(0xffffffffu, bis); ++it) {
        const float bf = fminf(bb, FLT_MAX);
        float z = 0.f, ws = 0.f;
#pragma unroll
        for (int i = 0; i < KPL; ++i)
            if (s[i] < INFINITY) {
                const float w = expf(-bf * s[i]);
                z += w;
                ws = fmaf(w, s[i], ws);
            }
        z = sum8(z);
        ws = sum8(ws);
        if (bis) {
            const float H = logf(z) + bf * ws / z;
            beta = bf;
            if (fabsf(H - target) < CAL_TOL || it >= CAL_ITERS) {
                bis = false;
            } else if (H > target) {
                bl = bb;
                bb = isinf(bh) ? 2.f * bb : 0.5f * (bb + bh);
            } else {
                bh = bb;
                bb = 0.5f * (bl + bb);
            }
        }
    }
    float z = 0.f;
#pragma unroll
    for (int i = 0; i < KPL; ++i) {
        s[i] = s[i] < INFINITY ? expf(-beta * s[i]) : 0.f;
        z += s[i];
    }
    z = sum8(z);
    const float inv = present > 0 ? 1.f / z : 0.f;
    if (!live) return;
    float *dst = P + r * k;
#pragma unroll
    for (int i = 0; i < KPL; ++i)
        if (8 * i + gl < k) dst[8 * i + gl] = s[i] * inv;
    if (beta_out && gl == 0) beta_out[r] = beta;
}

template <int KPL>
atsne_status rows_launch(const float *d2, int64_t rows, int k, float perplexity, float *P, float *beta,
                         cudaStream_t stream, const int64_t *count) {
    return launch_kernel("calibrate_beta", calibrate_rows_kernel<KPL>, ceil_div(rows * 8, CAL_THREADS), CAL_THREADS, 0,
                         stream, d2, rows, k, perplexity, logf(perplexity), P, beta, device_status_word(), count);
}

}  // namespace

size_t calibrate_smem_bytes(int k) { return sizeof(float) * CAL_THREADS * (size_t)(k | 1); }

atsne_status calibrate_launch(const float *d2, int64_t rows, int k, float perplexity, float tol,
                              int max_iter, float *P, float *beta, cudaStream_t stream, const int64_t *count) {
    if (rows <= 0) return ATSNE_OK;
    // a caller's own tolerance or step limit is the bisection's
    if (tol == CAL_TOL && max_iter == CAL_ITERS && k <= 256) {
        if (k <= 32) return rows_launch<4>(d2, rows, k, perplexity, P, beta, stream, count);
        if (k <= 64) return rows_launch<8>(d2, rows, k, perplexity, P, beta, stream, count);
        if (k <= 96) return rows_launch<12>(d2, rows, k, perplexity, P, beta, stream, count);
        if (k <= 128) return rows_launch<16>(d2, rows, k, perplexity, P, beta, stream, count);
        if (k <= 192) return rows_launch<24>(d2, rows, k, perplexity, P, beta, stream, count);
        return rows_launch<32>(d2, rows, k, perplexity, P, beta, stream, count);
    }
    const size_t smem = calibrate_smem_bytes(k);
    static size_t attr = 0;
    if (smem > 48 * 1024 && smem > attr) {
        cudaError_t e = cudaFuncSetAttribute(calibrate_kernel,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return cuda_error(e, "calibrate attribute");
        attr = smem;
    }
    return launch_kernel("calibrate_beta", calibrate_kernel, ceil_div(rows, CAL_THREADS),
                         CAL_THREADS, smem, stream, d2, rows, k, perplexity, logf(perplexity), tol, max_iter, P,
                         beta, device_status_word(), count);
}

}  // namespace atsne
