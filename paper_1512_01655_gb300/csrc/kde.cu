// Density-based view of the embedding and its approximation map (Sec. 5.2):
// per pixel p of a W x H image over the 2-D embedding, with a Gaussian kernel
// G(d, h) = exp(-d^2 / (2 h^2)) / (2 pi h^2),
//   F = sum_i G(|p - y_i|, h),  S = sum_{i selected} G,  R = sum_i rho_i G,
//   f = F / N (Eq. 12),  s = S / F (Eq. 13, selected share),
//   a = R / F (Sec. 5.2.2, rho-weighted mean),  alpha = 1 - a^k (the lens).
// Points farther than cutoff * h from a pixel are left out of its sums
// (cutoff 0: every point counts).
//
// A cluster of CTAs renders a 32 x 32 tile, each CTA its share of the points
// (every CL-th chunk of KDE_CHUNK), so that a tile over a dense cluster does not
// outlast the others. A CTA streams its points in index order and keeps those
// within reach of the tile's pixel centres in shared memory, in that order.
// Two warps own each 16 x 16 pixels, 4 x 2 per lane, and half of the kept
// points. A warp takes its points in order, a lane testing each against the
// warp's pixels: out of reach of all of them (skipped), within reach of all (no
// test per pixel) or of some. The kernel is separable, exp(-(dx^2 + dy^2) /
// 2h^2) = ex(dx) ey(dy): for 16 such points at a time the lanes compute the
// 16 + 16 factors, and a pixel then costs one FMA per sum. No atomics: each
// warp's sums are taken in point order and added in a fixed order, so the image
// does not depend on scheduling.
//
// Bound by the FP32 pipe (3 to 6 instructions per pixel and point in reach) and
// by the scan of all points for every tile (the call has no workspace to bin
// them in), about half of the time each. A pass with one exponential per pixel
// and point over 16 x 16 tiles took 1,000 us on 70,000 points and 1024 x 1024
// pixels (h 0.3, cutoff 4 h); this one takes 427 us, and its sums are closer to
// the FP64 ones (f 8e-7 to 1.2e-7).
#include <math.h>

#include "common.cuh"
#include "internal.h"
#include "tc_ptx.cuh"

namespace atsne {
namespace {

constexpr int KT = 32;             // tile side
constexpr int KDE_SHARES = 2;      // warps per 16 x 16 pixels
constexpr int KDE_WARPS = 4 * KDE_SHARES;  // 16 x 16 pixels each
constexpr int KDE_BLOCKS = 3;      // per SM
constexpr int KDE_THREADS = 32 * KDE_WARPS;
constexpr int KDE_PT = 4;          // points examined per thread and step
constexpr int KDE_CHUNK = KDE_PT * KDE_THREADS;
constexpr int KDE_BUF = KDE_CHUNK + 512;  // points kept: evaluated once there is no room for another chunk
constexpr int KDE_XS = 20;         // stride of a point's 16 factors (16-byte rows)

struct KdeSmem {
    float4 pt[KDE_BUF];  // x, y, selection weight, rho
    float ex[KDE_WARPS][16 * KDE_XS], ey[KDE_WARPS][16 * KDE_XS];
    float4 bp[KDE_WARPS][16];      // the points of a warp's batch
    int queue[KDE_WARPS][64];      // kept points in reach of the warp: index, | 1 << 30 where all pixels are in reach
    float cx[KT], cy[KT];          // pixel centres
    int wcount[2][KDE_WARPS];
};
static_assert(sizeof(float4) * KDE_BUF + sizeof(float) * KDE_WARPS * 32 * KDE_XS >= KDE_SHARES * 3 * KT * KT * sizeof(float),
              "the warps' sums take the points' and factors' place");

// Pixel centre i along one axis, in FP32 with one rounding: the decision
// "within cutoff * h" is the kernel's and is restated exactly so.
__device__ __forceinline__ float kde_centre(int i, float px, float x0) { return __fmaf_rn((float)i + 0.5f, px, x0); }

// The smallest and largest |c - v| over pixel centres c in [c0, c1] (FP32
// differences, monotone in c).
__device__ __forceinline__ void kde_reach(float c0, float c1, float v, float &lo, float &hi) {
    const float a = __fsub_rn(c0, v), b = __fsub_rn(c1, v);
    hi = fmaxf(fabsf(a), fabsf(b));
    lo = a <= 0.f && b >= 0.f ? 0.f : fminf(fabsf(a), fabsf(b));
}

__device__ __forceinline__ float kde_ex2(float x) {
    float r;
    asm("ex2.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

template <int CL>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(KDE_THREADS, KDE_BLOCKS)
kde_kernel(const float2 *__restrict__ Y, int64_t N, const float *__restrict__ rho,
           const uint8_t *__restrict__ sel, float x0, float y0, float px, int W, int H, float h,
           float cutoff, float lens_k, float *__restrict__ f_out, float *__restrict__ s_out,
           float *__restrict__ a_out, float *__restrict__ alpha_out) {
    extern __shared__ __align__(16) unsigned char kde_raw[];
    KdeSmem &sm = *reinterpret_cast<KdeSmem *>(kde_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tx = (blockIdx.x / CL) * KT, ty = blockIdx.y * KT, part = blockIdx.x % CL;
    const int wx = (warp & 1) * 16, wy = ((warp >> 1) & 1) * 16;  // the warp's pixels in the tile
    const int share = warp >> 2;                                  // and its share of the kept points
    const int lx = wx + (lane & 3) * 4, ly = wy + (lane >> 2) * 2;  // the lane's
    const float r = cutoff > 0.f ? __fmul_rn(cutoff, h) : INFINITY;
    const float r2 = __fmul_rn(r, r);
    const float c2 = -1.4426950408889634f / (2.f * h * h);  // ex(d) = 2^(c2 d^2)
    const float norm = 1.f / (2.f * 3.14159265358979f * h * h);
    if (tid < KT) sm.cx[tid] = kde_centre(tx + tid, px, x0);
    else if (tid < 2 * KT) sm.cy[tid - KT] = kde_centre(ty + tid - KT, px, y0);
    __syncthreads();
    float F[2][4], S[2][4], R[2][4], cx[4], cy[2];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        cx[i] = sm.cx[lx + i];
#pragma unroll
        for (int j = 0; j < 2; ++j) F[j][i] = S[j][i] = R[j][i] = 0.f;
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) cy[j] = sm.cy[ly + j];
    float *ex = sm.ex[warp], *ey = sm.ey[warp];
    float4 *bp = sm.bp[warp];
    int *queue = sm.queue[warp];

    // the queue's first n (at most 16) points added to the warp's pixels
    auto batch = [&](int n) {
        const int q = lane & 15;
        if (q < n) {
            const float4 p = sm.pt[queue[q] & 0xffff];
            const bool xs = lane < 16;  // lanes 0-15 the x factors, 16-31 the y factors
            const float *cc = xs ? sm.cx + wx : sm.cy + wy;
            const float v = xs ? p.x : p.y;
            float *o = (xs ? ex : ey) + q * KDE_XS;
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const float d = __fsub_rn(cc[i], v);
                o[i] = kde_ex2(c2 * (d * d));
            }
            if (xs) bp[q] = p;
        }
        __syncwarp();
#pragma unroll 2
        for (int t = 0; t < n; ++t) {
            const float4 p = bp[t];
            const float4 e4 = *reinterpret_cast<const float4 *>(ex + t * KDE_XS + (lane & 3) * 4);
            const float2 f2 = *reinterpret_cast<const float2 *>(ey + t * KDE_XS + (lane >> 2) * 2);
            const float e[4] = {e4.x, e4.y, e4.z, e4.w}, fy[2] = {f2.x, f2.y};
            if (queue[t] >> 30) {
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const float fs = fy[j] * p.z, fr = fy[j] * p.w;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        F[j][i] = fmaf(e[i], fy[j], F[j][i]);
                        S[j][i] = fmaf(e[i], fs, S[j][i]);
                        R[j][i] = fmaf(e[i], fr, R[j][i]);
                    }
                }
            } else {
                float dx[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) dx[i] = __fsub_rn(cx[i], p.x);
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const float dy = __fsub_rn(cy[j], p.y), dy2 = __fmul_rn(dy, dy);
                    const float fs = fy[j] * p.z, fr = fy[j] * p.w;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        // (left out, not added as 0: rho may be any value)
                        if (__fmaf_rn(dx[i], dx[i], dy2) <= r2) {
                            F[j][i] = fmaf(e[i], fy[j], F[j][i]);
                            S[j][i] = fmaf(e[i], fs, S[j][i]);
                            R[j][i] = fmaf(e[i], fr, R[j][i]);
                        }
                    }
                }
            }
        }
        __syncwarp();
    };
    const float rx0 = sm.cx[wx], rx1 = sm.cx[wx + 15], ry0 = sm.cy[wy], ry1 = sm.cy[wy + 15];
    // the kept points [0, n), in order
    auto evaluate = [&](int all) {
        const int first = share * all / KDE_SHARES, n = (share + 1) * all / KDE_SHARES;
        int qn = 0;
        for (int b = first; b < n; b += 32) {
            bool in = false, inner = false;
            if (b + lane < n) {
                const float4 p = sm.pt[b + lane];
                float xl, xh, yl, yh;
                kde_reach(rx0, rx1, p.x, xl, xh);
                kde_reach(ry0, ry1, p.y, yl, yh);
                in = __fmaf_rn(xl, xl, __fmul_rn(yl, yl)) <= r2;
                inner = __fmaf_rn(xh, xh, __fmul_rn(yh, yh)) <= r2;
            }
            const unsigned m = __ballot_sync(0xffffffffu, in);
            if (in) queue[qn + __popc(m & ((1u << lane) - 1u))] = (b + lane) | (inner ? 1 << 30 : 0);
            qn += __popc(m);
            __syncwarp();
            while (qn >= 16) {
                batch(16);
                qn -= 16;
                const int a = lane < qn ? queue[16 + lane] : 0;  // at most 31 left
                __syncwarp();
                if (lane < qn) queue[lane] = a;
                __syncwarp();
            }
        }
        if (qn > 0) batch(qn);
    };

    // kept: not beyond reach of the tile along either axis (false for NaN); the
    // bounds are a little wide, the warps decide
    const float wide = r * 1.00001f;
    const float bx0 = sm.cx[0] - wide - 1e-6f * fabsf(sm.cx[0]), bx1 = sm.cx[KT - 1] + wide + 1e-6f * fabsf(sm.cx[KT - 1]);
    const float by0 = sm.cy[0] - wide - 1e-6f * fabsf(sm.cy[0]), by1 = sm.cy[KT - 1] + wide + 1e-6f * fabsf(sm.cy[KT - 1]);
    int fill = 0, par = 0;
    float2 nxt[KDE_PT];  // the next chunk's points (a warp's are consecutive)
    const int first = warp * 32 * KDE_PT + lane;
#pragma unroll
    for (int u = 0; u < KDE_PT; ++u) {
        const int64_t i = part * KDE_CHUNK + first + 32 * u;
        nxt[u] = i < N ? Y[i] : make_float2(NAN, NAN);
    }
    for (int64_t c0 = part * KDE_CHUNK; c0 < N; c0 += CL * KDE_CHUNK, par ^= 1) {
        float2 y[KDE_PT];
        unsigned m[KDE_PT];
        int kept = 0;
#pragma unroll
        for (int u = 0; u < KDE_PT; ++u) {
            y[u] = nxt[u];
            const int64_t i = c0 + CL * KDE_CHUNK + first + 32 * u;
            nxt[u] = i < N ? Y[i] : make_float2(NAN, NAN);
            m[u] = __ballot_sync(0xffffffffu, y[u].x >= bx0 && y[u].x <= bx1 && y[u].y >= by0 && y[u].y <= by1);
            kept += __popc(m[u]);
        }
        if (lane == 0) sm.wcount[par][warp] = kept;
        __syncthreads();
        const unsigned wc = lane < KDE_WARPS ? (unsigned)sm.wcount[par][lane] : 0u;
        int pos = fill + (int)__reduce_add_sync(0xffffffffu, lane < warp ? wc : 0u);
        fill += (int)__reduce_add_sync(0xffffffffu, wc);
        if (kept) {
#pragma unroll
            for (int u = 0; u < KDE_PT; ++u) {
                if ((m[u] >> lane) & 1u) {
                    const int64_t i = c0 + first + 32 * u;
                    sm.pt[pos + __popc(m[u] & ((1u << lane) - 1u))] =
                        make_float4(y[u].x, y[u].y, sel ? (sel[i] ? 1.f : 0.f) : 0.f, rho ? rho[i] : 1.f);
                }
                pos += __popc(m[u]);
            }
        }
        if (fill > KDE_BUF - KDE_CHUNK) {  // uniform over the block
            __syncthreads();
            evaluate(fill);
            __syncthreads();
            fill = 0;
        }
    }
    __syncthreads();
    evaluate(fill);
    auto write = [&](int x, int y, float f, float sv, float rv) {
        const int ix = tx + x, iy = ty + y;
        if (ix >= W || iy >= H) return;
        const int64_t o = (int64_t)iy * W + ix;
        const float a = f > 0.f ? rv / f : 1.f;
        if (f_out) f_out[o] = f * norm / (float)N;
        if (s_out) s_out[o] = f > 0.f ? sv / f : 0.f;
        if (a_out) a_out[o] = a;
        if (alpha_out) alpha_out[o] = 1.f - powf(fmaxf(a, 0.f), lens_k);
    };
    // the warps' sums added over their shares, then over the cluster's CTAs,
    // each of which writes a part of the pixels
    constexpr int NP = KT * KT;
    __syncthreads();
    float *mine = reinterpret_cast<float *>(kde_raw);  // [share][3][NP]
    {
        float *o = mine + share * 3 * NP;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int at = (ly + j) * KT + lx;
            *reinterpret_cast<float4 *>(o + at) = make_float4(F[j][0], F[j][1], F[j][2], F[j][3]);
            *reinterpret_cast<float4 *>(o + NP + at) = make_float4(S[j][0], S[j][1], S[j][2], S[j][3]);
            *reinterpret_cast<float4 *>(o + 2 * NP + at) = make_float4(R[j][0], R[j][1], R[j][2], R[j][3]);
        }
    }
    __syncthreads();
    for (int q = tid; q < 3 * NP; q += KDE_THREADS)
        for (int u = 1; u < KDE_SHARES; ++u) mine[q] += mine[3 * NP * u + q];
    if (CL > 1) tc::cluster_sync();
    else __syncthreads();
    for (int q = part * (NP / CL) + tid; q < (part + 1) * (NP / CL); q += KDE_THREADS) {
        float v[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int c = 0; c < CL; ++c)
#pragma unroll
            for (int t = 0; t < 3; ++t)
                v[t] += CL == 1 ? mine[t * NP + q]
                                : __uint_as_float(tc::ld_cluster(tc::map_to_rank(tc::smem_u32(mine + t * NP + q), c)));
        write(q % KT, q / KT, v[0], v[1], v[2]);
    }
    if (CL > 1) tc::cluster_sync();
}

template <int CL>
atsne_status kde_launch_t(const float *Y, int64_t N, const float *rho, const uint8_t *selected, float x0, float y0,
                          float pixel, int W, int H, float h, float cutoff, float lens_k, float *f_out, float *s_out,
                          float *a_out, float *alpha_out, cudaStream_t stream) {
    const size_t smem = sizeof(KdeSmem);
    cudaError_t e = cudaFuncSetAttribute(kde_kernel<CL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_error(e, "kde attribute");
    const dim3 grid((unsigned)(ceil_div(W, KT) * CL), (unsigned)ceil_div(H, KT));
    return launch_kernel("kde_map", kde_kernel<CL>, grid, KDE_THREADS, smem, stream,
                         reinterpret_cast<const float2 *>(Y), N, rho, selected, x0, y0, pixel, W, H, h, cutoff,
                         lens_k, f_out, s_out, a_out, alpha_out);
}

}  // namespace

atsne_status kde_launch(const float *Y, int64_t N, const float *rho, const uint8_t *selected, float x0,
                        float y0, float pixel, int W, int H, float h, float cutoff, float lens_k,
                        float *f_out, float *s_out, float *a_out, float *alpha_out,
                        cudaStream_t stream) {
    // CTAs per tile: more where the image has few tiles to balance with (300 x
    // 400 pixels, 200,000 points: 1,597 us with one CTA scanning for each 16 x
    // 16 tile, 658 us with four per tile here, 470 us with eight; 1024 x 1024
    // and 70,000: 1,000, 427 and 468 us), fewer where a CTA's share would be
    // under one or two chunks (5,000 points on 1,100 x 500: 35, 37 and, with
    // two, 33 us)
    const int64_t tiles = (int64_t)ceil_div(W, KT) * ceil_div(H, KT);
#define KDE_ARGS Y, N, rho, selected, x0, y0, pixel, W, H, h, cutoff, lens_k, f_out, s_out, a_out, alpha_out, stream
    if (N >= 8 * KDE_CHUNK && tiles <= 4 * num_sms()) return kde_launch_t<8>(KDE_ARGS);
    if (N >= 16 * KDE_CHUNK) return kde_launch_t<4>(KDE_ARGS);
    if (N > KDE_CHUNK) return kde_launch_t<2>(KDE_ARGS);
    return kde_launch_t<1>(KDE_ARGS);
#undef KDE_ARGS
}

}  // namespace atsne
