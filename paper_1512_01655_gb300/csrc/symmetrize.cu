// Symmetrised joint P as CSR (Eq. 2 in the split form of Eq. 10, Sec. 4.3).
//
// Row r of P is the union of its forward entries F_r = N_r (k, fewer where a
// deletion left absent entries, index -1, Sec. 5.3.2) and its reverse entries
// R_r = {i : r in N_i}; a column in both (a mutual pair) gets
// (p_{c|r} + p_{r|c}) / 2N, formed from the same two operands on both sides,
// so p_rc and p_cr are bit-identical; a column in one of them gets its one
// conditional / 2N.
//   1. count: every entry (i -> j) counted into its target row; the atomic's
//             old value is the entry's place in j's reverse list.
//   2. scan:  offsets of the reverse lists.
//   3. place: (i, p_{j|i}) written to that place, one 8-byte write per entry.
//   4. merge: row r's k + |R_r| entries sorted by column, mutual pairs added,
//             the row kept in the workspace (its first |R_r| entries in its
//             reverse list's place, which it has read, the up to k others in k
//             places of its own) and its length kept. Rows of up to 512 entries
//             are sorted by a warp in registers (sym_merge_kernel), up to 1024
//             the same with more registers (sym_mid_kernel); of longer ones (hub
//             rows) only the length is taken, |F_r| + |R_r| less the neighbours
//             that list r.
//   5. scan:  row_ptr.
//   6. copy:  rows to their final places, scaled by 1 / 2N; a hub row is written
//             there by a CTA that takes each entry's rank from a bitmap of the
//             columns (sym_hub_kernel).
// A warp's sort moves one word per entry: column, forward/reverse bit and the
// entry's slot (where its value waits in shared memory) in 32 bits while the
// column fits (N < 2^21), else 64; a compare-exchange is a shuffle and a
// min/max. Sorting forward and reverse rows separately as (key, value) pairs in
// shared memory, with a binary search of each entry in the other list, twice,
// took 3.08, 13.7 and 1.63 ms (300,000 rows of separate clusters, 1,000,000
// Gamma rows, 70,000 byte rows with hubs; k = 90); this takes 1.62, 6.4 and
// 0.45 ms. The bounds are the atomics and the scatter of steps 1 and 3 (a
// 32-byte sector per 8-byte write) and the sorts' instructions.
#include <limits.h>

#include "common.cuh"
#include "internal.h"

namespace atsne {
namespace {

constexpr int SYM_WARPS = 4;
constexpr int SYM_BULK = 512;         // entries of a row sorted by sym_merge_kernel
constexpr int SYM_MID = 1024;         // by sym_mid_kernel
// Below so many rows an entry's key fits 32 bits: 21 column bits, the reverse
// bit, 10 slot bits. With one row more, the last column's reverse entry in the
// last slot would be all ones, the mark for no entry.
constexpr int64_t SYM_KEY32 = int64_t(1) << 21;
constexpr int HUB_THREADS = 1024;
constexpr int SYM_MAX_K = 512;
constexpr int64_t HUB_COLS = int64_t(1) << 19;   // columns per bitmap (64 KB, and as much for its prefix sums)

// A row's neighbour j of row i is valid; absent ones are skipped, others raise the status.
__device__ __forceinline__ bool valid_neighbour(int j, int64_t i, int64_t N, int *status) {
    if (j == -1) return false;
    if (j >= 0 && j < N && j != i) return true;
    raise_status(status, DEV_MALFORMED);
    return false;
}

__global__ void __launch_bounds__(256)
sym_count_kernel(const int32_t *__restrict__ idx, int64_t N, int k, int32_t *__restrict__ rank,
                 int32_t *__restrict__ rcnt, int *status) {
    const int lane = threadIdx.x & 31;
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= N) return;
    for (int t0 = lane; t0 < k; t0 += 128) {  // four atomics in flight per lane
        int j[4], n[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) j[u] = t0 + 32 * u < k ? idx[i * k + t0 + 32 * u] : -1;
#pragma unroll
        for (int u = 0; u < 4; ++u) n[u] = valid_neighbour(j[u], i, N, status) ? atomicAdd(&rcnt[j[u]], 1) : -1;
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (t0 + 32 * u < k) rank[i * k + t0 + 32 * u] = n[u];
    }
}

__global__ void __launch_bounds__(256)
sym_place_kernel(const int32_t *__restrict__ idx, const float *__restrict__ P, int64_t N, int k,
                 const int32_t *__restrict__ rank, const int64_t *__restrict__ roff, int2 *__restrict__ rev) {
    const int lane = threadIdx.x & 31;
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= N) return;
    for (int t0 = lane; t0 < k; t0 += 128) {
        int n[4], j[4];
        float p[4];
        int64_t at[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const bool on = t0 + 32 * u < k;
            n[u] = on ? rank[i * k + t0 + 32 * u] : -1;
            j[u] = on ? idx[i * k + t0 + 32 * u] : -1;
            p[u] = on ? P[i * k + t0 + 32 * u] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) at[u] = n[u] >= 0 ? roff[j[u]] + n[u] : -1;
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (at[u] >= 0) rev[at[u]] = make_int2((int)i, __float_as_int(p[u]));
    }
}

// Ascending bitonic sort of 32 R distinct keys, lane l's being elements
// l R .. l R + R - 1: exchanges between elements fewer than R apart stay in a
// lane, the others are shuffles.
template <int R, typename K>
__device__ __forceinline__ void warp_sort_keys(K (&k)[R], int lane) {
    // (the loops over sizes and lane distances stay loops: unrolled, the sorts of
    // all R overflow the instruction cache, the 300,000 rows took 0.99 ms instead of 0.79)
#pragma unroll 1
    for (int size = 2; size <= 32 * R; size <<= 1) {
        const bool lane_up = ((lane * R) & size) == 0;  // direction of this lane's elements, size >= R
#pragma unroll 1
        for (int stride = size >> 1; stride >= R; stride >>= 1) {
            const int lm = stride / R;
            const bool keep_min = ((lane & lm) == 0) == lane_up;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const K o = __shfl_xor_sync(0xffffffffu, k[r], lm);
                k[r] = keep_min ? min(k[r], o) : max(k[r], o);
            }
        }
#pragma unroll
        for (int stride = R >> 1; stride > 0; stride >>= 1) {
            if (stride < size) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    if (r & stride) continue;
                    const bool up = size >= R ? lane_up : (r & size) == 0;
                    const K a = k[r], b = k[r + stride], lo = min(a, b), hi = max(a, b);
                    k[r] = up ? lo : hi;
                    k[r + stride] = up ? hi : lo;
                }
            }
        }
    }
}

struct SymRow {
    const int32_t *idx;
    const float *P;
    int64_t N;
    int k;
    const int64_t *roff;
    int2 *rev;   // reverse lists (column, value); then the first entries of the union's rows, not yet scaled
    int2 *tail;  // their other entries, [N][k]
    int32_t *len;
    int *status;
};

// One row of at most 32 R entries by one warp; v, oc, ov: 32 R words of shared
// memory each (values by slot, then the row as it will be written).
template <int R, typename K>
__device__ __forceinline__ void sym_merge_row(const SymRow &s, int64_t r, int m, float *v, int *oc, float *ov,
                                              int lane) {
    constexpr int SB = R == 2 ? 6 : R == 4 ? 7 : R == 8 ? 8 : R == 16 ? 9 : 10;  // slot bits
    static_assert(1 << SB == 32 * R, "a slot per entry");
    constexpr K NONE = ~K(0);
    const int64_t b0 = s.roff[r], row = r * s.k;
    K key[R];
#pragma unroll
    for (int q = 0; q < R; ++q) {
        const int slot = q * 32 + lane;
        key[q] = NONE;
        if (slot < s.k) {
            const int j = s.idx[row + slot];
            v[slot] = s.P[row + slot];
            if (j >= 0 && j < s.N && j != r) key[q] = ((K)j << (SB + 1)) | (K)slot;
        } else if (slot < s.k + m) {
            const int2 e = s.rev[b0 + slot - s.k];
            v[slot] = __int_as_float(e.y);
            key[q] = ((K)e.x << (SB + 1)) | (K(1) << SB) | (K)slot;
        }
    }
    warp_sort_keys<R>(key, lane);
    __syncwarp();
    // a forward and a reverse entry of one column are neighbours, the forward
    // one first: the first of a column's entries heads it
    K before = __shfl_up_sync(0xffffffffu, key[R - 1], 1);
    const K after = __shfl_down_sync(0xffffffffu, key[0], 1);
    if (lane == 0) before = NONE;
    int heads = 0;
    bool twice = false;  // a column listed twice in the forward row
#pragma unroll
    for (int q = 0; q < R; ++q) {
        const K p = q ? key[q - 1] : before;
        const bool same = p != NONE && (p >> (SB + 1)) == (key[q] >> (SB + 1));
        heads += key[q] != NONE && !same;
        twice |= key[q] != NONE && same && !((key[q] >> SB) & 1);
    }
    if (twice) raise_status(s.status, DEV_MALFORMED);
    int incl = heads;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    int pos = incl - heads;
#pragma unroll
    for (int q = 0; q < R; ++q) {
        const K p = q ? key[q - 1] : before;
        const bool head = key[q] != NONE && !(p != NONE && (p >> (SB + 1)) == (key[q] >> (SB + 1)));
        if (head) {
            const K n = q + 1 < R ? key[q + 1] : lane < 31 ? after : NONE;
            float x = v[(int)(key[q] & ((K(1) << SB) - 1))];
            if (n != NONE && (n >> (SB + 1)) == (key[q] >> (SB + 1))) x += v[(int)(n & ((K(1) << SB) - 1))];
            oc[pos] = (int)(key[q] >> (SB + 1));
            ov[pos] = x;
            ++pos;
        }
    }
    __syncwarp();
    int2 *first = s.rev + b0, *rest = s.tail + (row - m);
    for (int t = lane; t < total; t += 32) (t < m ? first : rest)[t] = make_int2(oc[t], __float_as_int(ov[t]));
    if (lane == 0) s.len[r] = total;
}

template <typename K>
__global__ void __launch_bounds__(SYM_WARPS * 32)
sym_merge_kernel(SymRow s, int32_t *__restrict__ mid_rows, int32_t *__restrict__ hub_rows, int32_t *__restrict__ n_list) {
    __shared__ float v[SYM_WARPS][SYM_BULK], ov[SYM_WARPS][SYM_BULK];
    __shared__ int oc[SYM_WARPS][SYM_BULK];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t r = (int64_t)blockIdx.x * SYM_WARPS + w;
    if (r >= s.N) return;
    const int64_t m64 = s.roff[r + 1] - s.roff[r];
    if (m64 + s.k > SYM_BULK) {
        if (lane == 0) {
            if (m64 + s.k > SYM_MID) {
                hub_rows[atomicAdd(n_list + 1, 1)] = (int)r;
                s.len[r] = (int)m64;  // the forward entries follow in sym_mid_kernel
            } else {
                mid_rows[atomicAdd(n_list, 1)] = (int)r;
            }
        }
        return;
    }
    const int m = (int)m64, n = m + s.k;
    if (n <= 64) sym_merge_row<2, K>(s, r, m, v[w], oc[w], ov[w], lane);
    else if (n <= 128) sym_merge_row<4, K>(s, r, m, v[w], oc[w], ov[w], lane);
    else if (n <= 256) sym_merge_row<8, K>(s, r, m, v[w], oc[w], ov[w], lane);
    else sym_merge_row<16, K>(s, r, m, v[w], oc[w], ov[w], lane);
}

template <typename K>
__global__ void __launch_bounds__(SYM_WARPS * 32)
sym_mid_kernel(SymRow s, const int32_t *__restrict__ mid_rows, const int32_t *__restrict__ hub_rows,
               const int32_t *__restrict__ n_list) {
    __shared__ float v[SYM_WARPS][SYM_MID], ov[SYM_WARPS][SYM_MID];
    __shared__ int oc[SYM_WARPS][SYM_MID];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int q = blockIdx.x * SYM_WARPS + w; q < n_list[0]; q += gridDim.x * SYM_WARPS) {
        const int64_t r = mid_rows[q];
        sym_merge_row<32, K>(s, r, (int)(s.roff[r + 1] - s.roff[r]), v[w], oc[w], ov[w], lane);
        __syncwarp();
    }
    // the hub rows' lengths: eight lanes per forward entry, which adds one to its
    // row's reverse entries unless its column lists the row (and is among them)
    const int64_t items = (int64_t)n_list[1] * s.k;
    const int gl = lane & 7;
    const unsigned group = 0xffu << (lane & 24);
    for (int64_t q = (int64_t)(blockIdx.x * SYM_WARPS + w) * 4 + (lane >> 3); q < items;
         q += (int64_t)gridDim.x * SYM_WARPS * 4) {
        const int64_t r = hub_rows[q / s.k];
        const int c = s.idx[r * s.k + q % s.k];
        if (c < 0 || c >= s.N || c == r) continue;
        const int32_t *row = s.idx + (int64_t)c * s.k;
        bool mutual = false;
#pragma unroll 4
        for (int t = gl; t < s.k; t += 8) mutual |= row[t] == r;
        if (!__any_sync(group, mutual) && gl == 0) atomicAdd(&s.len[r], 1);
    }
}

// Hub rows, one CTA each, written to their places in the CSR: a bitmap of the
// columns of the union gives every entry its place (bits below it), HUB_COLS
// columns at a time. The reverse entries are set first, so a forward entry that
// finds its bit set is mutual; it adds its value to the one its partner has
// written. The range's values are then scaled.
__global__ void __launch_bounds__(HUB_THREADS)
sym_hub_kernel(SymRow s, const int32_t *__restrict__ hub_rows, const int32_t *__restrict__ n_list, int words,
               float inv2n, const int64_t *__restrict__ row_ptr, int32_t *col, float *val) {
    extern __shared__ uint32_t hub_smem[];
    uint32_t *bits = hub_smem, *below = hub_smem + words;  // below: set bits before each word, in this range
    __shared__ int wsum[HUB_THREADS / 32], wbase[HUB_THREADS / 32 + 1];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // words per warp, a multiple of 32
    const int per = (words + HUB_THREADS - 1) / HUB_THREADS * 32;
    for (int q = blockIdx.x; q < n_list[1]; q += gridDim.x) {
        const int64_t r = hub_rows[q], b0 = s.roff[r], m = s.roff[r + 1] - b0, row = r * s.k;
        int32_t *tc = col + row_ptr[r];
        float *tv = val + row_ptr[r];
        int64_t done = 0;  // entries of the ranges before
        for (int64_t c0 = 0; c0 < s.N; c0 += (int64_t)words * 32) {
            const int64_t c1 = min(s.N, c0 + (int64_t)words * 32);
            for (int t = tid; t < words; t += HUB_THREADS) bits[t] = below[t] = 0u;
            __syncthreads();
            for (int64_t t = tid; t < m; t += HUB_THREADS) {
                const int64_t c = s.rev[b0 + t].x;
                if (c >= c0 && c < c1) atomicOr(&bits[(c - c0) >> 5], 1u << ((c - c0) & 31));
            }
            __syncthreads();
            // at most one forward entry per thread (k <= SYM_MAX_K)
            int64_t fc = -1;
            bool mutual = false;
            if (tid < s.k) {
                const int j = s.idx[row + tid];
                if (j >= c0 && j < c1 && j != r) {
                    fc = j;
                    mutual = (bits[(fc - c0) >> 5] >> ((fc - c0) & 31)) & 1u;
                }
            }
            __syncthreads();
            if (fc >= 0) {
                // (the forward entries' own bits, in `below` until its sums are
                // made, show a column listed twice, mutual or not)
                const uint32_t bit = 1u << ((fc - c0) & 31);
                if (atomicOr(&below[(fc - c0) >> 5], bit) & bit) raise_status(s.status, DEV_MALFORMED);
                if (!mutual) atomicOr(&bits[(fc - c0) >> 5], bit);
            }
            __syncthreads();
            // a warp's stretch of words: each word's set bits before it in the
            // stretch, then the stretches' totals
            int run = 0;
            for (int t = warp * per + lane; t < (warp + 1) * per; t += 32) {
                const int n = t < words ? __popc(bits[t]) : 0;
                int incl = n;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int x = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += x;
                }
                if (t < words) below[t] = (uint32_t)(run + incl - n);
                run += __shfl_sync(0xffffffffu, incl, 31);
            }
            if (lane == 0) wsum[warp] = run;
            __syncthreads();
            if (warp == 0) {
                const int x = lane < HUB_THREADS / 32 ? wsum[lane] : 0;
                int incl = x;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                if (lane < HUB_THREADS / 32) wbase[lane] = incl - x;
                if (lane == 31) wbase[HUB_THREADS / 32] = incl;
            }
            __syncthreads();
            auto place = [&](int64_t c) {
                const int o = (int)(c - c0), u = o >> 5;
                return done + wbase[u / per] + below[u] + __popc(bits[u] & ((1u << (o & 31)) - 1u));
            };
            for (int64_t t = tid; t < m; t += HUB_THREADS) {
                const int2 e = s.rev[b0 + t];
                if (e.x >= c0 && e.x < c1) {
                    const int64_t at = place(e.x);
                    tc[at] = e.x;
                    tv[at] = __int_as_float(e.y);
                }
            }
            __syncthreads();
            if (fc >= 0) {
                const int64_t at = place(fc);
                const float p = s.P[row + tid];
                tc[at] = (int)fc;
                tv[at] = mutual ? p + tv[at] : p;
            }
            __syncthreads();
            const int64_t end = done + wbase[HUB_THREADS / 32];
            for (int64_t t = done + tid; t < end; t += HUB_THREADS) tv[t] *= inv2n;
            done = end;
        }
    }
}

__global__ void __launch_bounds__(256)
sym_copy_kernel(const int2 *__restrict__ rev, const int2 *__restrict__ tail, int64_t N, int k, float inv2n,
                const int64_t *__restrict__ roff, const int64_t *__restrict__ row_ptr, int32_t *__restrict__ col,
                float *__restrict__ val) {
    const int lane = threadIdx.x & 31;
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (r >= N) return;
    const int64_t b0 = roff[r], m = roff[r + 1] - b0, to = row_ptr[r], n = row_ptr[r + 1] - to;
    if (m + k > SYM_MID) return;  // a hub row, written in its place
    const int2 *first = rev + b0, *rest = tail + (r * k - m);
    for (int t0 = lane; t0 < n; t0 += 128) {  // four loads in flight per lane
        int2 e[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int t = t0 + 32 * u;
            if (t < n) e[u] = (t < m ? first : rest)[t];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int t = t0 + 32 * u;
            if (t < n) {
                col[to + t] = e[u].x;
                val[to + t] = __int_as_float(e[u].y) * inv2n;
            }
        }
    }
}

template <typename K>
atsne_status symmetrize_t(const int32_t *idx, const float *P, int64_t N, int k, int64_t *row_ptr, int32_t *col,
                          float *val, int64_t *nnz_dev, const SymWs &w, cudaStream_t stream) {
    int *status = device_status_word();
    cudaError_t e = cudaMemsetAsync(w.rcnt, 0, sizeof(int32_t) * N, stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(w.n_list, 0, 2 * sizeof(int32_t), stream);
    if (e != cudaSuccess) return cuda_error(e, "symmetrize memset");
    const float inv2n = (float)(0.5 / (double)N);
    const int row_blocks = ceil_div(N * 32, 256);
    ATSNE_TRY(launch_kernel("sym_count", sym_count_kernel, row_blocks, 256, 0, stream, idx, N, k, w.rank, w.rcnt,
                            status));
    ATSNE_TRY(scan_rowlen(w.rcnt, N, 0, w.roff, w.rtot, w.scan, stream));
    ATSNE_TRY(launch_kernel("sym_place", sym_place_kernel, row_blocks, 256, 0, stream, idx, P, N, k,
                            (const int32_t *)w.rank, (const int64_t *)w.roff, w.rev));
    const SymRow s{idx, P, N, k, w.roff, w.rev, w.tail, w.len, status};
    ATSNE_TRY(launch_kernel("sym_merge", sym_merge_kernel<K>, ceil_div(N, SYM_WARPS), SYM_WARPS * 32, 0, stream, s,
                            w.mid_rows, w.hub_rows, w.n_list));
    ATSNE_TRY(launch_kernel("sym_mid", sym_mid_kernel<K>, (int)hmin(4 * num_sms(), ceil_div(N, SYM_WARPS)),
                            SYM_WARPS * 32, 0, stream, s, (const int32_t *)w.mid_rows, (const int32_t *)w.hub_rows,
                            (const int32_t *)w.n_list));
    ATSNE_TRY(scan_rowlen(w.len, N, 0, row_ptr, nnz_dev, w.scan, stream));
    const int words = (int)((hmin(N, HUB_COLS) + 31) / 32);
    const size_t smem = (size_t)words * 8;
    // (the limit for any N: the attribute is the kernel's, and another thread's
    // smaller call may set it before this one's launch)
    e = cudaFuncSetAttribute(sym_hub_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(HUB_COLS / 4));
    if (e != cudaSuccess) return cuda_error(e, "sym_hub attribute");
    ATSNE_TRY(launch_kernel("sym_hub", sym_hub_kernel, (int)hmin(4 * num_sms(), N), HUB_THREADS, smem, stream, s,
                            (const int32_t *)w.hub_rows, (const int32_t *)w.n_list, words, inv2n,
                            (const int64_t *)row_ptr, col, val));
    return launch_kernel("sym_copy", sym_copy_kernel, row_blocks, 256, 0, stream, (const int2 *)w.rev,
                         (const int2 *)w.tail, N, k, inv2n, (const int64_t *)w.roff, (const int64_t *)row_ptr, col, val);
}

}  // namespace

size_t symmetrize_workspace(Carver &c, int64_t N, int k, SymWs *ws) {
    SymWs w;
    // the counters first: small calls spend most of the count on the atomics, and
    // these took 9 to 16 us (2,000 rows) by where the counters fell in memory; here,
    // with the allocations of a whole similarity matrix, 10, behind the lists 16
    w.rcnt = c.take<int32_t>((size_t)N);
    w.len = c.take<int32_t>((size_t)N);
    w.roff = c.take<int64_t>((size_t)N + 1);
    w.rtot = c.take<int64_t>(1);
    w.mid_rows = c.take<int32_t>((size_t)N);
    w.hub_rows = c.take<int32_t>((size_t)N);
    w.n_list = c.take<int32_t>(2);
    w.scan = c.take<int64_t>(scan_partials_count(N));
    w.rev = c.take<int2>((size_t)N * k);
    w.tail = c.take<int2>((size_t)N * k);
    w.rank = reinterpret_cast<int32_t *>(w.tail);  // read by the placement, before the merge writes
    if (ws) *ws = w;
    return c.bytes();
}

atsne_status symmetrize_launch(const int32_t *idx, const float *P, int64_t N, int k,
                               int64_t *row_ptr, int32_t *col, float *val, int64_t *nnz_dev,
                               const SymWs &w, cudaStream_t stream) {
    if (k > SYM_MAX_K) return set_error(ATSNE_EUNSUPPORTED, "symmetrize: k=%d above %d", k, SYM_MAX_K);
    if (N < SYM_KEY32) return symmetrize_t<uint32_t>(idx, P, N, k, row_ptr, col, val, nnz_dev, w, stream);
    return symmetrize_t<unsigned long long>(idx, P, N, k, row_ptr, col, val, nnz_dev, w, stream);
}

}  // namespace atsne
