// The exact kNN's contraction with a fixed threshold per query row (Eq. 8).
//
// A streaming top-k has to buffer about ksel (1 + ln(n / ksel)) keys per row,
// most of them before its bound has settled, and has to keep that bound: the
// counting, the updates and the survivors' walk, not the MMAs, then set the
// pace. Here the threshold is fixed before the stream. Three kernels:
//
//   knn_sample   gathers S pseudo-random corpus rows (one of each of S equal
//                ranges of positions, shuffled).
//   knn_filter   (SAMPLE) the contraction of every query row with those S
//                rows; each row keeps only the largest value of every block of
//                8, 32 or 64 sampled columns.
//   knn_tau      one warp per row: the rank-th largest block value becomes the
//                row's threshold (rank chosen on the host so that fewer than
//                ksel corpus keys lie below the threshold with a probability
//                of about 10^-3). A row's known bound (a hint or a radius)
//                takes its place where it is lower.
//   knn_filter   (main) the contraction with the whole corpus; every key below
//                the row's threshold is appended to the row's buffers.
//
// The threshold only decides how much is buffered: the merge requires ksel (or,
// certified, a proof that the k nearest are among the buffered), and a row that
// misses it goes to the adaptive kernel of knn_tc.cu.
//
// Measured against the adaptive kernel on all rows (one GB300, kernels alone):
// 1,000,000 x 128 Gamma clusters, one BF16 pass, ksel 360: 270 ms to 176 ms
// (+ 7 ms for the thresholds), 1.45 PFLOP/s of 2 N^2 D (1.64 with the K step of
// the norms), at the clock that the power limit leaves; 200,000 x 128, three
// passes, ksel 128: 22.7 to 14.0 ms; 50,021 x 50 log-normal, ksel 188: 4.6 to 0.96
// ms; 70,000 x 784 bytes: 6.4 to 4.5 ms; 7,013 queries against 107,013 x 50: 9.1
// to 0.3 ms. With fewer columns a larger share of them survives, and appending
// sets the pace: 100,000 x 128, one pass, tensor pipe active 49%, issue 67%.
//
// Layout. Two CTAs on neighbouring SMs form a pair (cta_group::2): M = 256
// query rows, 128 per CTA, against N = 256 corpus rows, of which each CTA
// stages half. A pair then reads each operand byte once from L2 and once from
// each shared memory, half of what two single CTAs read; the single-CTA form
// of this contraction asks shared memory for more bytes per cycle than it has.
// Per CTA: warp 0 issues the TMA loads, warp 1 (of the even CTA) the MMAs, and
// FC::NEPI warps the epilogue, FC::NEPI / 4 per TMEM lane quadrant, each taking
// 64 of a tile's 256 columns. A 32-column chunk without a survivor of any of the
// warp's rows (most of them in a large corpus, few at 50,000 rows) costs one
// tcgen05.ld, a tree of three-input maxima (18 instructions) and one vote; one
// with survivors a vote per group of eight columns and the groups' appends.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <float.h>
#include <math.h>
#include <string.h>

#include "common.cuh"
#include "internal.h"
#include "knn_keys.cuh"
#include "tc_ptx.cuh"

namespace atsne {
namespace {

using namespace tc;

constexpr int F_BM = 128;  // query rows per CTA
constexpr int F_BN = 256;  // corpus rows per tile
constexpr int F_BH = 128;  // of which each CTA of the pair stages half
constexpr uint64_t F_DRAIN_NS = 1000000000ull;

// PASSES: 1 (one BF16 pass, the column norms folded into the contraction) or 3
// (BF16 hi/lo, keys from the FP32 norms). With PASSES = 3 and every low half
// zero the stages are single-pass ones.
template <int PASSES>
struct FC {
    static constexpr int NEPI = 4 * F_PARTS;
    static constexpr int THREADS = 64 + 32 * NEPI;
    static constexpr int CW = F_BN / F_PARTS;  // columns of a tile per epilogue warp
    static constexpr int NCH = CW / 32;
    static_assert(NCH == 2, "both chunks of a part are loaded at once");
    static constexpr bool FOLD = PASSES == 1;
    static constexpr int OP_BYTES = F_BM * 128;              // one operand's k-block (64 BF16) per CTA
    static constexpr int EXT_BYTES = FOLD ? F_BM * 32 : 0;   // the norm pieces of a tile's half
    static constexpr int STAGE_BYTES = 2 * OP_BYTES * (PASSES == 3 ? 2 : 1) + EXT_BYTES;
    static constexpr int STAGES = PASSES == 3 ? 3 : 6;
    static constexpr int MAX_STAGES = 6;
};

template <int PASSES>
struct __align__(1024) FSmem {
    unsigned char stage[FC<PASSES>::STAGES][FC<PASSES>::STAGE_BYTES];
    unsigned char a_ext[FC<PASSES>::FOLD ? F_BM * 32 : 16];   // 1024-aligned
    float ny[PASSES == 3 ? FC<PASSES>::NEPI : 1][2][32];      // two chunks' norms per epilogue warp
    uint64_t full[FC<PASSES>::MAX_STAGES];
    uint64_t empty[FC<PASSES>::MAX_STAGES];
    uint64_t acc_full[2];
    uint64_t acc_empty[2];
    uint64_t drain;
    uint64_t ext_bar;
    // per stage, the last load this CTA issued: its number from 1, its bytes
    uint32_t load_no[FC<PASSES>::MAX_STAGES], load_bytes[FC<PASSES>::MAX_STAGES];
    // F_RADIUS: per row of three units in turn, its keys and the parts done with it
    int row_cnt[3][F_BM], row_done[3][F_BM];
    uint32_t tmem_base;
    int abort_flag;
    int zero;
};

struct FParams {
    CUtensorMap tm_a_hi, tm_a_lo, tm_b_hi, tm_b_lo, tm_a_ext, tm_b_ext;
    const float *nrm;        // PASSES = 3: corpus ||x||^2
    const unsigned *lo_max;  // as in the adaptive kernel
    const float *tau;        // [Q] key thresholds
    const int64_t *qcount;   // if given, the rows in use (device; at most Q)
    int64_t Q, N;
    int KB, last_steps;      // k-blocks; K = 16 steps of the last one
    int splits;              // split sp takes the column tiles sp, sp + splits, ...
    int cap;
    Cand *cand;              // [Q][splits * buffers per split][cap]
    int4 *meta;
    float *minima;           // SAMPLE: [Q][m] block maxima of the accumulators
    int m, blk;              // blk: columns per block (8, 32 or 64)
    int *status;
    uint64_t wait_ns;
};

// F_SAMPLE: the sampled rows' block maxima. F_RADIUS: few keys lie below the
// thresholds, and the four parts of a row append to one buffer, counted in shared
// memory: a row's room is its own wherever its points lie (a buffer per part
// for any distribution took four times the memory).
enum : int { F_MAIN = 0, F_SAMPLE = 1, F_RADIUS = 2 };
template <int PASSES, int MODE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(FC<PASSES>::THREADS, 1)
knn_filter_kernel(const __grid_constant__ FParams p) {
    using C = FC<PASSES>;
    constexpr bool SAMPLE = MODE == F_SAMPLE, RADIUS = MODE == F_RADIUS;
    constexpr int PARTS = RADIUS ? 1 : F_PARTS;  // buffers per row and split
    extern __shared__ __align__(16) unsigned char f_raw[];
    const uint32_t pad = (1024u - (smem_u32(f_raw) & 1023u)) & 1023u;
    FSmem<PASSES> &s = *reinterpret_cast<FSmem<PASSES> *>(f_raw + pad);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const bool lo_on = PASSES == 3 && !(p.lo_max && *p.lo_max == 0u);
    const int nst = PASSES == 3 && !lo_on ? C::MAX_STAGES : C::STAGES;
    const int sbytes = PASSES == 3 && !lo_on ? C::STAGE_BYTES / 2 : C::STAGE_BYTES;

    if (threadIdx.x == 0) {
        for (int i = 0; i < C::MAX_STAGES; ++i) {
            mbar_init(&s.full[i], 1);
            mbar_init(&s.empty[i], 1);
            s.load_no[i] = 0;
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&s.acc_full[i], 1);
            mbar_init(&s.acc_empty[i], 2 * C::NEPI);  // every epilogue warp of the pair
        }
        mbar_init(&s.drain, 1);
        mbar_init(&s.ext_bar, 1);
        s.abort_flag = 0;
        s.zero = 0;
        fence_mbar_init();
    }
    if (RADIUS)
        for (int i = threadIdx.x; i < 3 * F_BM; i += blockDim.x) (&s.row_cnt[0][0])[i] = (&s.row_done[0][0])[i] = 0;
    if (threadIdx.x == 32) {
        tma_prefetch_desc(&p.tm_a_hi);
        tma_prefetch_desc(&p.tm_b_hi);
    }
    __syncthreads();
    if (warp == 1) {
        tmem_alloc_pair(&s.tmem_base, 512);
        tmem_relinquish_pair();
    }
    fence_before_sync();
    __syncthreads();
    cluster_sync();  // both CTAs' barriers and TMEM exist before either signals the other
    fence_after_sync();
    const uint32_t tbase = s.tmem_base;
    const int64_t Q = p.qcount ? min(*p.qcount, p.Q) : p.Q;
    const int pairs = (int)((Q + 2 * F_BM - 1) / (2 * F_BM));
    const int64_t n_units = (int64_t)pairs * p.splits;
    const int64_t u0 = blockIdx.x >> 1, ustep = gridDim.x >> 1;
    const int64_t cstep = (int64_t)p.splits * F_BN;
    // an expired wait stops both CTAs' roles at their next wait
    auto give_up = [&]() {
        s.abort_flag = 1;
        st_cluster(map_to_rank(smem_u32(&s.abort_flag), rank ^ 1u), 1u);
        raise_status(p.status, DEV_TIMEOUT);
    };

    if (warp == 0) {
        if (lane == 0) {
            // ---------------- TMA producer (each CTA its own halves, counted on the even CTA's barriers) ----
            int stage = 0;
            uint32_t phase = 0, loads = 0;
            bool ok = true;
            const uint32_t full0 = map_to_rank(smem_u32(&s.full[0]), 0);
            const uint32_t stage0 = smem_u32(&s.stage[0][0]);
            if (C::FOLD) {
                if (rank == 0) mbar_arrive_expect_tx(&s.ext_bar, 2 * F_BM * 32);
                tma_load_2d_pair(smem_u32(s.a_ext), &p.tm_a_ext, 0, 0, map_to_rank(smem_u32(&s.ext_bar), 0));
            }
            for (int64_t u = u0; u < n_units && ok; u += ustep) {
                const int pt = (int)(u % pairs), sp = (int)(u / pairs);
                const int ar = (2 * pt + (int)rank) * F_BM;
                for (int64_t ct = (int64_t)sp * F_BN; ct < p.N && ok; ct += cstep) {
                    const int br = (int)ct + (int)rank * F_BH;
                    for (int kb = 0; kb < p.KB; ++kb) {
                        if (!mbar_wait(&s.empty[stage], phase ^ 1u, &s.abort_flag, p.wait_ns)) {
                            ok = false;
                            break;
                        }
                        const uint32_t st = stage0 + stage * sbytes;
                        const uint32_t fb = full0 + 8 * stage;
                        const bool ext = C::FOLD && kb + 1 == p.KB;
                        const uint32_t bytes = sbytes - (ext ? 0 : C::EXT_BYTES);
                        if (rank == 0) mbar_arrive_expect_tx(&s.full[stage], 2 * bytes);
                        s.load_no[stage] = ++loads;
                        s.load_bytes[stage] = bytes;
                        tma_load_2d_pair(st, &p.tm_a_hi, kb * 64, ar, fb);
                        tma_load_2d_pair(st + C::OP_BYTES, &p.tm_b_hi, kb * 64, br, fb);
                        if (ext) tma_load_2d_pair(st + 2 * C::OP_BYTES, &p.tm_b_ext, 0, br, fb);
                        if (PASSES == 3 && lo_on) {
                            tma_load_2d_pair(st + 2 * C::OP_BYTES, &p.tm_a_lo, kb * 64, ar, fb);
                            tma_load_2d_pair(st + 3 * C::OP_BYTES, &p.tm_b_lo, kb * 64, br, fb);
                        }
                        if (++stage == nst) {
                            stage = 0;
                            phase ^= 1u;
                        }
                    }
                }
            }
            if (!ok) give_up();
            if (C::FOLD && rank == 0) mbar_wait(&s.ext_bar, 0, &s.zero, F_DRAIN_NS);
        }
    } else if (warp == 1) {
        if (rank == 0) {
            // ---------------- MMA issuer (for the pair): the warp runs the loop, one lane issues ----------------
            const uint32_t idesc = idesc_bf16_f32(2 * F_BM, F_BN);
            int stage = 0, acc = 0;
            uint32_t phase = 0, acc_phase = 0;
            bool ok = true;
            const uint64_t a0 = sw128_kmajor_desc(smem_u32(&s.stage[0][0]));
            const uint64_t op = C::OP_BYTES >> 4;  // operands of a stage, in descriptor units
            const uint64_t ext_a = sw32_kmajor_desc(smem_u32(s.a_ext));
            const uint64_t ext_b0 = sw32_kmajor_desc(smem_u32(&s.stage[0][0]) + 2 * C::OP_BYTES);
            if (C::FOLD) ok = __all_sync(0xffffffffu, mbar_wait(&s.ext_bar, 0, &s.abort_flag, p.wait_ns));
            for (int64_t u = u0; u < n_units && ok; u += ustep) {
                const int sp = (int)(u / pairs);
                for (int64_t ct = (int64_t)sp * F_BN; ct < p.N && ok; ct += cstep) {
                    ok = __all_sync(0xffffffffu,
                                    mbar_wait(&s.acc_empty[acc], acc_phase ^ 1u, &s.abort_flag, p.wait_ns));
                    if (!ok) break;
                    fence_after_sync();
                    const uint32_t d = tbase + (uint32_t)(acc * F_BN);
                    for (int kb = 0; kb < p.KB; ++kb) {
                        ok = __all_sync(0xffffffffu, mbar_wait(&s.full[stage], phase, &s.abort_flag, p.wait_ns));
                        if (!ok) break;
                        fence_after_sync();
                        const uint64_t so = (uint64_t)((uint32_t)(stage * sbytes) >> 4);
                        const uint64_t a_hi = a0 + so, b_hi = a_hi + op, a_lo = b_hi + op, b_lo = a_lo + op;
                        const bool last = kb + 1 == p.KB;
                        // the last k-block's steps past the row's end multiply zeros: left out
                        const int steps = last ? p.last_steps : 4;
                        if (elect_one()) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) {  // 32 bytes of each row per MMA
                                if (k < steps) {
                                    mma_bf16_pair(d, a_hi + 2 * k, b_hi + 2 * k, idesc, (kb | k) != 0);
                                    if (PASSES == 3 && lo_on) {
                                        mma_bf16_pair(d, a_hi + 2 * k, b_lo + 2 * k, idesc, 1u);
                                        mma_bf16_pair(d, a_lo + 2 * k, b_hi + 2 * k, idesc, 1u);
                                    }
                                }
                            }
                            if (C::FOLD && last)  // the norms: -1/2 (h1 + h2 + h3) per column
                                mma_bf16_pair(d, ext_a, ext_b0 + so, idesc, 1u);
                            mma_commit_pair(&s.empty[stage]);
                            if (last) mma_commit_pair(&s.acc_full[acc]);
                        }
                        __syncwarp();
                        if (++stage == nst) {
                            stage = 0;
                            phase ^= 1u;
                        }
                    }
                    if (++acc == 2) {
                        acc = 0;
                        acc_phase ^= 1u;
                    }
                }
            }
            if (elect_one()) {
                if (!ok) give_up();
                mma_commit_pair(&s.drain);
            }
            __syncwarp();
        }
    } else {
        // ---------------- epilogue ----------------
        const int e = warp - 2;
        const int quarter = warp & 3;  // the TMEM lane quadrant this warp may read
        const int part = e >> 2;
        const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
        const uint32_t acc_empty0 = map_to_rank(smem_u32(&s.acc_empty[0]), 0);
        const int subs = p.splits * PARTS;
        int slot = 0;  // RADIUS: of the unit's counters
        int acc = 0;
        uint32_t acc_phase = 0;
        bool ok = true;
        for (int64_t u = u0; u < n_units && ok; u += ustep) {
            const int pt = (int)(u % pairs), sp = (int)(u / pairs);
            const int64_t c0 = (int64_t)sp * F_BN;
            const int64_t row = ((int64_t)2 * pt + rank) * F_BM + quarter * 32 + lane;
            const bool live = row < Q;
            // survivors are the values v above thr: v = x.y - ||y||^2/2 with
            // the norms folded in (key = -2 v), else v = -key
            float thr = INFINITY;
            Cand *buf = nullptr;
            float *mrow = nullptr;
            float tau = -INFINITY;
            int cnt = 0;
            int *row_cnt = RADIUS ? &s.row_cnt[slot][quarter * 32 + lane] : nullptr;
            if (live) {
                if (SAMPLE) {
                    mrow = p.minima + row * p.m;
                } else {
                    // finite, so that a padded column (v = -inf) never passes
                    tau = p.tau[row];
                    const float tf = fminf(tau, FLT_MAX);
                    thr = C::FOLD ? -0.5f * tf : -tf;
                    buf = p.cand + ((size_t)row * subs + (size_t)sp * PARTS + (RADIUS ? 0 : part)) * p.cap;
                }
            }
            float nyn[C::NCH];
            if (!C::FOLD) {
#pragma unroll
                for (int q = 0; q < C::NCH; ++q) {
                    const int64_t cc = c0 + part * C::CW + q * 32 + lane;
                    nyn[q] = cc < p.N ? -p.nrm[cc] : -INFINITY;
                }
            }
            for (int64_t ct = c0; ct < p.N; ct += cstep) {
                float nyc[C::NCH];
                if (!C::FOLD) {
#pragma unroll
                    for (int q = 0; q < C::NCH; ++q) {
                        nyc[q] = nyn[q];
                        const int64_t cc = ct + cstep + part * C::CW + q * 32 + lane;
                        nyn[q] = cc < p.N ? -p.nrm[cc] : -INFINITY;
                    }
                }
                ok = mbar_wait(&s.acc_full[acc], acc_phase, &s.abort_flag, p.wait_ns);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) {
                    if (lane == 0) give_up();
                    break;
                }
                fence_after_sync();
                const uint32_t taddr = tbase + lane_base + (uint32_t)(acc * F_BN + part * C::CW);
                const int colb0 = (int)ct + part * C::CW;
                // both chunks at once, and the accumulator is free for the next
                // tile's MMAs as soon as they have arrived
                uint32_t ra[32], rb[32];
                tmem_ld32(taddr, ra);
                tmem_ld32(taddr + 32u, rb);
                if (!C::FOLD) {
                    s.ny[e][0][lane] = nyc[0];
                    s.ny[e][1][lane] = nyc[1];
                }
                tmem_ld_wait(ra);
                tmem_ld_wait(rb);
                fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(acc_empty0 + 8 * acc);
                float pm = -INFINITY;  // SAMPLE: the largest value of this part
#pragma unroll
                for (int c = 0; c < C::NCH; ++c) {
                    uint32_t(&r)[32] = (c & 1) ? rb : ra;
                    const float *nyw = s.ny[PASSES == 3 ? e : 0][c & 1];
                    float v[32];
                    if (C::FOLD) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
                    } else {
                        const float4 *n4p = reinterpret_cast<const float4 *>(nyw);
                        const float2 two = make_float2(2.f, 2.f);
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const float4 n4 = n4p[q];
                            const float2 a = __ffma2_rn(two, make_float2(__uint_as_float(r[4 * q]), __uint_as_float(r[4 * q + 1])),
                                                        make_float2(n4.x, n4.y));
                            const float2 b = __ffma2_rn(two, make_float2(__uint_as_float(r[4 * q + 2]), __uint_as_float(r[4 * q + 3])),
                                                        make_float2(n4.z, n4.w));
                            v[4 * q] = a.x;
                            v[4 * q + 1] = a.y;
                            v[4 * q + 2] = b.x;
                            v[4 * q + 3] = b.y;
                        }
                    }
                    float g[4];  // the largest of each 8
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        g[q] = max3(max3(v[8 * q], v[8 * q + 1], v[8 * q + 2]),
                                    max3(v[8 * q + 3], v[8 * q + 4], v[8 * q + 5]), fmaxf(v[8 * q + 6], v[8 * q + 7]));
                    const float gm = fmaxf(max3(g[0], g[1], g[2]), g[3]);
                    if (SAMPLE) {
                        const int64_t at = colb0 + c * 32;
                        if (p.blk == 8) {
                            if (live) *reinterpret_cast<float4 *>(mrow + (at >> 3)) = make_float4(g[0], g[1], g[2], g[3]);
                        } else if (p.blk == 32) {
                            if (live) mrow[at >> 5] = gm;
                        } else {
                            pm = fmaxf(pm, gm);
                            if (c + 1 == C::NCH && live) mrow[colb0 / C::CW] = pm;
                        }
                    } else if (__any_sync(0xffffffffu, gm > thr)) {
                        const int col = colb0 + c * 32;
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            if (!__any_sync(0xffffffffu, g[q] > thr)) continue;
                            // a buffer without room for eight more is closed (the row is
                            // given up). Closed for want of room for a chunk's 32,
                            // the shorter buffers gave up rows that fitted them (60,000 x
                            // 32, k = 30, four clusters in blocks of 64 rows: 2.55
                            // ms, 1.63 now)
                            if (!RADIUS && cnt > p.cap - 8) thr = INFINITY;
                            if (RADIUS) {
                                // a lane's keys of the group take their places at once
                                int n = 0;
#pragma unroll
                                for (int j = 0; j < 8; ++j) n += v[8 * q + j] > thr;
                                if (n > 0) {
                                    cnt = atomicAdd(row_cnt, n);
                                    if (cnt > p.cap - n) thr = INFINITY;  // full
                                }
                            }
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                const float x = v[8 * q + j];
                                if (x > thr) buf[cnt++] = Cand{C::FOLD ? -2.f * x : -x, col + 8 * q + j};
                            }
                        }
                    }
                }
                if (++acc == 2) {
                    acc = 0;
                    acc_phase ^= 1u;
                }
            }
            if (!ok) break;
            if (RADIUS) {
                // the last part to finish the row's unit writes its count and
                // clears it. A unit's counters are taken again three units
                // later: its tiles start when every warp has arrived for the
                // tile two before, which lies past the unit
                __threadfence_block();
                if (live && atomicAdd(&s.row_done[slot][quarter * 32 + lane], 1) == F_PARTS - 1) {
                    const int n = atomicExch(row_cnt, 0);
                    s.row_done[slot][quarter * 32 + lane] = 0;
                    p.meta[(size_t)row * subs + sp] = make_int4(min(n, p.cap), __float_as_int(tau), n > p.cap, META_FIRST);
                }
                slot = slot == 2 ? 0 : slot + 1;
            } else if (!SAMPLE && live) {
                p.meta[(size_t)row * subs + (size_t)sp * F_PARTS + part] =
                    make_int4(cnt, __float_as_int(tau), thr == INFINITY, META_FIRST);
            }
        }
    }
    fence_before_sync();
    __syncthreads();
    // all MMAs of the pair complete before TMEM is released, and the commit has
    // signalled this CTA before it may leave
    if (threadIdx.x == 32) mbar_wait(&s.drain, 0, &s.zero, F_DRAIN_NS);
    __syncwarp();
    cluster_sync();  // no CTA leaves while its peer may still signal it or use its shared memory
    if (s.abort_flag) {
        // After an expired wait the two producers may have stopped at
        // different loads. Once neither issues any more, the even CTA makes up
        // the counts of the loads only one of them issued and waits for every
        // copy in flight to land.
        if (rank == 0 && threadIdx.x == 0)
            for (int i = 0; i < nst; ++i) {
                const uint32_t mine = s.load_no[i];
                const uint32_t peer = ld_cluster(map_to_rank(smem_u32(&s.load_no[i]), 1));
                const uint32_t last = max(mine, peer);
                if (mine > peer) mbar_complete_tx(&s.full[i], s.load_bytes[i]);
                if (peer > mine)
                    mbar_arrive_expect_tx(&s.full[i], ld_cluster(map_to_rank(smem_u32(&s.load_bytes[i]), 1)));
                if (last) mbar_wait(&s.full[i], ((last - 1) / nst) & 1u, &s.zero, F_DRAIN_NS);
            }
        __syncthreads();
        __syncwarp();
        cluster_sync();
    }
    fence_after_sync();
    if (warp == 1) tmem_dealloc_pair(tbase, 512);
}

// Sampled corpus row i: one position of range (i * F_MIX) mod S of S equal
// ranges of [0, N) (S a power of two: a permutation, so that neighbouring
// sampled columns come from distant positions), jittered by a hash (the
// finaliser of MurmurHash3's 32-bit form, A. Appleby, public domain) so that no
// periodic layout of the corpus is met in step. F_MIX is Knuth's golden ratio
// multiplier.
constexpr unsigned F_MIX = 2654435761u;
__device__ __forceinline__ int64_t sample_position(unsigned i, unsigned S, int64_t N) {
    const unsigned r = (i * F_MIX) & (S - 1);
    unsigned h = r * 0x9e3779b9u + 0x7f4a7c15u;
    h ^= h >> 16;
    h *= 0x85ebca6bu;
    h ^= h >> 13;
    h *= 0xc2b2ae35u;
    h ^= h >> 16;
    const int64_t a = (int64_t)r * N / S, b = ((int64_t)r + 1) * N / S;
    return a + (int64_t)(((uint64_t)h * (uint64_t)(b - a)) >> 32);
}

// The sampled rows' BF16 copies and norm pieces, one warp per row. Bound by its
// few MB of copies.
__global__ void __launch_bounds__(256)
knn_sample_kernel(const uint16_t *__restrict__ hi, const float *__restrict__ nrm, int64_t N, int Dp, int S,
                  uint16_t *__restrict__ shi, __nv_bfloat16 *__restrict__ sext, __nv_bfloat16 *__restrict__ aext) {
    const int lane = threadIdx.x & 31;
    const int i = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (blockIdx.x == 0) fold_query_slice(aext);
    if (i >= S) return;
    const int64_t src = sample_position((unsigned)i, (unsigned)S, N);
    const uint4 *a = reinterpret_cast<const uint4 *>(hi + src * Dp);
    uint4 *b = reinterpret_cast<uint4 *>(shi + (int64_t)i * Dp);
    for (int t = lane; t < (Dp >> 3); t += 32) b[t] = a[t];
    if (lane < 16) sext[(int64_t)i * 16 + lane] = norm_piece(nrm[src], lane);
}

// The rank-th largest of a row's m block values (m <= 1024), by bisection on
// the values' order-preserving bits, counting the values held in registers.
// Whole warp.
__device__ __forceinline__ float rank_largest(const float *mr, int m, int rank, int lane) {
    const int per = (m + 31) / 32;
    uint32_t u[32];
#pragma unroll
    for (int t = 0; t < 32; ++t) {
        u[t] = 0u;
        if (t < per && t * 32 + lane < m) u[t] = float_key(mr[t * 32 + lane]);
    }
    // the largest threshold with at least `rank` values at or above it, or
    // any that has exactly `rank` (a dozen counts instead of 32)
    uint32_t lo = 0xffffffffu, hi = 0u;
#pragma unroll
    for (int t = 0; t < 32; ++t)
        if (t < per) {
            if (t * 32 + lane < m) lo = min(lo, u[t]);
            hi = max(hi, u[t]);
        }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    while (lo < hi) {
        const uint32_t mid = hi - ((hi - lo) >> 1);
        int c = 0;
#pragma unroll
        for (int t = 0; t < 32; ++t)
            if (t < per) c += u[t] >= mid;
        c = (int)__reduce_add_sync(0xffffffffu, (unsigned)c);
        if (c >= rank) {
            lo = mid;
            if (c == rank) break;
        } else {
            hi = mid - 1u;
        }
    }
    return key_of_bits(lo);
}

struct TauParams {
    const float *minima;  // [Q][m], or nullptr (no sample)
    int m, rank;
    const float *bound;   // [Q] radius or hint (squared distances), or nullptr
    const int32_t *qlist;
    const float *nrm, *qnrm;     // corpus / separate queries
    const float4 *st, *qst;
    const unsigned *gmax;
    float acc_coef, sq_coef;
    const int64_t *qcount;
    int64_t Q, N;
    float *tau;
};

// Threshold of each query row, one warp per row: the rank-th largest block
// value by bisection on the values' order-preserving bits, counting the m
// values held in registers (m <= 1024). A few hundred instructions per row.
__global__ void __launch_bounds__(128) knn_tau_kernel(TauParams p) {
    const int lane = threadIdx.x & 31;
    const int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t Q = p.qcount ? min(*p.qcount, p.Q) : p.Q;
    if (row >= Q) return;
    float tau = INFINITY;
    if (p.minima) {
        const float v = rank_largest(p.minima + row * p.m, p.m, p.rank, lane);
        if (isfinite(v)) tau = -2.f * v;
    }
    if (p.bound) {
        // the radius, or the hint (an upper bound of the k-th squared
        // distance), as a key threshold widened by twice the key error bound,
        // so that no point inside is filtered out: such a point's norm is at
        // most ||x|| + sqrt(bound)
        const bool cross = p.qnrm != nullptr;
        const int q = cross ? (int)row : (p.qlist ? p.qlist[row] : (int)row);
        const float rad = p.bound[row];
        if (q >= 0 && (cross || q < p.N) && isfinite(rad)) {
            const float4 st = cross ? p.qst[row] : p.st[q];
            const float nx = cross ? p.qnrm[row] : p.nrm[q];
            const float widen = 2.f * key_error_bound_capped(st, p.gmax, p.acc_coef, p.sq_coef,
                                                             st.x + sqrtf(fmaxf(rad, 0.f)) * (1.f + 1e-6f) + 1e-30f) +
                                1e-6f * (fabsf(rad) + nx);
            tau = fminf(tau, rad - nx + widen);
        }
    }
    if (lane == 0) p.tau[row] = tau;
}

// Starting thresholds of the rows given up for too few keys (marked +inf), one
// warp per row, in the modes without a certificate: the adaptive kernel tightens
// a threshold only as it meets nearer keys, and from +inf its first tiles
// overflow the buffers of a row whose columns are split over many units. Merge
// and adaptive launch of a list of rows, started from +inf and from here: 7,000
// rows of 100,000 x 50 (lognormal) 4.87 and 0.28 ms, 500 rows of 70,000 x 784
// (bytes) 1.47 and 0.38 ms, 20,000 rows of 200,000 x 128 865 and 663 us. A row
// that failed the certificate stays at +inf: it needs keys past the k-th by
// twice their error bound, and starting there cost more where nearly all keys
// lie that close (3,000 equal rows, FP32: 0.12 and 1.2 ms).
__global__ void __launch_bounds__(128)
knn_retry_tau_kernel(const float *__restrict__ minima, int m, int rank, const int32_t *__restrict__ rows,
                     const int32_t *__restrict__ count, float *__restrict__ tau) {
    const int lane = threadIdx.x & 31, n = *count;
    for (int i = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); i < n; i += (int)(gridDim.x * blockDim.x) >> 5) {
        const int64_t r = rows[i];
        if (!isinf(tau[r])) continue;
        const float v = rank_largest(minima + r * m, m, rank, lane);
        if (lane == 0 && isfinite(v)) tau[r] = -2.f * v;
    }
}

template <int PASSES>
size_t f_smem_bytes() {
    return sizeof(FSmem<PASSES>) + 1024;
}
static_assert(sizeof(FSmem<1>) + 1024 <= 232448, "filter shared memory above 227 KB");
static_assert(sizeof(FSmem<3>) + 1024 <= 232448, "filter shared memory above 227 KB");

template <int PASSES, int MODE>
atsne_status f_launch(const FParams &p, int64_t units, cudaStream_t stream) {
    const size_t smem = f_smem_bytes<PASSES>();
    cudaError_t e = cudaFuncSetAttribute(knn_filter_kernel<PASSES, MODE>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_error(e, "knn_filter attribute");
    const int grid = 2 * (int)hmin(units, num_sms() / 2);
    return launch_kernel(MODE == F_SAMPLE ? "knn_bound" : "knn_filter", knn_filter_kernel<PASSES, MODE>, grid,
                         FC<PASSES>::THREADS, smem, stream, p);
}

}  // namespace

// The critical path, in column tiles, of Qp row pairs against `tiles` column
// tiles in s splits over the SM pairs: waves of units, each its tiles and about
// two tiles of start-up.
double filter_path(int64_t Qp, int64_t tiles, int s) {
    const int64_t C = num_sms() / 2 > 0 ? num_sms() / 2 : 1;
    return (double)((Qp * s + C - 1) / C) * (double)((tiles + s - 1) / s + 2);
}

// A split costs the fixed threshold nothing but a few more (shorter) buffers per
// row, so it is chosen for the last wave: the fewest splits whose critical path
// is within 2% of the shortest found. The splits take the tiles in turn, so that
// neighbours that follow one another in the corpus (sorted by class) spread over
// them.
int filter_splits(int64_t Qp, int64_t tiles, int max_splits) {
    double best = filter_path(Qp, tiles, 1);
    for (int s = 2; s <= max_splits && s <= tiles; ++s) best = fmin(best, filter_path(Qp, tiles, s));
    for (int s = 1; s <= max_splits && s <= tiles; ++s)
        if (filter_path(Qp, tiles, s) <= 1.02 * best) return s;
    return 1;
}

atsne_status knn_filter_launch(const TcPlan &pl, const TcWs &w, const FilterArgs &a, cudaStream_t stream) {
    FParams p;
    memset(&p, 0, sizeof(p));
    ATSNE_TRY(tc_map_bf16(&p.tm_a_hi, a.a_hi, a.a_rows, pl.Dp, F_BM));
    p.tm_a_lo = p.tm_b_lo = p.tm_a_hi;
    p.qcount = a.qcount;
    p.Q = a.Q;
    p.KB = pl.Dp / 64;
    p.last_steps = (a.D - 64 * (p.KB - 1) + 15) / 16;
    p.status = device_status_word();
    p.wait_ns = pipeline_wait_ns();
    const int64_t pairs = (a.Q + 2 * F_BM - 1) / (2 * F_BM);
    TauParams t;
    memset(&t, 0, sizeof(t));
    if (pl.S > 0) {
        ATSNE_TRY(launch_kernel("knn_sample", knn_sample_kernel, ceil_div((int64_t)pl.S * 32, 256), 256, 0, stream,
                                (const uint16_t *)w.hi, (const float *)w.nrm, a.N, pl.Dp, pl.S, w.shi,
                                reinterpret_cast<__nv_bfloat16 *>(w.sext), reinterpret_cast<__nv_bfloat16 *>(w.aext)));
        ATSNE_TRY(tc_map_bf16(&p.tm_b_hi, w.shi, pl.S, pl.Dp, F_BH));
        ATSNE_TRY(tc_map_ext(&p.tm_a_ext, w.aext, F_BM, F_BM));
        ATSNE_TRY(tc_map_ext(&p.tm_b_ext, w.sext, pl.S, F_BH));
        p.N = pl.S;
        p.splits = filter_splits(pairs, pl.S / F_BN, 16);
        p.minima = w.minima;
        p.m = pl.S / pl.blk;
        p.blk = pl.blk;
        ATSNE_TRY((f_launch<1, F_SAMPLE>(p, pairs * p.splits, stream)));
        t.minima = w.minima;
        t.m = p.m;
        t.rank = pl.rank;
    }
    t.bound = a.radius ? a.radius : a.hint;
    t.qlist = a.qlist;
    t.nrm = w.nrm;
    t.qnrm = a.cross ? w.qnrm : nullptr;
    t.st = reinterpret_cast<const float4 *>(w.stats);
    t.qst = reinterpret_cast<const float4 *>(w.qstats);
    t.gmax = w.gmax;
    t.acc_coef = a.acc_coef;
    t.sq_coef = a.sq_coef;
    t.qcount = a.qcount;
    t.Q = a.Q;
    t.N = a.N;
    t.tau = w.tau;
    ATSNE_TRY(launch_kernel("knn_tau", knn_tau_kernel, ceil_div(a.Q * 32, 128), 128, 0, stream, t));

    ATSNE_TRY(tc_map_bf16(&p.tm_b_hi, w.hi, a.N, pl.Dp, F_BH));
    p.tm_b_lo = p.tm_b_hi;
    p.N = a.N;
    p.nrm = w.nrm;
    p.tau = w.tau;
    p.splits = pl.fsplits;
    p.cap = pl.fcap;
    p.cand = reinterpret_cast<Cand *>(w.cand);
    p.meta = reinterpret_cast<int4 *>(w.meta);
    if (pl.passes == 3) {
        ATSNE_TRY(tc_map_bf16(&p.tm_a_lo, a.a_lo, a.a_rows, pl.Dp, F_BM));
        ATSNE_TRY(tc_map_bf16(&p.tm_b_lo, w.lo, a.N, pl.Dp, F_BH));
        p.tm_a_ext = p.tm_b_ext = p.tm_a_hi;
        p.lo_max = a.lo_max;
        return a.radius ? f_launch<3, F_RADIUS>(p, pairs * p.splits, stream) : f_launch<3, F_MAIN>(p, pairs * p.splits, stream);
    }
    // the norm pieces' rows are padded to a whole tile with +inf (norm_pieces)
    ATSNE_TRY(tc_map_ext(&p.tm_a_ext, w.aext, F_BM, F_BM));
    ATSNE_TRY(tc_map_ext(&p.tm_b_ext, w.bext, (a.N + F_BN - 1) / F_BN * F_BN, F_BH));
    return a.radius ? f_launch<1, F_RADIUS>(p, pairs * p.splits, stream) : f_launch<1, F_MAIN>(p, pairs * p.splits, stream);
}

atsne_status knn_retry_tau_launch(const TcPlan &pl, const TcWs &w, cudaStream_t stream) {
    return launch_kernel("knn_retry_tau", knn_retry_tau_kernel, 2 * num_sms(), 128, 0, stream, (const float *)w.minima,
                         pl.S / pl.blk, pl.rank2, (const int32_t *)w.retry_rows, (const int32_t *)(w.flag_count + 1),
                         w.tau);
}

}  // namespace atsne
