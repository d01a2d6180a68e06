// Transfers of the Lagrange levels on the tensor cores (Sec. 2.2.2: v~_a += T_t u~_b for every
// admissible pair (a, b) of translation t), with f16 operands split in two.
//
// Split.  Every operand value x is written as hi + lo with hi = f16(x s) and lo = f16(x s - hi),
// s a power of two, and a product is hi hi + hi lo + lo hi in FP32 accumulators.  Both
// roundings are to nearest, so hi + lo carries 22 bits plus sign and the dropped lo lo term
// is below 2^-24 of the product; the TF32 split used before truncated (hi: 11 bits, lo: 11 bits of
// the rest), which is four to eight times coarser, and f16 runs at twice the TF32 rate.  The
// scale keeps the largest value of a row between 2^13 and 2^14, so a value keeps its 22 bits
// down to 2^-15 of its row's largest, and below that an absolute error of 2^-39 of it.
//
// Rows are split once per box (k_rows_split), the operators once per plan (k_op_image); both
// are stored in the order in which the kernels copy them, so the transfer itself converts
// nothing: its copying threads only move 16-byte segments.
#include <cmath>

#include "ffm_internal.cuh"
#include "tc_common.cuh"

namespace ffm {

constexpr int HK = 32;            // K values (source nodes) per chunk
constexpr int HROW = 2 * HK;      // halves per row and chunk: hi part, then lo part (128 bytes)
constexpr int HM = 128;           // rows (pairs times right-hand sides) per tile
constexpr int H_LBO = 128, H_SBO = (HK / 8) * 128;

// a power of two s with max s in [2^13, 2^14), and its inverse (both finite and normal)
__device__ __forceinline__ void row_scale(float mx, float &s, float &inv) {
    int e = 0;
    if (mx > 0.f && mx <= 3.4028235e38f) {
        e = 13 - ilogbf(mx);
        e = max(-120, min(120, e));
    }
    s = __int_as_float((127 + e) << 23);
    inv = __int_as_float((127 - e) << 23);
}

__device__ __forceinline__ void half_split(float x, __half &hi, __half &lo) {
    hi = __float2half_rn(x);
    lo = __float2half_rn(x - __half2float(hi));
}

// Rows of n floats as f16 hi / lo images, one warp per row: chunk kc of row i holds the hi
// parts of values 32 kc .. + 31, then their lo parts (zero past n); inv[i] = 1 / scale.
__global__ void __launch_bounds__(256) k_rows_split(const float *__restrict__ u, int64_t nrow, int n, int nk,
                                                    __half *__restrict__ img, float *__restrict__ inv) {
    const int64_t i = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (i >= nrow) return;
    const float *row = u + i * n;
    float mx = 0.f;
    for (int k = lane; k < n; k += 32) mx = fmaxf(mx, fabsf(row[k]));
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    float s, si;
    row_scale(mx, s, si);
    if (lane == 0) inv[i] = si;
    __half *out = img + i * (int64_t)nk * HROW;
    for (int k = 2 * lane; k < nk * HK; k += 64) {
        __half h0, l0, h1, l1;
        half_split(k < n ? row[k] * s : 0.f, h0, l0);
        half_split(k + 1 < n ? row[k + 1] * s : 0.f, h1, l1);
        __half *o = out + (k / HK) * HROW + (k % HK);
        *reinterpret_cast<__half2 *>(o) = __halves2half2(h0, h1);
        *reinterpret_cast<__half2 *>(o + HK) = __halves2half2(l0, l1);
    }
}

// Operators as the images the transfer copies: per translation t and row block blk, nk chunks of
// the hi parts of npad rows x 32 values in K-major core matrices, then the lo parts.  Block blk
// holds rows (blk % bpc) nb .. of component blk / bpc.  A complex operator is the real matrix
// of its action on interleaved (re, im) rows: rows 2i, 2i + 1 = (Re, -Im), (Im, Re) of T(i, j) at
// columns 2j, 2j + 1.
template <bool CPLX>
__global__ void __launch_bounds__(256) k_op_image(const float *__restrict__ T, int n_trans, int r, int rk, int nb,
                                                  int bpc, int npad, int nk, float scale, __half *__restrict__ img) {
    const int t = blockIdx.x, blk = blockIdx.y, nblk = gridDim.y;
    const int comp = blk / bpc, row0 = (blk % bpc) * nb;
    const int rows = CPLX ? 2 * r : r, cols = CPLX ? 2 * rk : rk;
    const float *Tt = T + ((size_t)comp * n_trans + t) * r * rk * (CPLX ? 2 : 1);
    __half *out = img + ((size_t)t * nblk + blk) * nk * npad * HROW;
    const int per = npad * HK;  // values per chunk
    for (int e = threadIdx.x; e < nk * per; e += blockDim.x) {
        const int kc = e / per, o = e - kc * per;
        const int k = kc * HK + ((o >> 6) & 3) * 8 + (o & 7), i = ((o >> 8) << 3) + ((o >> 3) & 7), ri = row0 + i;
        float v = 0.f;
        if (i < nb && ri < rows && k < cols) {
            if constexpr (CPLX) {
                const float *z = Tt + 2 * ((size_t)(ri >> 1) * rk + (k >> 1));
                const int ci = ri & 1, cj = k & 1;
                v = ci == cj ? z[0] : (cj ? -z[1] : z[1]);
            } else {
                v = Tt[(size_t)ri * rk + k];
            }
        }
        __half h, l;
        half_split(v * scale, h, l);
        __half *c = out + (size_t)kc * npad * HROW;
        c[o] = h;
        c[per + o] = l;
    }
}

constexpr int PAIR_MAXBLK = 16;
struct PairArgs {
    const uint32_t *bt_off, *bt_src, *bt_tgt;  // pairs grouped by translation
    int n_trans, nrhs, nblk;
    const __half *u;    // row images of (source box, right-hand side)
    const float *uinv;
    const __half *T;    // operator images
    float tinv;
    int nk, npad, tcols;
    int stack;          // hi and lo rows of T in one MMA operand of 2 npad rows
    int ostride;        // floats between rows of v~
    int nout[PAIR_MAXBLK];
    int64_t ooff[PAIR_MAXBLK];  // first float of the block's columns in v~
    float *vt;
    int *err;
    int tries;
};

// ---- transfer by translation
//
// What bounds it: the traffic of gathered rows, operators and scattered sums between L2 and the
// SMs, so a block streams all three at once and never stops at a tile's end.  The rows of a
// translation's pairs (times right-hand sides) are cut into tiles of 128; a unit is a tile times
// a row block of the operator (at most 256 rows), and the blocks of one persistent grid take
// units in turn, so that neighbouring blocks read the same operator.  Per unit and chunk of 32 K
// values:
//   warps 0-3   copy the tile's rows (hi and lo, 16 KB) with cp.async, rows past the tile's pairs
//               zero-filled; the row numbers of the next unit are fetched while this one is copied
//   thread 0    also starts the bulk copy of the operator's chunk (128 npad bytes)
//   warp 8      issues the MMAs into one of two TMEM accumulators
//   warps 4-7   read the other accumulator, undo the scales and add it into v~: 32 columns at a
//               time through shared memory, so that eight lanes add 128 consecutive bytes
// The MMAs of a K step are hi [hi; lo] (one operand of 2 npad rows, accumulated apart) and lo hi
// up to 128 operator rows, else three of npad rows into one accumulator.
// NSTG chunks are in flight: 8 at npad = 64 (24 KB each), 4 at 224 (45 KB).
//
// Measured on GB300, transfers of one apply, against the kernel before it (a block per 256-pair
// tile, which split its FP32 rows into TF32 for every pair, no overlap of tiles): gradient sphere 300k
// (r = 216, three operators) 6.54 -> 3.12 ms, double layer 200k (K = 648) 2.16 -> 0.97, Laplace volume
// 250k at 1e-4 (r = 216) 1.47 -> 0.79, 100k x 8 right-hand sides (r = 64) 1.68 -> 0.72, clustered
// 10M (r = 64) 21.8 -> 14.0.  Complex operators (Helmholtz volume 120k at 1e-4, 432 real rows), on
// CUDA cores before: 24.4 -> 2.4 ms.
constexpr int PAIR_T = 288;
constexpr int PAIR_ST = 36;  // floats per row of the epilogue's staging (conflict-free float4)

static size_t pair_stage(int npad) { return (size_t)HM * HROW * 2 + (size_t)npad * HROW * 2; }
static size_t pair_smem(int nstg, int npad, int n_trans) {
    return nstg * pair_stage(npad) + 4 * 32 * PAIR_ST * sizeof(float) + sizeof(uint32_t) * ((size_t)n_trans + 1);
}

template <int NSTG>
__global__ void __launch_bounds__(PAIR_T, 1) k_lag_pairs(const __grid_constant__ PairArgs A) {
    constexpr int LOOK = NSTG - 1;  // chunks a copying thread runs ahead of the one it hands over
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t s_afull[NSTG], s_bfull[NSTG], s_empty[NSTG], s_accfull[2], s_accempty[2], s_done;
    __shared__ uint32_t s_tmem, s_carry, s_w[PAIR_T / 32];
    __shared__ int s_bad;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t stage = (uint32_t)(HM * HROW * 2 + A.npad * HROW * 2);
    float *stag = reinterpret_cast<float *>(smem + (size_t)NSTG * stage);
    uint32_t *pre = reinterpret_cast<uint32_t *>(stag + 4 * 32 * PAIR_ST);  // tiles before translation t
    if (warp == 8) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&s_tmem)),
                     "r"(2 * A.tcols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        s_bad = 0;
        s_carry = 0;
        for (int i = 0; i < NSTG; ++i) {
            mbar_init(&s_afull[i], 128);
            mbar_init(&s_bfull[i], 1);
            mbar_init(&s_empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&s_accfull[i], 1);
            mbar_init(&s_accempty[i], 128);
        }
        mbar_init(&s_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // tiles of every translation, prefix sums
    for (int t0 = 0; t0 < A.n_trans; t0 += PAIR_T) {
        const int t = t0 + tid;
        uint32_t c = 0;
        if (t < A.n_trans) c = (uint32_t)(((uint64_t)(A.bt_off[t + 1] - A.bt_off[t]) * A.nrhs + HM - 1) / HM);
        uint32_t inc = c;
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        if (lane == 31) s_w[warp] = inc;
        __syncthreads();
        uint32_t before = s_carry;
        for (int w = 0; w < warp; ++w) before += s_w[w];
        if (t < A.n_trans) pre[t] = before + inc - c;
        __syncthreads();
        if (tid == PAIR_T - 1) s_carry = before + inc;
        __syncthreads();
    }
    if (tid == 0) pre[A.n_trans] = s_carry;
    __syncthreads();
    const uint32_t tmem = s_tmem;
    const int64_t units = (int64_t)s_carry * A.nblk;
    // translation, first row and row count of the tile of unit un
    auto locate = [&](int64_t un, int &t, uint32_t &p0, uint64_t &row0, int &nrows) {
        const uint32_t tile = (uint32_t)(un / A.nblk);
        int lo = 0, hi = A.n_trans;  // last t with pre[t] <= tile
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (pre[mid] <= tile)
                lo = mid;
            else
                hi = mid;
        }
        t = lo;
        p0 = A.bt_off[t];
        const uint64_t all = (uint64_t)(A.bt_off[t + 1] - p0) * A.nrhs;
        row0 = (uint64_t)(tile - pre[t]) * HM;
        nrows = (int)min((uint64_t)HM, all - row0);
    };
    bool ok = true;
    if (warp < 4) {
        // ---- copies: lane handles rows 32 warp + 8 g + lane % 8 (g < 4), 16-byte segment lane / 8 of
        // the hi and of the lo part: conflict-free core-matrix stores, 64 contiguous bytes per row
        constexpr uint32_t NONE = 0xffffffffu;
        const uint32_t dst0 = smem_addr(smem) + (uint32_t)((4 * warp) * H_SBO + (lane >> 3) * H_LBO + (lane & 7) * 16);
        int t = 0, tn = 0;
        uint32_t rows[4], rnext[4];
        auto fetch = [&](int64_t un, int &tt, uint32_t (&out)[4]) {
            uint32_t p0;
            uint64_t row0;
            int n;
            locate(un, tt, p0, row0, n);
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const int q = 32 * warp + 8 * g + (lane & 7);
                out[g] = NONE;
                if (q < n) {
                    const uint64_t R = row0 + q;
                    const uint32_t pr = A.nrhs == 1 ? (uint32_t)R : (uint32_t)(R / (uint32_t)A.nrhs);
                    out[g] = A.bt_src[p0 + pr] * (uint32_t)A.nrhs + (uint32_t)(R - (uint64_t)pr * A.nrhs);
                }
            }
        };
        int64_t un = blockIdx.x;
        if (un < units) fetch(un, t, rows);
        uint32_t c = 0;
        auto hand_over = [&](uint32_t done) {  // this thread's copies of chunk `done` have landed
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_arrive(&s_afull[done % NSTG]);
        };
        for (; un < units && ok; un += gridDim.x) {
            if (un + gridDim.x < units) fetch(un + gridDim.x, tn, rnext);
            const int blk = (int)(un % A.nblk);
            const __half *Tb = A.T + ((size_t)t * A.nblk + blk) * A.nk * A.npad * HROW;
            for (int kc = 0; kc < A.nk; ++kc, ++c) {
                const uint32_t slot = c % NSTG;
                if (c >= NSTG && !mbar_wait(&s_empty[slot], ((c / NSTG) - 1) & 1, A.tries, A.err)) {
                    ok = false;
                    break;
                }
                if (tid == 0) {
                    mbar_expect(&s_bfull[slot], (uint32_t)A.npad * HROW * 2);
                    bulk_g2s(smem + (size_t)slot * stage + HM * HROW * 2, Tb + (size_t)kc * A.npad * HROW,
                             (uint32_t)A.npad * HROW * 2, &s_bfull[slot]);
                }
                const uint32_t dst = dst0 + slot * stage;
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    const bool have = rows[g] != NONE;
                    const __half *src = A.u + ((size_t)(have ? rows[g] : 0u) * A.nk + kc) * HROW + (lane >> 3) * 8;
                    cp_async16_zfill(dst + g * H_SBO, src, have ? 16u : 0u);
                    cp_async16_zfill(dst + g * H_SBO + HM * HK * 2, src + HK, have ? 16u : 0u);
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
                asm volatile("cp.async.wait_group %0;" ::"n"(LOOK) : "memory");
                if (c >= LOOK) hand_over(c - LOOK);
            }
            t = tn;
#pragma unroll
            for (int g = 0; g < 4; ++g) rows[g] = rnext[g];
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (ok)
            for (uint32_t d = c > LOOK ? c - LOOK : 0; d < c; ++d) hand_over(d);
        // the operator copies of the last chunks (all others have been consumed)
        if (tid == 0)
            for (uint32_t d = c > NSTG ? c - NSTG : 0; d < c; ++d)
                mbar_wait(&s_bfull[d % NSTG], (d / NSTG) & 1, DRAIN_TRIES);
    } else if (warp == 8) {
        if (lane == 0) {
            // ---- MMA thread
            const uint32_t id1 = idesc_f16(A.npad), id2 = A.stack ? idesc_f16(2 * A.npad) : id1;
            const uint32_t base = smem_addr(smem);
            uint32_t c = 0, i = 0;
            for (int64_t un = blockIdx.x; un < units && ok; un += gridDim.x, ++i) {
                const uint32_t buf = i & 1;
                if (i >= 2 && !mbar_wait(&s_accempty[buf], ((i >> 1) - 1) & 1, A.tries, A.err)) {
                    ok = false;
                    break;
                }
                const uint32_t d = tmem + buf * (uint32_t)A.tcols;
                for (int kc = 0; kc < A.nk; ++kc, ++c) {
                    const uint32_t slot = c % NSTG, par = (c / NSTG) & 1;
                    if (!mbar_wait(&s_bfull[slot], par, A.tries, A.err) ||
                        !mbar_wait(&s_afull[slot], par, A.tries, A.err)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t ah = base + slot * stage, al = ah + HM * HK * 2, bh = ah + HM * HROW * 2;
                    const uint32_t bl = bh + (uint32_t)A.npad * HK * 2;
#pragma unroll
                    for (int ks = 0; ks < HK / 16; ++ks) {
                        const uint64_t dah = umma_desc(ah + ks * 2 * H_LBO, H_LBO, H_SBO);
                        const uint64_t dal = umma_desc(al + ks * 2 * H_LBO, H_LBO, H_SBO);
                        const uint64_t dbh = umma_desc(bh + ks * 2 * H_LBO, H_LBO, H_SBO);
                        const uint32_t acc = kc > 0 || ks > 0;
                        mma_f16(d, dah, dbh, id2, acc);
                        if (A.stack) {
                            mma_f16(d + (uint32_t)A.npad, dal, dbh, id1, 1u);
                        } else {
                            mma_f16(d, dah, umma_desc(bl + ks * 2 * H_LBO, H_LBO, H_SBO), id1, 1u);
                            mma_f16(d, dal, dbh, id1, 1u);
                        }
                    }
                    tc_commit(&s_empty[slot]);
                }
                if (ok) tc_commit(&s_accfull[buf]);
            }
            // everything issued is done before the block gives up its shared memory and TMEM
            tc_commit(&s_done);
            mbar_wait(&s_done, 0, DRAIN_TRIES);
        }
    } else {
        // ---- epilogue: warp w reads lanes 32 (w - 4) .. + 31
        const int q = warp - 4;
        float *st = stag + q * 32 * PAIR_ST;
        const bool vec = (A.ostride & 3) == 0;
        // rows of this warp with pairs (<= 0: none), this lane's row of v~ and its source's scale;
        // fetched one unit ahead, a chain of dependent loads
        auto fetch = [&](int64_t un, int &mine, int64_t &drow, float &inv) {
            int t, n;
            uint32_t p0;
            uint64_t row0;
            locate(un, t, p0, row0, n);
            mine = n - 32 * q;
            if (lane < mine) {
                const uint64_t R = row0 + 32 * q + lane;
                const uint32_t pr = A.nrhs == 1 ? (uint32_t)R : (uint32_t)(R / (uint32_t)A.nrhs);
                const uint32_t m = (uint32_t)(R - (uint64_t)pr * A.nrhs);
                drow = (int64_t)A.bt_tgt[p0 + pr] * A.nrhs + m;
                inv = A.uinv[(int64_t)A.bt_src[p0 + pr] * A.nrhs + m];
            }
        };
        int mine = 0, mine_n = 0;
        int64_t drow = 0, drow_n = 0;
        float inv = 0.f, inv_n = 0.f;
        uint32_t i = 0;
        if (blockIdx.x < units) fetch(blockIdx.x, mine_n, drow_n, inv_n);
        for (int64_t un = blockIdx.x; un < units; un += gridDim.x, ++i) {
            mine = mine_n;
            drow = drow_n;
            inv = inv_n;
            if (un + gridDim.x < units) fetch(un + gridDim.x, mine_n, drow_n, inv_n);
            const int blk = (int)(un % A.nblk), nout = A.nout[blk];
            const uint32_t buf = i & 1;
            const bool w_ok = mbar_wait(&s_accfull[buf], (i >> 1) & 1, A.tries, A.err);
            if (!__all_sync(0xffffffffu, w_ok)) {
                ok = false;
                break;
            }
            tc_fence_after();
            const uint32_t d = tmem + buf * (uint32_t)A.tcols + ((uint32_t)(32 * q) << 16);
            float *out = A.vt + A.ooff[blk];
            if (mine > 0) {
                for (int c0 = 0; c0 < nout; c0 += 32) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int cc = c0 + 16 * h;
                        if (cc >= A.npad) break;
                        uint32_t v[16], w[16];
                        tmem_ld16(v, d + (uint32_t)cc);
                        if (A.stack) tmem_ld16(w, d + (uint32_t)(A.npad + cc));
                        tmem_wait_ld();
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            float x[4];
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                float y = __uint_as_float(v[4 * k + j]);
                                if (A.stack) y += __uint_as_float(w[4 * k + j]);
                                x[j] = y * inv * A.tinv;
                            }
                            *reinterpret_cast<float4 *>(st + lane * PAIR_ST + 16 * h + 4 * k) =
                                make_float4(x[0], x[1], x[2], x[3]);
                        }
                    }
                    __syncwarp();
                    if (vec) {
                        const int col = c0 + (lane & 7) * 4;
#pragma unroll
                        for (int it = 0; it < 8; ++it) {
                            const int row = it * 4 + (lane >> 3);
                            const int64_t dr = __shfl_sync(0xffffffffu, drow, row);
                            if (row < mine && col < nout)
                                atomicAdd(reinterpret_cast<float4 *>(out + dr * A.ostride + col),
                                          *reinterpret_cast<const float4 *>(st + row * PAIR_ST + (lane & 7) * 4));
                        }
                    } else {
                        for (int row = 0; row < min(mine, 32); ++row) {
                            const int64_t dr = __shfl_sync(0xffffffffu, drow, row);
                            if (c0 + lane < nout) atomicAdd(out + dr * A.ostride + c0 + lane, st[row * PAIR_ST + lane]);
                        }
                    }
                    __syncwarp();
                }
            }
            tc_fence_before();
            mbar_arrive(&s_accempty[buf]);
        }
    }
    if (!ok) s_bad = 1;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid == 0 && s_bad) atomicOr(A.err, 1);
    if (warp == 8)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * A.tcols));
}

// Operator images of a Lagrange level (F.T is in place).  The scale is common to the level's
// translations: the kernels decay at most as 1/R^2 and the distances of a level's node pairs
// differ by at most a factor of about ten, so every translation keeps its bits.
void build_operator_image(ffm_plan_s *p, int l, const double oxy[3], double dl, cudaStream_t s) {
    FarLevel &F = p->far[l];
    const bool cplx = p->kind == FFM_HELMHOLTZ;
    const int r = F.r1 * F.r1 * F.r1, rk = p->kind == FFM_LAPLACE_DL ? 3 * r : r;
    const int rows = cplx ? 2 * r : r, K = cplx ? 2 * rk : rk, ncomp = p->kind == FFM_LAPLACE_GRAD ? 3 : 1;
    F.h_bpc = cdiv(rows, 256);
    F.h_nb = ((int)cdiv(rows, F.h_bpc) + 15) / 16 * 16;
    F.h_nk = cdiv(K, HK);
    const int nblk = F.h_bpc * ncomp;
    // the largest |T|: the closest node pair of the closest translation
    double rmin = INFINITY;
    for (const int4 &m : F.h_trans_m) {
        const double x = oxy[0] + m.x * dl, y = oxy[1] + m.y * dl, z = oxy[2] + m.z * dl;
        rmin = std::min(rmin, std::sqrt(x * x + y * y + z * z));
    }
    const double dist = std::max(dl, rmin - std::sqrt(3.0) * dl);
    const bool square = p->kind == FFM_LAPLACE_DL || p->kind == FFM_LAPLACE_GRAD;
    const double amax = 1.0 / (4.0 * PI * (square ? dist * dist : dist));
    int e = 13 - (int)std::ceil(std::log2(amax));
    e = std::max(-120, std::min(120, e));
    F.h_inv = (float)std::ldexp(1.0, -e);
    const size_t n = (size_t)F.n_trans * nblk * F.h_nk * F.h_nb * HROW;
    F.Th = p->mem.get<uint16_t>(n);
    dim3 g(F.n_trans, nblk);
    const float sc = (float)std::ldexp(1.0, e);
    if (cplx)
        FFM_LAUNCH(k_op_image<true>, g, 256, 0, s, F.T, F.n_trans, r, rk, F.h_nb, F.h_bpc, F.h_nb, F.h_nk, sc, (__half *)F.Th);
    else
        FFM_LAUNCH(k_op_image<false>, g, 256, 0, s, F.T, F.n_trans, r, rk, F.h_nb, F.h_bpc, F.h_nb, F.h_nk, sc, (__half *)F.Th);
}

template <int NSTG>
static void launch_pairs(const PairArgs &A, unsigned grid, cudaStream_t s) {
    const size_t sm = pair_smem(NSTG, A.npad, A.n_trans);
    // per device and cheap: set before every launch (plans may live on several devices)
    FFM_CUDA(cudaFuncSetAttribute(k_lag_pairs<NSTG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    FFM_LAUNCH_NAMED("k_lag_pairs", k_lag_pairs<NSTG>, grid, PAIR_T, sm, s, A);
}

// v~ += T u~ for all pairs of the level: u has rows of K floats per (source box, right-hand side),
// v~ rows of `rows` floats per (target box, right-hand side) and component
void lag_pairs(const ffm_plan_s *p, int l, const float *u, int nrhs, float *vt, Alloc &tmp, cudaStream_t s) {
    const FarLevel &F = p->far[l];
    const bool cplx = p->kind == FFM_HELMHOLTZ;
    const int r = F.r1 * F.r1 * F.r1, rk = p->kind == FFM_LAPLACE_DL ? 3 * r : r;
    const int rows = cplx ? 2 * r : r, K = cplx ? 2 * rk : rk, ncomp = p->kind == FFM_LAPLACE_GRAD ? 3 : 1;
    const int64_t nrow = (int64_t)p->by[l].nb * nrhs;
    PairArgs A{};
    __half *img = tmp.get<__half>((size_t)nrow * F.h_nk * HROW);
    float *inv = tmp.get<float>(nrow);
    FFM_LAUNCH(k_rows_split, cdiv(nrow, 8), 256, 0, s, u, nrow, K, F.h_nk, img, inv);
    A.bt_off = F.bt_off;
    A.bt_src = F.bt_src;
    A.bt_tgt = F.bt_tgt;
    A.n_trans = F.n_trans;
    A.nrhs = nrhs;
    A.nblk = F.h_bpc * ncomp;
    A.u = img;
    A.uinv = inv;
    A.T = (const __half *)F.Th;
    A.tinv = F.h_inv;
    A.nk = F.h_nk;
    A.npad = F.h_nb;
    A.stack = F.h_nb <= 128;
    A.tcols = 32;
    while (A.tcols < (A.stack ? 2 : 1) * A.npad) A.tcols <<= 1;
    A.ostride = rows;
    const int64_t vblk = (int64_t)rows * nrhs * p->bx[l].nb;
    for (int b = 0; b < A.nblk; ++b) {
        const int row0 = (b % F.h_bpc) * F.h_nb;
        A.nout[b] = std::min(F.h_nb, rows - row0);
        A.ooff[b] = (b / F.h_bpc) * vblk + row0;
    }
    A.vt = vt;
    A.err = p->dev_err;
    A.tries = p->wait_tries;
    const int64_t most = ((int64_t)F.n_trans + F.n_adm * nrhs / HM) * A.nblk;  // at least the number of units
    const unsigned grid = (unsigned)std::min<int64_t>(most, 152);
    if (A.npad <= 64)
        launch_pairs<8>(A, grid, s);
    else if (A.npad <= 128)
        launch_pairs<6>(A, grid, s);
    else
        launch_pairs<4>(A, grid, s);
    tmp.drop(inv);
    tmp.drop(img);
}

}  // namespace ffm
