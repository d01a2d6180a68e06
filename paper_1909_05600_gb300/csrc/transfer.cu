// Transfers of the Lagrange levels on the tensor cores (Sec. 2.2.2: v~_a += T_t u~_b for every
// admissible pair (a, b) of translation t), with f16 operands split in two.
//
// Split.  Every operand value x is written as hi + lo with hi = f16(x s) and lo = f16(x s - hi),
// s a power of two, and a product is hi hi + hi lo + lo hi in FP32 accumulators.  Both
// roundings are to nearest: |lo| is at most 2^-11 of the value, hi + lo is within 2^-22 of it, and the
// dropped lo lo term is at most 2^-22 of the product (x = y = 1 + 2^-11 reach it; over random operands each of the
// three is 2^-24.3 in the root mean square, and a row's sum of 216 products is off by 1e-8).  The TF32 split used
// before truncated (hi: 11 bits, lo: 11 bits of the rest), which is four to eight times coarser, and f16
// runs at twice the TF32 rate.  The scale keeps the largest value of a row between 2^13 and 2^14, so a
// value keeps its 22 bits down to 2^-15 of its row's largest, and below that an absolute error of at most 2^-38
// of it.
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
constexpr uint32_t A_BYTES = HM * HROW * 2;  // a tile's rows, one chunk

// The gathered rows lie in shared memory as 128-byte rows (hi, then lo) in the 128-byte swizzle:
// 16-byte segment c of row i at 128 i + 16 (c ^ (i % 8)).  A warp's cp.async writes whole 128-byte
// lines of it (4 wavefronts for 4 rows); in the no-swizzle core-matrix order the same copies, 64
// bytes of a row spread over four lines, took 26 wavefronts.
// Descriptor words: the high ones are constants (rows: 128-byte swizzle, 1024 bytes between 8-row
// groups; operator: no swizzle, H_SBO), the low ones address / 16 and the K stride.
constexpr uint32_t A_DHI = (1024u >> 4) | (1u << 14) | (2u << 29), B_DHI = ((uint32_t)H_SBO >> 4) | (1u << 14);
__device__ __forceinline__ uint32_t a_dlo(uint32_t saddr) { return (saddr >> 4) | (1u << 16); }
__device__ __forceinline__ uint32_t b_dlo(uint32_t saddr) { return (saddr >> 4) | ((uint32_t)(H_LBO >> 4) << 16); }

// The MMAs of one stage (CPS chunks of 32 K values: the chunks' rows, then the operator's chunks) into
// accumulator d: hi hi + hi lo + lo hi per K step of 16.  alo, blo: low descriptor words of the stage's
// first chunk.  STACK: the operator's hi and lo rows as one operand of 2 npad rows, so that hi hi and
// hi lo are one MMA (lo hi joins hi lo in columns npad ..).  The issuing thread's own instructions
// are what a small stage waits for (its 4 MMAs took 1200 cycles with 64-bit descriptors formed
// for each and two barriers per chunk), so they are kept to an add and the MMA.
template <int CPS, bool STACK>
__device__ __forceinline__ void stage_mma(uint32_t d, uint32_t alo, uint32_t blo, uint32_t npad, uint32_t id1,
                                          uint32_t id2, bool first) {
#pragma unroll
    for (int kc = 0; kc < CPS; ++kc) {
#pragma unroll
        for (int ks = 0; ks < HK / 16; ++ks) {
            const uint32_t ah = alo + kc * (A_BYTES >> 4) + ks * 2, al = ah + (HK * 2 >> 4);
            const uint32_t bh = blo + kc * npad * (HROW * 2 >> 4) + ks * (2 * H_LBO >> 4);
            const uint32_t acc = kc > 0 || ks > 0 || !first;
            mma_f16(d, ah, A_DHI, bh, B_DHI, id2, acc);
            if constexpr (STACK) {
                mma_f16(d + npad, al, A_DHI, bh, B_DHI, id1, 1u);
            } else {
                mma_f16(d, ah, A_DHI, bh + npad * (HK * 2 >> 4), B_DHI, id1, 1u);
                mma_f16(d, al, A_DHI, bh, B_DHI, id1, 1u);
            }
        }
    }
}

// dynamic shared memory from its first 1024-byte boundary (the swizzle repeats every 1024 bytes)
__device__ __forceinline__ unsigned char *aligned_smem(unsigned char *p) {
    return p + ((1024u - (smem_addr(p) & 1023u)) & 1023u);
}

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

// The two scales' inverses (powers of two) as factors f1 f2 = a b of about equal size: a value times f1, then f2,
// stays between the value and the result, so it leaves FP32's range only where the result does
// (densities of 1e34 and more did, with a and b one after the other).
__device__ __forceinline__ void even_factors(float a, float b, float &f1, float &f2) {
    const int e = (__float_as_int(a) >> 23) + (__float_as_int(b) >> 23) - 254, h = e >> 1;  // |e| <= 240
    f1 = __int_as_float((127 + h) << 23);
    f2 = __int_as_float((127 + e - h) << 23);
}

__device__ __forceinline__ void half_split(float x, __half &hi, __half &lo) {
    hi = __float2half_rn(x);
    lo = __float2half_rn(x - __half2float(hi));
}

// Rows of n floats as f16 hi / lo images, one warp per row: chunk kc of row i holds the hi
// parts of values 32 kc .. + 31, then their lo parts (zero past n).  The scale is the row's own
// (its inverse in inv[i]), or with `common` that of the largest value of the row's column (right-hand side
// i % nrhs): never one of several columns, whose magnitudes have nothing to do with each other.
__global__ void __launch_bounds__(256) k_rows_split(const float *__restrict__ u, int64_t nrow, int n, int nk,
                                                    __half *__restrict__ img, float *__restrict__ inv,
                                                    const uint32_t *__restrict__ common, int nrhs) {
    const int64_t i = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (i >= nrow) return;
    const float *row = u + i * n;
    float mx = 0.f;
    if (common) {
        mx = __uint_as_float(common[nrhs == 1 ? 0 : i % nrhs]);
    } else {
        for (int k = lane; k < n; k += 32) mx = fmaxf(mx, fabsf(row[k]));
        for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    float s, si;
    row_scale(mx, s, si);
    if (lane == 0 && !common) inv[i] = si;
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

// Operators as the images the transfers copy: per translation t and row block blk, nk chunks of
// the hi parts of npad rows x 32 values in K-major core matrices, then the lo parts.  Block blk
// holds rows (blk % bpc) nb .. of component blk / bpc.  A complex operator is the real matrix
// of its action on interleaved (re, im) rows: rows 2i, 2i + 1 = (Re, -Im), (Im, Re) of T(i, j) at
// columns 2j, 2j + 1.  The values are k_lag_table's (the same FP32 expressions), formed here so that no
// FP32 operator is written and read back; with the node count a template parameter the index
// arithmetic is free of divisions (volume 250k at 1e-4: table and image 0.54 + 0.34 -> 0.36 ms).
template <int KIND, int R1>
__global__ void __launch_bounds__(256) k_op_image(const int4 *__restrict__ m, const __grid_constant__ LagGeo geo, int nb,
                                                  int bpc, int npad, int nk, float scale, __half *__restrict__ img) {
    constexpr int r = R1 * R1 * R1;
    constexpr bool CPLX = KIND == FFM_HELMHOLTZ;
    constexpr int rows = CPLX ? 2 * r : r, cols = CPLX ? 2 * r : KIND == FFM_LAPLACE_DL ? 3 * r : r;
    __shared__ float node[R1];
    if (threadIdx.x < R1) node[threadIdx.x] = geo.hnode[threadIdx.x];
    __syncthreads();
    const int t = blockIdx.x, blk = blockIdx.y, nblk = gridDim.y;
    const int comp = blk / bpc, row0 = (blk % bpc) * nb;
    const int4 mt = m[t];
    const float r0x = (float)(geo.oxy[0] + mt.x * geo.dl), r0y = (float)(geo.oxy[1] + mt.y * geo.dl),
                r0z = (float)(geo.oxy[2] + mt.z * geo.dl);
    const float c4pi = 0.07957747154594767f;  // 1 / (4 pi)
    auto diff = [&](int i, int j, float (&d)[3]) {
        d[0] = r0x + (node[i / (R1 * R1)] - node[j / (R1 * R1)]);
        d[1] = r0y + (node[i / R1 % R1] - node[j / R1 % R1]);
        d[2] = r0z + (node[i % R1] - node[j % R1]);
    };
    auto value = [&](int i, int j, int c) {  // component c of the derivative kernels
        float d[3];
        diff(i, j, d);
        const float r2 = fmaf(d[0], d[0], fmaf(d[1], d[1], d[2] * d[2])), rr = sqrtf(r2);
        if constexpr (KIND == FFM_LAPLACE) return c4pi / rr;
        const float dc = c == 0 ? d[0] : c == 1 ? d[1] : d[2];
        return (KIND == FFM_LAPLACE_GRAD ? -c4pi : c4pi) * dc / (r2 * rr);
    };
    __half *out = img + ((size_t)t * nblk + blk) * nk * npad * HROW;
    const int per = npad * HK;  // values per chunk
    for (int e = threadIdx.x; e < nk * per / 2; e += blockDim.x) {  // two columns each
        const int kc = 2 * e / per, o = 2 * e - kc * per;
        const int k = kc * HK + ((o >> 6) & 3) * 8 + (o & 7), i = ((o >> 8) << 3) + ((o >> 3) & 7), ri = row0 + i;
        float v0 = 0.f, v1 = 0.f;
        if (i < nb && ri < rows) {
            if constexpr (CPLX) {
                if (k < cols) {
                    float d[3], sn, cs;
                    diff(ri >> 1, k >> 1, d);
                    const float rr = sqrtf(fmaf(d[0], d[0], fmaf(d[1], d[1], d[2] * d[2]))), a = c4pi / rr;
                    sincosf(geo.k * rr, &sn, &cs);
                    const float re = a * cs, im = a * sn;
                    v0 = ri & 1 ? im : re;
                    v1 = ri & 1 ? re : -im;
                }
            } else {
                if (k < cols) v0 = value(ri, k % r, KIND == FFM_LAPLACE_DL ? k / r : comp);
                if (k + 1 < cols) v1 = value(ri, (k + 1) % r, KIND == FFM_LAPLACE_DL ? (k + 1) / r : comp);
            }
        }
        __half h0, l0, h1, l1;
        half_split(v0 * scale, h0, l0);
        half_split(v1 * scale, h1, l1);
        __half *c = out + (size_t)kc * npad * HROW;
        *reinterpret_cast<__half2 *>(c + o) = __halves2half2(h0, h1);
        *reinterpret_cast<__half2 *>(c + per + o) = __halves2half2(l0, l1);
    }
}

template <int R1>
static void launch_op_image(int kind, dim3 g, const int4 *m, const LagGeo &geo, int nb, int bpc, int nk, float sc,
                            __half *img, cudaStream_t s) {
    auto run = [&](auto k) { FFM_LAUNCH_NAMED("k_op_image", k, g, 256, 0, s, m, geo, nb, bpc, nb, nk, sc, img); };
    switch (kind) {
        case FFM_HELMHOLTZ: run(k_op_image<FFM_HELMHOLTZ, R1>); break;
        case FFM_LAPLACE_DL: run(k_op_image<FFM_LAPLACE_DL, R1>); break;
        case FFM_LAPLACE_GRAD: run(k_op_image<FFM_LAPLACE_GRAD, R1>); break;
        default: run(k_op_image<FFM_LAPLACE, R1>); break;
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
    int part;           // chunks per accumulator fill (all of them but for complex operators)
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
//   warps 9-12  fetch the row numbers (source, target, source scale) of coming units, one warp a unit,
//               into a ring in shared memory: a chain of dependent loads that no copying or adding
//               thread waits for
//   warps 0-3   copy the tile's rows (hi and lo, 16 KB) with cp.async, rows past the tile's pairs
//               zero-filled
//   thread 0    also starts the bulk copy of the operator's chunk (128 npad bytes)
//   warp 8      issues the MMAs into one of two TMEM accumulators
//   warps 4-7   read the other accumulator, undo the scales and add it into v~: 32 columns at a
//               time through shared memory, so that eight lanes add 128 consecutive bytes
//               (complex operators: also warps 13-16, see SUM)
// The MMAs of a K step are hi [hi; lo] (one operand of 2 npad rows, accumulated apart) and lo hi
// up to 128 operator rows, else three of npad rows into one accumulator.
// NSTG stages of CPS chunks are in flight: 4 of two at npad = 64 (48 KB each), 4 of one at 224 (45 KB).
//
// Measured on GB300 (level 7 of clustered 10M, 68M pairs of r = 64): 11.7 ms with the row numbers fetched
// by the copying and adding threads themselves, 9.85 with index warps, 6.98 with rows in the swizzled
// layout, 6.14 with the lean MMA loop.  Transfers of one apply, against the kernel before it (a block per
// 256-pair tile, which split its FP32 rows into TF32 for every pair, no overlap of tiles): gradient
// sphere 300k (r = 216, three operators) 6.54 -> 1.78 ms, Laplace volume 250k at 1e-4 (r = 216) 1.47 ->
// 0.45, 100k x 8 right-hand sides (r = 64) 1.68 -> 0.41.  Complex operators (Helmholtz volume 120k at
// 1e-4, 432 real rows), on CUDA cores before: 24.4 -> 1.77 ms (1.91 with both halves of K scattered).
constexpr int PAIR_T = 416, PAIR_TS = PAIR_T + 128;  // threads; with SUM
// Chunks per accumulator fill of a complex operator.  With 1, 2, 4, 8 and 14 (all of K) the transfer of the Helmholtz
// volume 120k at 1e-4 takes 3.02, 2.27, 1.77, 1.69 and 1.64 ms; the product of a plane-wave density in a volume of
// 40k points (k = 3, 1e-4) is 2.7, 2.9, 3.7 and 5.1e-7 of the oracle's FFM for the first four.  FP32
// multiply-adds on CUDA cores, with the basis constants of their time, took 24.4 ms and gave 6.1e-7.
constexpr int PAIR_PART = 4;
// Most translations of a level: the near offsets of the parents take at most four values per axis, their children's
// at most nine, and the 64 offsets that stay near are none of them.
constexpr int MAX_TRANS = 9 * 9 * 9 - 4 * 4 * 4;
constexpr int PAIR_IXW = 4;  // index warps
constexpr int PAIR_IX = 4;   // units whose row numbers are held
constexpr int PAIR_ST = 36;  // floats per row of the epilogue's staging (conflict-free float4)

static size_t pair_smem(int nchunk, int npad, int n_trans, bool sum) {
    return 1024 + nchunk * (A_BYTES + (size_t)npad * HROW * 2) + (sum ? 8 : 4) * 32 * PAIR_ST * sizeof(float) +
           sizeof(uint32_t) * ((size_t)n_trans + 1);
}

// SUM (complex operators): a tensor-core accumulation truncates at every step, so hi hi is accumulated over
// A.part chunks only; the epilogue adds the fills of a unit in FP32 registers, rounded to nearest, and
// scatters the unit once.  Two warps per lane quarter (4-7 and 13-16) then take half of the columns each.
template <int NSTG, int CPS, bool STACK, bool SUM>
__global__ void __launch_bounds__(SUM ? PAIR_TS : PAIR_T, 1) k_lag_pairs(const __grid_constant__ PairArgs A) {
    constexpr int T = SUM ? PAIR_TS : PAIR_T, EPW = SUM ? 8 : 4;  // threads, epilogue warps
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = aligned_smem(smem_raw);
    __shared__ __align__(8) uint64_t s_full[NSTG], s_empty[NSTG], s_accfull[2], s_accempty[2], s_done;
    __shared__ __align__(8) uint64_t s_ixfull[PAIR_IX], s_ixempty[PAIR_IX];
    __shared__ uint32_t s_src[PAIR_IX][HM];  // row of the images, NONE past the tile's pairs
    __shared__ uint32_t s_dst[PAIR_IX][HM];  // row of v~
    __shared__ float s_inv[PAIR_IX][HM];
    __shared__ int s_trans[PAIR_IX];
    __shared__ uint32_t s_tmem, s_carry, s_cmax, s_w[T / 32];
    constexpr uint32_t NONE = 0xffffffffu;
    __shared__ int s_bad;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t bbytes = (uint32_t)A.npad * HROW * 2 * CPS, stage = CPS * A_BYTES + bbytes;
    float *stag = reinterpret_cast<float *>(smem + (size_t)NSTG * stage);
    uint32_t *pre = reinterpret_cast<uint32_t *>(stag + EPW * 32 * PAIR_ST);  // tiles before translation t
    if (warp == 8) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&s_tmem)),
                     "r"(2 * A.tcols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        s_bad = 0;
        s_cmax = 0;
        s_carry = 0;
        for (int i = 0; i < NSTG; ++i) {
            mbar_init(&s_full[i], 129);  // the copying threads, and the operator copy's byte count
            mbar_init(&s_empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&s_accfull[i], 1);
            mbar_init(&s_accempty[i], EPW);
        }
        for (int i = 0; i < PAIR_IX; ++i) {
            mbar_init(&s_ixfull[i], 1);
            mbar_init(&s_ixempty[i], 4 + EPW);
        }
        mbar_init(&s_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // tiles of every translation, prefix sums
    for (int t0 = 0; t0 < A.n_trans; t0 += T) {
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
        if (tid == T - 1) s_carry = before + inc;
        __syncthreads();
    }
    if (tid == 0) pre[A.n_trans] = s_carry;
    __syncthreads();
    const uint32_t tmem = s_tmem;
    const int64_t units = (int64_t)s_carry * A.nblk;
    auto block_of = [&](int64_t un) { return (int)(un % A.nblk); };  // row block of unit un
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
    if (warp > 8 && warp < 9 + PAIR_IXW) {
        // ---- row numbers: warp w takes units w - 9, w - 9 + PAIR_IXW, ... of this block
        uint32_t i = warp - 9;
        for (int64_t un = blockIdx.x + (int64_t)i * gridDim.x; un < units; un += (int64_t)PAIR_IXW * gridDim.x, i += PAIR_IXW) {
            const uint32_t k = i % PAIR_IX;
            int t, n;
            uint32_t p0;
            uint64_t row0;
            locate(un, t, p0, row0, n);
            uint32_t src[4], dst[4];
            float inv[4];
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const int q = 32 * g + lane;
                src[g] = NONE;
                dst[g] = 0u;
                inv[g] = 0.f;
                if (q < n) {
                    const uint64_t R = row0 + q;
                    const uint32_t pr = A.nrhs == 1 ? (uint32_t)R : (uint32_t)(R / (uint32_t)A.nrhs);
                    const uint32_t m = (uint32_t)(R - (uint64_t)pr * A.nrhs);
                    src[g] = A.bt_src[p0 + pr] * (uint32_t)A.nrhs + m;
                    dst[g] = A.bt_tgt[p0 + pr] * (uint32_t)A.nrhs + m;
                }
            }
#pragma unroll
            for (int g = 0; g < 4; ++g)
                if (src[g] != NONE) inv[g] = A.uinv[src[g]];
            const bool w_ok = i < PAIR_IX || mbar_wait(&s_ixempty[k], ((i / PAIR_IX) - 1) & 1, A.tries, A.err);
            if (!__all_sync(0xffffffffu, w_ok)) {
                ok = false;
                break;
            }
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                s_src[k][32 * g + lane] = src[g];
                s_dst[k][32 * g + lane] = dst[g];
                s_inv[k][32 * g + lane] = inv[g];
            }
            if (lane == 0) s_trans[k] = t;
            __syncwarp();
            if (lane == 0) mbar_arrive(&s_ixfull[k]);
        }
    } else if (warp < 4) {
        // ---- copies: lane handles 16-byte segment lane % 8 of rows 32 warp + 4 g + lane / 8 (g < 8)
        const uint32_t r0 = 32 * warp + (lane >> 3), sg = lane & 7;
        const uint32_t dst0 = smem_addr(smem) + r0 * 128, sw0 = (sg ^ (r0 & 7)) * 16, sw1 = (sg ^ ((r0 + 4) & 7)) * 16;
        uint32_t c = 0, i = 0;
        for (int64_t un = blockIdx.x; un < units && ok; un += gridDim.x, ++i) {
            const uint32_t ix = i % PAIR_IX;
            const bool i_ok = mbar_wait(&s_ixfull[ix], (i / PAIR_IX) & 1, A.tries, A.err);
            if (!__all_sync(0xffffffffu, i_ok)) {
                ok = false;
                break;
            }
            const int t = s_trans[ix], blk = block_of(un);
            const __half *src[8];
            uint32_t bytes[8];
#pragma unroll
            for (int g = 0; g < 8; ++g) {
                const uint32_t row = s_src[ix][r0 + 4 * g];
                bytes[g] = row != NONE ? 16u : 0u;
                src[g] = A.u + (size_t)(row != NONE ? row : 0u) * A.nk * HROW + sg * 8;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&s_ixempty[ix]);
            const __half *Tb = A.T + ((size_t)t * A.nblk + blk) * A.nk * A.npad * HROW;
            for (int kc = 0; kc < A.nk; kc += CPS, ++c) {
                const uint32_t slot = c % NSTG;
                const bool w_ok = c < NSTG || mbar_wait(&s_empty[slot], ((c / NSTG) - 1) & 1, A.tries, A.err);
                if (!__all_sync(0xffffffffu, w_ok)) {
                    ok = false;
                    break;
                }
                if (tid == 0) {
                    mbar_expect(&s_full[slot], bbytes);
                    bulk_g2s(smem + (size_t)slot * stage + CPS * A_BYTES, Tb + (size_t)kc * A.npad * HROW, bbytes,
                             &s_full[slot]);
                }
                const uint32_t dst = dst0 + slot * stage;
#pragma unroll
                for (int g = 0; g < 8; ++g) {
#pragma unroll
                    for (int j = 0; j < CPS; ++j)
                        cp_async16_zfill(dst + j * A_BYTES + g * 512 + ((g & 1) ? sw1 : sw0), src[g] + j * HROW, bytes[g]);
                    src[g] += CPS * HROW;
                }
                cp_async_arrive(&s_full[slot]);
            }
        }
        // After a give-up some warps may have copied further than others: all arrive on every stage any of
        // them started, so that the operator copies can be waited for.
        if (!ok) atomicOr(&s_bad, 1);
        asm volatile("cp.async.wait_all;" ::: "memory");
        atomicMax(&s_cmax, c);
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (s_bad) {
            const uint32_t last = *reinterpret_cast<volatile uint32_t *>(&s_cmax);
            for (; c < last; ++c) {
                if (tid == 0) mbar_arrive(&s_full[c % NSTG]);
                mbar_arrive(&s_full[c % NSTG]);
            }
        }
        if (tid == 0)
            for (uint32_t d = c > NSTG ? c - NSTG : 0; d < c; ++d)
                mbar_wait(&s_full[d % NSTG], (d / NSTG) & 1, DRAIN_TRIES);
    } else if (warp == 8) {
        if (lane == 0) {
            // ---- MMA thread
            const uint32_t id1 = idesc_f16(A.npad), id2 = STACK ? idesc_f16(2 * A.npad) : id1;
            const uint32_t alo = a_dlo(smem_addr(smem)), blo = b_dlo(smem_addr(smem) + CPS * A_BYTES);
            uint32_t f = 0, slot = 0, par = 0;  // accumulator fills
            for (int64_t un = blockIdx.x; un < units && ok; un += gridDim.x) {
                for (int k0 = 0; k0 < A.nk && ok; k0 += A.part, ++f) {
                    const uint32_t buf = f & 1;
                    if (f >= 2 && !mbar_wait(&s_accempty[buf], ((f >> 1) - 1) & 1, A.tries, A.err)) {
                        ok = false;
                        break;
                    }
                    const uint32_t d = tmem + buf * (uint32_t)A.tcols;
                    const int k1 = min(k0 + A.part, A.nk);
                    for (int kc = k0; kc < k1; kc += CPS) {
                        if (!mbar_wait(&s_full[slot], par, A.tries, A.err)) {
                            ok = false;
                            break;
                        }
                        fence_proxy_async();  // the rows came by cp.async, through the generic proxy
                        tc_fence_after();
                        const uint32_t off = slot * (stage >> 4);
                        stage_mma<CPS, STACK>(d, alo + off, blo + off, (uint32_t)A.npad, id1, id2, kc == k0);
                        tc_commit(&s_empty[slot]);
                        if (++slot == NSTG) {
                            slot = 0;
                            par ^= 1;
                        }
                    }
                    if (ok) tc_commit(&s_accfull[buf]);
                }
            }
            // everything issued is done before the block gives up its shared memory and TMEM
            tc_commit(&s_done);
            mbar_wait(&s_done, 0, DRAIN_TRIES);
        }
    } else {
        // ---- epilogue: warp w reads lanes 32 (w % 4) .. + 31
        const int q = warp & 3;
        float *st = stag + (q + (warp > 8 ? 4 : 0)) * 32 * PAIR_ST;
        const bool vec = (A.ostride & 3) == 0;
        uint32_t i = 0, f = 0;  // units, accumulator fills
        for (int64_t un = blockIdx.x; un < units && ok; un += gridDim.x, ++i) {
            const uint32_t ix = i % PAIR_IX;
            const int blk = block_of(un), nout = A.nout[blk];
            const bool i_ok = mbar_wait(&s_ixfull[ix], (i / PAIR_IX) & 1, A.tries, A.err);
            if (!__all_sync(0xffffffffu, i_ok)) {
                ok = false;
                break;
            }
            float f1, f2;
            even_factors(s_inv[ix][32 * q + lane], A.tinv, f1, f2);
            const uint32_t drow = s_dst[ix][32 * q + lane];
            // rows of this warp with pairs (a prefix)
            const int mine = __popc(__ballot_sync(0xffffffffu, s_src[ix][32 * q + lane] != NONE));
            if (lane == 0) mbar_arrive(&s_ixempty[ix]);
            float *out = A.vt + A.ooff[blk];
            // the staged columns c0 .. c0 + 31 of the block into v~
            auto scatter = [&](int c0) {
                __syncwarp();
                if (vec) {
                    const int col = c0 + (lane & 7) * 4;
#pragma unroll
                    for (int it = 0; it < 8; ++it) {
                        const int row = it * 4 + (lane >> 3);
                        const uint32_t dr = __shfl_sync(0xffffffffu, drow, row);
                        if (row < mine && col < nout)
                            atomicAdd(reinterpret_cast<float4 *>(out + (size_t)dr * A.ostride + col),
                                      *reinterpret_cast<const float4 *>(st + row * PAIR_ST + (lane & 7) * 4));
                    }
                } else {
                    for (int row = 0; row < mine; ++row) {
                        const uint32_t dr = __shfl_sync(0xffffffffu, drow, row);
                        if (c0 + lane < nout)
                            atomicAdd(out + (size_t)dr * A.ostride + c0 + lane, st[row * PAIR_ST + lane]);
                    }
                }
                __syncwarp();
            };
            auto fill_ready = [&] {
                const bool w_ok = mbar_wait(&s_accfull[f & 1], (f >> 1) & 1, A.tries, A.err);
                ok = __all_sync(0xffffffffu, w_ok);
                tc_fence_after();
                return ok;
            };
            auto fill_done = [&] {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&s_accempty[f & 1]);
                ++f;
            };
            if constexpr (SUM) {
                const int cb = warp > 8 ? 64 : 0;  // first column of this warp
                float sum[64];
#pragma unroll
                for (int c = 0; c < 64; ++c) sum[c] = 0.f;
                for (int k0 = 0; k0 < A.nk; k0 += A.part) {
                    if (!fill_ready()) break;
                    const uint32_t d = tmem + (f & 1) * (uint32_t)A.tcols + ((uint32_t)(32 * q) << 16) + (uint32_t)cb;
                    if (mine > 0) {
#pragma unroll
                        for (int c0 = 0; c0 < 64; c0 += 16) {
                            if (cb + c0 < A.npad) {
                                uint32_t v[16], w[16];
                                tmem_ld16(v, d + (uint32_t)c0);
                                tmem_ld16(w, d + (uint32_t)(A.npad + c0));
                                tmem_wait_ld();
#pragma unroll
                                for (int j = 0; j < 16; ++j) sum[c0 + j] += __uint_as_float(v[j]) + __uint_as_float(w[j]);
                            }
                        }
                    }
                    fill_done();
                }
                if (!ok) break;
#pragma unroll
                for (int c0 = 0; c0 < 64; c0 += 32)
                    if (mine > 0 && cb + c0 < nout) {
#pragma unroll
                        for (int k = 0; k < 32; k += 4)
                            *reinterpret_cast<float4 *>(st + lane * PAIR_ST + k) =
                                make_float4(sum[c0 + k] * f1 * f2, sum[c0 + k + 1] * f1 * f2, sum[c0 + k + 2] * f1 * f2,
                                            sum[c0 + k + 3] * f1 * f2);
                        scatter(cb + c0);
                    }
            } else {
                if (!fill_ready()) break;
                const uint32_t d = tmem + (f & 1) * (uint32_t)A.tcols + ((uint32_t)(32 * q) << 16);
                if (mine > 0) {
                    for (int c0 = 0; c0 < nout; c0 += 32) {
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int cc = c0 + 16 * h;
                            if (cc >= A.npad) break;
                            uint32_t v[16], w[16];
                            tmem_ld16(v, d + (uint32_t)cc);
                            if constexpr (STACK) tmem_ld16(w, d + (uint32_t)(A.npad + cc));
                            tmem_wait_ld();
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                float x[4];
#pragma unroll
                                for (int j = 0; j < 4; ++j) {
                                    float y = __uint_as_float(v[4 * k + j]);
                                    if constexpr (STACK) y += __uint_as_float(w[4 * k + j]);
                                    x[j] = y * f1 * f2;
                                }
                                *reinterpret_cast<float4 *>(st + lane * PAIR_ST + 16 * h + 4 * k) =
                                    make_float4(x[0], x[1], x[2], x[3]);
                            }
                        }
                        scatter(c0);
                    }
                }
                fill_done();
            }
        }
    }
    if (!ok) atomicOr(&s_bad, 1);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid == 0 && s_bad) atomicOr(A.err, 1);
    if (warp == 8)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * A.tcols));
}

// Operator images of a Lagrange level.  The scale is common to the level's
// translations: the kernels decay at most as 1/R^2 and the distances of a level's node pairs
// differ by at most a factor of about ten, so every translation keeps its bits.
void build_operator_image(ffm_plan_s *p, int l, const LagGeo &geo, cudaStream_t s) {
    const double *oxy = geo.oxy, dl = geo.dl;
    FarLevel &F = p->far[l];
    const bool cplx = p->kind == FFM_HELMHOLTZ;
    const int r = F.r1 * F.r1 * F.r1, rk = p->kind == FFM_LAPLACE_DL ? 3 * r : r;
    const int rows = cplx ? 2 * r : r, K = cplx ? 2 * rk : rk, ncomp = p->kind == FFM_LAPLACE_GRAD ? 3 : 1;
    // Complex levels: at most 128 rows, so that hi hi has an accumulator of its own (k_lag_pairs, SUM).
    F.h_bpc = cdiv(rows, cplx ? 128 : 256);
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
    switch (F.r1) {
        case 2: launch_op_image<2>(p->kind, g, F.trans_m, geo, F.h_nb, F.h_bpc, F.h_nk, sc, (__half *)F.Th, s); break;
        case 3: launch_op_image<3>(p->kind, g, F.trans_m, geo, F.h_nb, F.h_bpc, F.h_nk, sc, (__half *)F.Th, s); break;
        case 4: launch_op_image<4>(p->kind, g, F.trans_m, geo, F.h_nb, F.h_bpc, F.h_nk, sc, (__half *)F.Th, s); break;
        case 5: launch_op_image<5>(p->kind, g, F.trans_m, geo, F.h_nb, F.h_bpc, F.h_nk, sc, (__half *)F.Th, s); break;
        case 6: launch_op_image<6>(p->kind, g, F.trans_m, geo, F.h_nb, F.h_bpc, F.h_nk, sc, (__half *)F.Th, s); break;
        case 7: launch_op_image<7>(p->kind, g, F.trans_m, geo, F.h_nb, F.h_bpc, F.h_nk, sc, (__half *)F.Th, s); break;
        case 8: launch_op_image<8>(p->kind, g, F.trans_m, geo, F.h_nb, F.h_bpc, F.h_nk, sc, (__half *)F.Th, s); break;
        default: fail(FFM_EUNSUPPORTED, "Chebyshev nodes per axis outside 2..8");
    }
}

// The dynamic shared memory that an instance may use is a property of the function, shared by all threads and
// plans: it is set to the largest size of the instance (operator rows NPAD, translations MAX_TRANS), so
// that no thread lowers it between another's setting and launch.  Per device and cheap: set before every
// launch (plans may live on several devices).
template <int NSTG, int CPS, bool STACK, int NPAD, bool SUM = false>
static void launch_pairs(const PairArgs &A, unsigned grid, cudaStream_t s) {
    FFM_CUDA(cudaFuncSetAttribute(k_lag_pairs<NSTG, CPS, STACK, SUM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)pair_smem(NSTG * CPS, NPAD, MAX_TRANS, SUM)));
    FFM_LAUNCH_NAMED("k_lag_pairs", (k_lag_pairs<NSTG, CPS, STACK, SUM>), grid, SUM ? PAIR_TS : PAIR_T,
                     pair_smem(NSTG * CPS, A.npad, A.n_trans, SUM), s, A);
}

// v~ += T u~ for all pairs of the level: u has rows of K floats per (source box, right-hand side),
// v~ rows of `rows` floats per (target box, right-hand side) and component
void lag_pairs(const ffm_plan_s *p, int l, const float *u, int nrhs, float *vt, Alloc &tmp, cudaStream_t s) {
    const FarLevel &F = p->far[l];
    if (!F.bt_off) fail(FFM_ECUDA, "transfer by translation on a level without grouped pairs");
    const bool cplx = p->kind == FFM_HELMHOLTZ;
    const int r = F.r1 * F.r1 * F.r1, rk = p->kind == FFM_LAPLACE_DL ? 3 * r : r;
    const int rows = cplx ? 2 * r : r, K = cplx ? 2 * rk : rk, ncomp = p->kind == FFM_LAPLACE_GRAD ? 3 : 1;
    const int64_t nrow = (int64_t)p->by[l].nb * nrhs;
    PairArgs A{};
    __half *img = tmp.get<__half>((size_t)nrow * F.h_nk * HROW);
    float *inv = tmp.get<float>(nrow);
    FFM_LAUNCH(k_rows_split, cdiv(nrow, 8), 256, 0, s, u, nrow, K, F.h_nk, img, inv, (const uint32_t *)nullptr, nrhs);
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
    A.part = cplx ? PAIR_PART : F.h_nk;
    A.npad = F.h_nb;
    const bool stack = A.npad <= 128;
    A.tcols = 32;
    while (A.tcols < (stack ? 2 : 1) * A.npad) A.tcols <<= 1;
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
    // stages of two chunks where the K extent allows: half the barrier round trips
    if (cplx)
        launch_pairs<5, 1, true, 128, true>(A, grid, s);
    else if (A.npad <= 64 && A.nk % 2 == 0)
        launch_pairs<4, 2, true, 64>(A, grid, s);
    else if (A.npad <= 64)
        launch_pairs<8, 1, true, 64>(A, grid, s);
    else if (stack)
        launch_pairs<6, 1, true, 128>(A, grid, s);
    else
        launch_pairs<4, 1, false, 256>(A, grid, s);
    tmp.drop(inv);
    tmp.drop(img);
}

// ---- target-stationary transfer (real operators, r <= 64)
//
// For levels whose targets have many partners (volumes: 290-360 of 665 translations).  A block owns
// TG_M = 128 consecutive target boxes (TMEM lane = box) and runs over the level's translations; the
// products accumulate and each target's v~ is written once: no adds to memory, no grouping of the
// pairs, and no pair lists at all.  The source box of a target at a translation is found from its
// parent's near table (k_near_table): the near source boxes of the parent level by their offset (at
// most 4 per axis), each with its first child and the mask of its children's octants.
//
// What bounds it: the gathered rows' and the operators' way from L2 (48 KB a step at most).  A step is
// one translation: warps 9-12 look up the step's 128 sources in turn and leave them in a shared ring, so
// that no copying thread waits for a lookup; warps 0-3 copy the source rows (hi and lo images,
// 16-byte cp.async segments, rows without a partner zero-filled without a read), thread 0 starts
// the bulk copy of T_t's image, warp 8 issues hi [hi; lo] (N = 2 npad) and lo hi, 4 steps in flight (8
// where K <= 32).  Nothing is converted on the way.
// Rows of different sources meet in one accumulator, so all rows of a right-hand side share one scale
// (k_level_max; a block works on one right-hand side, and the others have scales of their own): a
// value keeps its 22 bits down to 2^-15 of its column's largest, and below that an absolute error of 2^-38
// of it, which is lost beside that source's own potential at every target.
//
// One long tensor-core accumulation loses accuracy, so the block alternates between two TMEM
// accumulators every TG_DRAIN translations; warps 4-7 add each finished one into FP32 registers
// while the other fills.  Every wait is bounded as in k_lag_pairs.
//
// Measured on GB300, level 7 of clustered 10M (193k targets, 68M pairs): 3.52 ms, 0.53 us a step
// (the kernel before it, FP32 rows split into TF32 by the copying warps: 7.9 ms).  Lists of the
// pairs by tile and translation instead of the near tables cost 64 ms of plan at 1e8 points.
constexpr int TG_M = 128;
constexpr int TG_DRAIN = 8;        // translations per accumulator fill
constexpr int TG_T = 416;
constexpr int TG_IX = 8;           // steps whose sources are held

// octants of each box's children, one bit each (children are in octant order)
__global__ void k_child_masks(const uint32_t *__restrict__ first_child, const int4 *__restrict__ gc, int64_t n,
                              uint8_t *__restrict__ mask) {
    const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= n) return;
    uint32_t m = 0;
    for (uint32_t c = first_child[b]; c < first_child[b + 1]; ++c) {
        const int4 g = gc[c];
        m |= 1u << ((g.x & 1) << 2 | (g.y & 1) << 1 | (g.z & 1));
    }
    mask[b] = (uint8_t)m;
}

// Near table of every target box of a level, one warp per box: entry (kx, ky, kz) - base of the offset
// k = g_X - g_Y of a near source box holds its first child and child mask (mask 0: no such box).
__global__ void __launch_bounds__(256) k_near_table(int64_t n, const uint32_t *__restrict__ off,
                                                    const uint32_t *__restrict__ src, const int4 *__restrict__ gx,
                                                    const int4 *__restrict__ gy, const uint32_t *__restrict__ fcy,
                                                    const uint8_t *__restrict__ mask, int3 base, int *__restrict__ err,
                                                    uint2 *__restrict__ table) {
    const int64_t a = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (a >= n) return;
    uint2 *t = table + a * 64;
    t[lane] = t[32 + lane] = make_uint2(0u, 0u);
    __syncwarp();
    const int4 p = gx[a];
    for (uint32_t e = off[a] + lane; e < off[a + 1]; e += 32) {
        const uint32_t b = src[e];
        const int4 q = gy[b];
        const unsigned kx = p.x - q.x - base.x, ky = p.y - q.y - base.y, kz = p.z - q.z - base.z;
        if (kx < 4u && ky < 4u && kz < 4u)
            t[(kx * 4 + ky) * 4 + kz] = make_uint2(fcy[b], mask[b]);
        else
            atomicOr(err, 1);  // not possible: |sigma + k| < 2 holds for at most four integers k
    }
}

// The target-stationary transfer of a Lagrange level made possible (ts_ok), where the plan's rule, the
// option, the autotuner or its cache asks for it.
void prepare_target_stationary(ffm_plan_s *p, int l, cudaStream_t s) {
    FarLevel &F = p->far[l];
    if (F.mode != 1 || F.n_adm == 0 || F.ts_ok || !F.Th || p->kind != FFM_LAPLACE || F.r1 > 4 || l == 0 || !p->nr_off[l - 1])
        return;
    const int64_t nx = p->bx[l - 1].nb, ny = p->by[l - 1].nb;
    Alloc tmp;
    tmp.stream = s;
    uint8_t *mask = tmp.get<uint8_t>(ny);
    FFM_LAUNCH(k_child_masks, cdiv(ny, 256), 256, 0, s, p->by[l - 1].first_child, p->by[l].g, ny, mask);
    F.ts_near = p->mem.get<uint2>(nx * 64);
    FFM_LAUNCH(k_near_table, cdiv(nx, 8), 256, 0, s, nx, p->nr_off[l - 1], p->nr_src[l - 1], p->bx[l - 1].g, p->by[l - 1].g,
               p->by[l - 1].first_child, mask, near_base(p, l - 1), p->dev_err, F.ts_near);
    F.ts_ok = true;
}

// largest |u| of right-hand side blockIdx.y over the level's nb rows of r values, as float bits (0 for an all-zero
// column)
__global__ void k_level_max(const float *__restrict__ u, int64_t nb, int r, int nrhs, uint32_t *__restrict__ out) {
    const int m = blockIdx.y;
    const int64_t n = nb * r;
    float mx = 0.f;
    if (nrhs == 1) {
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
            mx = fmaxf(mx, fabsf(u[i]));
    } else {  // one row per warp and turn
        const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
        for (int64_t b = (int64_t)blockIdx.x * nw + (threadIdx.x >> 5); b < nb; b += (int64_t)gridDim.x * nw)
            for (int k = lane; k < r; k += 32) mx = fmaxf(mx, fabsf(u[(b * nrhs + m) * r + k]));
    }
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0 && mx > 0.f) atomicMax(out + m, __float_as_uint(mx));
}

struct TargetArgs {
    const uint32_t *tgt, *parent;
    const int4 *g, *trans;  // coordinates of the target boxes, translations
    const uint2 *near;      // near tables of the parents
    int3 base;
    int64_t n_tgt;
    int n_trans, nrhs, nk, npad, r, tcols;
    const __half *u;        // row images of (source box, right-hand side), one scale per right-hand side
    const uint32_t *umax;   // the scales' values (k_level_max)
    const __half *T;
    float tinv;
    float *vt;
    int *err;
    int tries;
};

template <int NSTG, int CPS>
__global__ void __launch_bounds__(TG_T, 1) k_lag_targets(const __grid_constant__ TargetArgs A) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = aligned_smem(smem_raw);
    __shared__ __align__(8) uint64_t s_full[NSTG], s_empty[NSTG], s_accfull[2], s_accempty[2], s_done;
    __shared__ __align__(8) uint64_t s_ixfull[TG_IX], s_ixempty[TG_IX];
    __shared__ uint32_t s_src[TG_IX][TG_M];  // the step's source box by row, NONE without a partner
    __shared__ uint32_t s_tmem, s_cmax;
    __shared__ int s_bad;
    constexpr uint32_t NONE = 0xffffffffu;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m = blockIdx.y;
    const int64_t x0 = (int64_t)blockIdx.x * TG_M;
    const uint32_t bbytes = (uint32_t)A.npad * HROW * 2 * CPS, stage = CPS * A_BYTES + bbytes;
    if (warp == 8) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&s_tmem)),
                     "r"(2 * A.tcols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        s_bad = 0;
        s_cmax = 0;
        for (int i = 0; i < NSTG; ++i) {
            mbar_init(&s_full[i], 129);  // the copying threads, and the operator copy's byte count
            mbar_init(&s_empty[i], 1);
        }
        for (int i = 0; i < TG_IX; ++i) {
            mbar_init(&s_ixfull[i], 1);
            mbar_init(&s_ixempty[i], 4);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&s_accfull[i], 1);
            mbar_init(&s_accempty[i], 4);
        }
        mbar_init(&s_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    const uint32_t nsteps = (uint32_t)A.n_trans;
    bool ok = true;
    if (warp > 8) {
        // ---- sources: warp w looks up steps w - 9, w - 9 + 4, ...; lane: rows lane, lane + 32, ...
        int4 g[4];
        const uint2 *near[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int64_t x = x0 + 32 * k + lane;
            near[k] = nullptr;
            if (x < A.n_tgt) {
                const uint32_t box = A.tgt[x];
                g[k] = A.g[box];
                near[k] = A.near + (size_t)A.parent[box] * 64;
            }
        }
        for (uint32_t s = warp - 9; s < nsteps; s += 4) {
            const uint32_t ix = s % TG_IX;
            const int4 m4 = A.trans[s];
            uint2 e[4];
            uint32_t oct[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                e[k] = make_uint2(0u, 0u);
                oct[k] = 0;
                if (near[k]) {
                    const int qx = g[k].x - m4.x, qy = g[k].y - m4.y, qz = g[k].z - m4.z;
                    const unsigned kx = (g[k].x >> 1) - (qx >> 1) - A.base.x, ky = (g[k].y >> 1) - (qy >> 1) - A.base.y,
                                   kz = (g[k].z >> 1) - (qz >> 1) - A.base.z;
                    oct[k] = (qx & 1) << 2 | (qy & 1) << 1 | (qz & 1);
                    if (kx < 4u && ky < 4u && kz < 4u) e[k] = __ldg(near[k] + (kx * 4 + ky) * 4 + kz);
                }
            }
            const bool w_ok = s < TG_IX || mbar_wait(&s_ixempty[ix], ((s / TG_IX) - 1) & 1, A.tries, A.err);
            if (!__all_sync(0xffffffffu, w_ok)) {
                ok = false;
                break;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
                s_src[ix][32 * k + lane] =
                    (e[k].y >> oct[k] & 1u) ? e[k].x + __popc(e[k].y & ((1u << oct[k]) - 1u)) : NONE;
            __syncwarp();
            if (lane == 0) mbar_arrive(&s_ixfull[ix]);
        }
    } else if (warp < 4) {
        // ---- copies: lane handles 16-byte segment lane % 8 of rows 32 warp + 4 g + lane / 8 (g < 8)
        const uint32_t r0 = 32 * warp + (lane >> 3), sg = lane & 7;
        const uint32_t dst0 = smem_addr(smem) + r0 * 128, sw0 = (sg ^ (r0 & 7)) * 16, sw1 = (sg ^ ((r0 + 4) & 7)) * 16;
        uint32_t c = 0;
        for (uint32_t s = 0; s < nsteps && ok; ++s) {
            const uint32_t ix = s % TG_IX;
            const bool i_ok = mbar_wait(&s_ixfull[ix], (s / TG_IX) & 1, A.tries, A.err);
            if (!__all_sync(0xffffffffu, i_ok)) {
                ok = false;
                break;
            }
            const __half *p[8];
            uint32_t n[8];
#pragma unroll
            for (int g = 0; g < 8; ++g) {
                const uint32_t sb = s_src[ix][r0 + 4 * g];
                n[g] = sb != NONE ? 16u : 0u;
                p[g] = A.u + ((size_t)(sb != NONE ? sb : 0u) * A.nrhs + m) * (CPS * HROW) + sg * 8;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&s_ixempty[ix]);
            const uint32_t slot = c % NSTG;
            const bool w_ok = c < NSTG || mbar_wait(&s_empty[slot], ((c / NSTG) - 1) & 1, A.tries, A.err);
            if (!__all_sync(0xffffffffu, w_ok)) {
                ok = false;
                break;
            }
            if (tid == 0) {
                mbar_expect(&s_full[slot], bbytes);
                bulk_g2s(smem + (size_t)slot * stage + CPS * A_BYTES, A.T + (size_t)s * CPS * A.npad * HROW, bbytes,
                         &s_full[slot]);
            }
            const uint32_t dst = dst0 + slot * stage;
#pragma unroll
            for (int g = 0; g < 8; ++g)
#pragma unroll
                for (int j = 0; j < CPS; ++j)
                    cp_async16_zfill(dst + j * A_BYTES + g * 512 + ((g & 1) ? sw1 : sw0), p[g] + j * HROW, n[g]);
            cp_async_arrive(&s_full[slot]);
            ++c;
        }
        // After a give-up some warps may have copied further than others: all arrive on every stage any of
        // them started, so that the operator copies can be waited for.
        if (!ok) atomicOr(&s_bad, 1);
        asm volatile("cp.async.wait_all;" ::: "memory");
        atomicMax(&s_cmax, c);
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (s_bad) {
            const uint32_t last = *reinterpret_cast<volatile uint32_t *>(&s_cmax);
            for (; c < last; ++c) {
                if (tid == 0) mbar_arrive(&s_full[c % NSTG]);
                mbar_arrive(&s_full[c % NSTG]);
            }
        }
        if (tid == 0)
            for (uint32_t d = c > NSTG ? c - NSTG : 0; d < c; ++d)
                mbar_wait(&s_full[d % NSTG], (d / NSTG) & 1, DRAIN_TRIES);
    } else if (warp == 8) {
        if (lane == 0) {
            // ---- MMA thread
            const uint32_t id1 = idesc_f16(A.npad), id2 = idesc_f16(2 * A.npad);
            const uint32_t alo = a_dlo(smem_addr(smem)), blo = b_dlo(smem_addr(smem) + CPS * A_BYTES);
            uint32_t slot = 0, par = 0;
            for (uint32_t s = 0; s < nsteps; ++s) {
                const uint32_t fill = s / TG_DRAIN, buf = fill & 1;
                if (s % TG_DRAIN == 0 && fill >= 2 &&
                    !mbar_wait(&s_accempty[buf], ((fill >> 1) - 1) & 1, A.tries, A.err)) {
                    ok = false;
                    break;
                }
                if (!mbar_wait(&s_full[slot], par, A.tries, A.err)) {
                    ok = false;
                    break;
                }
                fence_proxy_async();  // the rows came by cp.async, through the generic proxy
                tc_fence_after();
                const uint32_t off = slot * (stage >> 4);
                stage_mma<CPS, true>(tmem + buf * (uint32_t)A.tcols, alo + off, blo + off, (uint32_t)A.npad, id1, id2,
                                     s % TG_DRAIN == 0);
                tc_commit(&s_empty[slot]);
                if (s % TG_DRAIN == TG_DRAIN - 1 || s + 1 == nsteps) tc_commit(&s_accfull[buf]);
                if (++slot == NSTG) {
                    slot = 0;
                    par ^= 1;
                }
            }
            // everything issued is done before the block gives up its shared memory and TMEM
            tc_commit(&s_done);
            mbar_wait(&s_done, 0, DRAIN_TRIES);
        }
    } else {
        // ---- sums: warp w holds lanes 32 (w - 4) .. + 31
        const int q = warp - 4;
        float sum[64];
#pragma unroll
        for (int c = 0; c < 64; ++c) sum[c] = 0.f;
        const uint32_t fills = (nsteps + TG_DRAIN - 1) / TG_DRAIN;
        for (uint32_t f = 0; f < fills; ++f) {
            const uint32_t buf = f & 1;
            const bool w_ok = mbar_wait(&s_accfull[buf], (f >> 1) & 1, A.tries, A.err);
            if (!__all_sync(0xffffffffu, w_ok)) {
                ok = false;
                break;
            }
            tc_fence_after();
            const uint32_t d = tmem + buf * (uint32_t)A.tcols + ((uint32_t)(32 * q) << 16);
#pragma unroll
            for (int c0 = 0; c0 < 64; c0 += 16) {
                if (c0 < A.npad) {
                    uint32_t v[16], w[16];
                    tmem_ld16(v, d + (uint32_t)c0);
                    tmem_ld16(w, d + (uint32_t)(A.npad + c0));
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 16; ++j) sum[c0 + j] += __uint_as_float(v[j]) + __uint_as_float(w[j]);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&s_accempty[buf]);
        }
        const int64_t x = x0 + 32 * q + lane;
        if (ok && x < A.n_tgt) {
            float us, ui, f1, f2;
            row_scale(__uint_as_float(A.umax[m]), us, ui);
            even_factors(ui, A.tinv, f1, f2);
            float *dst = A.vt + ((size_t)A.tgt[x] * A.nrhs + m) * A.r;
#pragma unroll
            for (int c = 0; c < 64; ++c) sum[c] = sum[c] * f1 * f2;
            if (A.r == 64) {
#pragma unroll
                for (int c = 0; c < 64; c += 4)
                    *reinterpret_cast<float4 *>(dst + c) = make_float4(sum[c], sum[c + 1], sum[c + 2], sum[c + 3]);
            } else {
#pragma unroll
                for (int c = 0; c < 64; ++c)
                    if (c < A.r) dst[c] = sum[c];
            }
        }
    }
    if (!ok) atomicOr(&s_bad, 1);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid == 0 && s_bad) atomicOr(A.err, 1);
    if (warp == 8)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * A.tcols));
}

static size_t target_smem(int nchunk, int npad) { return 1024 + (size_t)nchunk * (A_BYTES + npad * HROW * 2); }

// (the attribute as in launch_pairs: the instance's largest size, 64 operator rows)
template <int NSTG, int CPS>
static void launch_targets(const TargetArgs &A, dim3 grid, cudaStream_t s) {
    FFM_CUDA(cudaFuncSetAttribute(k_lag_targets<NSTG, CPS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)target_smem(NSTG * CPS, 64)));
    FFM_LAUNCH_NAMED("k_lag_targets", (k_lag_targets<NSTG, CPS>), grid, TG_T, target_smem(NSTG * CPS, A.npad), s, A);
}

// v~ = sum over each target's partners of T u~ (rows of targets without partners untouched)
void lag_targets(const ffm_plan_s *p, int l, const float *u, int nrhs, float *vt, Alloc &tmp, cudaStream_t s) {
    const FarLevel &F = p->far[l];
    const int r = F.r1 * F.r1 * F.r1;
    const int64_t nrow = (int64_t)p->by[l].nb * nrhs;
    TargetArgs A{};
    __half *img = tmp.get<__half>((size_t)nrow * F.h_nk * HROW);
    uint32_t *mx = tmp.get<uint32_t>(nrhs);
    FFM_CUDA(cudaMemsetAsync(mx, 0, sizeof(uint32_t) * nrhs, s));
    const int64_t nb = p->by[l].nb;
    const dim3 gm((unsigned)std::min<int64_t>(cdiv(nb * r, 1024), std::max(1, 152 * 8 / nrhs)), nrhs);
    FFM_LAUNCH(k_level_max, gm, 256, 0, s, u, nb, r, nrhs, mx);
    FFM_LAUNCH(k_rows_split, cdiv(nrow, 8), 256, 0, s, u, nrow, r, F.h_nk, img, (float *)nullptr, (const uint32_t *)mx, nrhs);
    A.tgt = F.tgt;
    A.parent = p->parent[l];
    A.g = p->bx[l].g;
    A.trans = F.trans_m;
    A.near = F.ts_near;
    A.base = near_base(p, l - 1);
    A.n_trans = F.n_trans;
    A.n_tgt = F.n_tgt;
    A.nrhs = nrhs;
    A.nk = F.h_nk;
    A.npad = F.h_nb;
    A.r = r;
    A.tcols = 32;
    while (A.tcols < 2 * A.npad) A.tcols <<= 1;
    A.u = img;
    A.umax = mx;
    A.T = (const __half *)F.Th;
    A.tinv = F.h_inv;
    A.vt = vt;
    A.err = p->dev_err;
    A.tries = p->wait_tries;
    const dim3 grid(cdiv(F.n_tgt, TG_M), nrhs);
    if (A.nk == 2)
        launch_targets<4, 2>(A, grid, s);
    else  // r <= 27
        launch_targets<8, 1>(A, grid, s);
    tmp.drop(mx);
    tmp.drop(img);
}

}  // namespace ffm
