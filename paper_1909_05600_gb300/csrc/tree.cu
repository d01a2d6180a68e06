// Plan construction on the device (Sec. 2.2.1, 2.2.2, 2.2.4 and Sec. 3.1):
//   bounding cubes of equal edge, Morton keys, stable radix sort, per-level box tables,
//   and the descent-only pair lists (children of near pairs split into admissible and
//   near pairs), grouped by target box and keyed by integer box translation.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "ffm_internal.cuh"

namespace ffm {

// ==================================================================== scan

constexpr int SCAN_T = 512;
constexpr int SCAN_IPT = 8;
constexpr int SCAN_TILE = SCAN_T * SCAN_IPT;

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v) {
    int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// Block-wide exclusive scan of one value per thread; returns the block total in *tot.
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t *sm_warp, uint32_t *tot) {
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    uint32_t inc = warp_incl_scan(v);
    if (lane == 31) sm_warp[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < nw ? sm_warp[lane] : 0;
        uint32_t wi = warp_incl_scan(w);
        if (lane < nw) sm_warp[lane] = wi - w;
        if (lane == nw - 1) *tot = wi;
    }
    __syncthreads();
    return inc - v + sm_warp[warp];
}

__global__ void k_scan_reduce(const uint32_t *__restrict__ in, int64_t n, uint32_t *__restrict__ bsum) {
    int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
    uint32_t s = 0;
    for (int i = threadIdx.x; i < SCAN_TILE; i += SCAN_T) {
        int64_t g = base + i;
        if (g < n) s += in[g];
    }
    __shared__ uint32_t sw[32];
    __shared__ uint32_t tot;
    block_excl_scan(s, sw, &tot);
    if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

__global__ void k_scan_bsums(uint32_t *bsum, int64_t nb, uint32_t *d_total) {
    __shared__ uint32_t sw[32];
    __shared__ uint32_t tot;
    uint32_t carry = 0;
    for (int64_t c = 0; c < nb; c += blockDim.x) {
        int64_t i = c + threadIdx.x;
        uint32_t v = i < nb ? bsum[i] : 0;
        uint32_t e = block_excl_scan(v, sw, &tot);
        if (i < nb) bsum[i] = e + carry;
        carry += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0 && d_total) *d_total = carry;
}

__global__ void k_scan_down(const uint32_t *in, uint32_t *out, int64_t n, const uint32_t *__restrict__ bsum) {
    __shared__ uint32_t tile[SCAN_TILE];
    __shared__ uint32_t sw[32];
    __shared__ uint32_t tot;
    int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
    for (int i = threadIdx.x; i < SCAN_TILE; i += SCAN_T) {
        int64_t g = base + i;
        tile[i] = g < n ? in[g] : 0;
    }
    __syncthreads();
    uint32_t loc[SCAN_IPT];
    uint32_t s = 0;
#pragma unroll
    for (int j = 0; j < SCAN_IPT; ++j) {
        loc[j] = s;
        s += tile[threadIdx.x * SCAN_IPT + j];
    }
    uint32_t e = block_excl_scan(s, sw, &tot) + bsum[blockIdx.x];
#pragma unroll
    for (int j = 0; j < SCAN_IPT; ++j) tile[threadIdx.x * SCAN_IPT + j] = loc[j] + e;
    __syncthreads();
    for (int i = threadIdx.x; i < SCAN_TILE; i += SCAN_T) {
        int64_t g = base + i;
        if (g < n) out[g] = tile[i];
    }
}

// The whole scan in one block, tile after tile with a running carry: one launch instead
// of three for the small scans of a plan.  A tile takes about 1.3 us in one block, the three
// launches about 8 us together, so up to six tiles.
constexpr int64_t SCAN_SMALL = 6 * SCAN_TILE;
__global__ void __launch_bounds__(SCAN_T) k_scan_small(const uint32_t *in, uint32_t *out, int64_t n,
                                                       uint32_t *d_total) {
    __shared__ uint32_t tile[SCAN_TILE];
    __shared__ uint32_t sw[32];
    __shared__ uint32_t tot;
    uint32_t carry = 0;
    for (int64_t base = 0; base < n; base += SCAN_TILE) {
        for (int i = threadIdx.x; i < SCAN_TILE; i += SCAN_T) {
            int64_t g = base + i;
            tile[i] = g < n ? in[g] : 0;
        }
        __syncthreads();
        uint32_t loc[SCAN_IPT];
        uint32_t sum = 0;
#pragma unroll
        for (int j = 0; j < SCAN_IPT; ++j) {
            loc[j] = sum;
            sum += tile[threadIdx.x * SCAN_IPT + j];
        }
        uint32_t e = block_excl_scan(sum, sw, &tot) + carry;
#pragma unroll
        for (int j = 0; j < SCAN_IPT; ++j) tile[threadIdx.x * SCAN_IPT + j] = loc[j] + e;
        __syncthreads();
        for (int i = threadIdx.x; i < SCAN_TILE; i += SCAN_T) {
            int64_t g = base + i;
            if (g < n) out[g] = tile[i];
        }
        carry += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0 && d_total) *d_total = carry;
}

void scan_u32(const uint32_t *in, uint32_t *out, int64_t n, uint32_t *d_total, Alloc &al, cudaStream_t s) {
    if (n <= 0) {
        if (d_total) FFM_CUDA(cudaMemsetAsync(d_total, 0, sizeof(uint32_t), s));
        return;
    }
    if (n <= SCAN_SMALL) {
        FFM_LAUNCH(k_scan_small, 1, SCAN_T, 0, s, in, out, n, d_total);
        return;
    }
    int64_t nb = cdiv(n, SCAN_TILE);
    uint32_t *bsum = al.get<uint32_t>(nb);
    FFM_LAUNCH(k_scan_reduce, (unsigned)nb, SCAN_T, 0, s, in, n, bsum);
    FFM_LAUNCH(k_scan_bsums, 1, 1024, 0, s, bsum, nb, d_total);
    FFM_LAUNCH(k_scan_down, (unsigned)nb, SCAN_T, 0, s, in, out, n, bsum);
}

// ============================================================== radix sort

constexpr int RS_T = 256;
constexpr int RS_ITEMS = 16;
constexpr int RS_TILE = RS_T * RS_ITEMS;

template <class K>
__global__ void k_rs_bits(const K *__restrict__ k, int64_t n, unsigned long long *orand) {
    unsigned long long o = 0, a = ~0ull;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        unsigned long long v = (unsigned long long)k[i];
        o |= v;
        a &= v;
    }
    for (int off = 16; off; off >>= 1) {
        o |= __shfl_xor_sync(0xffffffffu, o, off);
        a &= __shfl_xor_sync(0xffffffffu, a, off);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicOr(&orand[0], o);
        atomicAnd(&orand[1], a);
    }
}

template <class K>
__global__ void k_rs_hist(const K *__restrict__ kin, int64_t n, int shift, uint32_t *__restrict__ hist, int nblk) {
    __shared__ uint32_t c[256];
    c[threadIdx.x] = 0;
    __syncthreads();
    int64_t t0 = (int64_t)blockIdx.x * RS_TILE;
    for (int r = 0; r < RS_ITEMS; ++r) {
        int64_t i = t0 + r * RS_T + threadIdx.x;
        if (i < n) atomicAdd(&c[(uint32_t)(kin[i] >> shift) & 255u], 1u);
    }
    __syncthreads();
    hist[(int64_t)threadIdx.x * nblk + blockIdx.x] = c[threadIdx.x];
}

__device__ __forceinline__ unsigned long long ld_stream(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.volatile.global.u64 %0, [%1];" : "=l"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t ld_stream(const uint32_t *p) {
    uint32_t v;
    asm volatile("ld.volatile.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}

// Stable scatter staged in shared memory.  A block owns a tile of RS_TILE elements; warp w
// takes the tile's elements w RS_ITEMS 32 .. in order, 32 per round.  Each element's rank
// within its warp's digit run comes from a warp match mask and a warp-private count per
// digit (no block barrier per round); the warps' counts are then turned into offsets within
// the tile's digit runs (in element order: warps in turn), and each element is placed in a
// shared-memory copy of the tile, which ends up sorted by digit.  The block then writes that
// copy in order: consecutive threads write consecutive slots of one digit's run in the
// output (its start from the scanned digit-major histogram), so the stores are coalesced.
// The tile's own digit counts are differences of consecutive entries of the scanned
// histogram.
template <class K>
__global__ void __launch_bounds__(RS_T) k_rs_scatter(const K *__restrict__ kin, const uint32_t *__restrict__ vin,
                                                     int64_t n, int shift, const uint32_t *__restrict__ off,
                                                     int nblk, K *__restrict__ kout, uint32_t *__restrict__ vout) {
    extern __shared__ __align__(16) unsigned char rs_smem[];
    K *skey = reinterpret_cast<K *>(rs_smem);
    uint32_t *sval = reinterpret_cast<uint32_t *>(skey + RS_TILE);
    __shared__ uint32_t base[256], start[256];
    __shared__ uint32_t wc[RS_T / 32][256];  // per warp and digit: counts, then offsets in the tile
    __shared__ uint32_t wtot[RS_T / 32];
    int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t t0 = (int64_t)blockIdx.x * RS_TILE;
    const int tile_n = (int)min((int64_t)RS_TILE, n - t0);
#pragma unroll
    for (int d = 0; d < 256; d += 32) wc[warp][d + lane] = 0u;
    {
        const int64_t flat = (int64_t)tid * nblk + blockIdx.x;
        const uint32_t b = off[flat];
        const uint32_t c = flat + 1 < 256LL * nblk ? off[flat + 1] - b : (uint32_t)(n - b);
        base[tid] = b;
        // exclusive prefix of the tile's digit counts (digit = thread)
        uint32_t inc = c;
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        if (lane == 31) wtot[warp] = inc;
        __syncthreads();
        uint32_t before = 0;
        for (int w = 0; w < warp; ++w) before += wtot[w];
        start[tid] = before + inc - c;
    }
    // warp-local stable ranks, RS_ITEMS rounds of 32 consecutive elements; every load of the
    // warp is issued first (volatile, so the compiler keeps them here, all in flight)
    K keys[RS_ITEMS];
    uint32_t vals[RS_ITEMS], rk[RS_ITEMS], dg[RS_ITEMS];
    const int64_t w0 = t0 + (int64_t)warp * RS_ITEMS * 32;
#pragma unroll
    for (int r = 0; r < RS_ITEMS; ++r) {
        const int64_t i = w0 + r * 32 + lane;
        keys[r] = (K)0;
        vals[r] = 0u;
        if (i < n) {
            keys[r] = ld_stream(kin + i);
            vals[r] = ld_stream(vin + i);
        }
    }
#pragma unroll
    for (int r = 0; r < RS_ITEMS; ++r) {
        const int64_t i = w0 + r * 32 + lane;
        const bool valid = i < n;
        const uint32_t d = valid ? ((uint32_t)(keys[r] >> shift) & 255u) : 256u;
        dg[r] = d;
        const uint32_t peers = __match_any_sync(0xffffffffu, d);
        const uint32_t lt = peers & ((1u << lane) - 1u);
        rk[r] = valid ? wc[warp][d] + __popc(lt) : 0u;
        __syncwarp();
        if (valid && lt == 0) wc[warp][d] += __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    {
        // digit tid: the warps' runs in turn, after the runs of the smaller digits
        uint32_t o = start[tid];
#pragma unroll
        for (int w = 0; w < RS_T / 32; ++w) {
            const uint32_t c = wc[w][tid];
            wc[w][tid] = o;
            o += c;
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RS_ITEMS; ++r)
        if (dg[r] < 256u) {
            const uint32_t pos = wc[warp][dg[r]] + rk[r];
            skey[pos] = keys[r];
            sval[pos] = vals[r];
        }
    __syncthreads();
    for (int i = tid; i < tile_n; i += RS_T) {
        K key = skey[i];
        uint32_t d = (uint32_t)(key >> shift) & 255u;
        uint32_t gp = base[d] + (uint32_t)i - start[d];
        kout[gp] = key;
        vout[gp] = sval[i];
    }
}

template <class K>
static void radix_sort(K *keys, uint32_t *vals, int64_t n, int nbits, Alloc &al, cudaStream_t s) {
    if (n <= 1) return;
    unsigned long long *orand = al.get<unsigned long long>(2);
    unsigned long long init[2] = {0ull, ~0ull};
    FFM_CUDA(cudaMemcpyAsync(orand, init, sizeof init, cudaMemcpyHostToDevice, s));
    FFM_LAUNCH(k_rs_bits<K>, std::min<unsigned>(cdiv(n, 256), 1024u), 256, 0, s, keys, n, orand);
    unsigned long long h[2];
    FFM_CUDA(cudaMemcpyAsync(h, orand, sizeof h, cudaMemcpyDeviceToHost, s));
    FFM_CUDA(cudaStreamSynchronize(s));
    unsigned long long vary = h[0] ^ h[1];
    int nblk = (int)cdiv(n, RS_TILE);
    uint32_t *hist = al.get<uint32_t>((size_t)256 * nblk);
    K *k2 = al.get<K>(n);
    uint32_t *v2 = al.get<uint32_t>(n);
    K *ka = keys, *kb = k2;
    uint32_t *va = vals, *vb = v2;
    const size_t scatter_smem = (size_t)RS_TILE * (sizeof(K) + sizeof(uint32_t));
    FFM_CUDA(cudaFuncSetAttribute(k_rs_scatter<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)scatter_smem));
    for (int shift = 0; shift < nbits; shift += 8) {
        if (((vary >> shift) & 255ull) == 0) continue;
        FFM_LAUNCH(k_rs_hist<K>, nblk, RS_T, 0, s, ka, n, shift, hist, nblk);
        scan_u32(hist, hist, (int64_t)256 * nblk, nullptr, al, s);
        FFM_LAUNCH(k_rs_scatter<K>, nblk, RS_T, scatter_smem, s, ka, va, n, shift, hist, nblk, kb, vb);
        std::swap(ka, kb);
        std::swap(va, vb);
    }
    if (ka != keys) {
        FFM_CUDA(cudaMemcpyAsync(keys, ka, sizeof(K) * n, cudaMemcpyDeviceToDevice, s));
        FFM_CUDA(cudaMemcpyAsync(vals, va, sizeof(uint32_t) * n, cudaMemcpyDeviceToDevice, s));
    }
}

void radix_sort_u64(uint64_t *keys, uint32_t *vals, int64_t n, int nbits, Alloc &al, cudaStream_t s) {
    radix_sort<unsigned long long>((unsigned long long *)keys, vals, n, nbits, al, s);
}

// ========================================================== bounding cubes

__device__ __forceinline__ unsigned long long ord_enc(double d) {
    unsigned long long u = (unsigned long long)__double_as_longlong(d);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}
static double ord_dec(unsigned long long k) {
    unsigned long long u = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
    double d;
    memcpy(&d, &u, sizeof d);
    return d;
}

// out[0..2] = encoded min, out[3..5] = encoded max, out[6] = non-finite flag.  Minima and maxima in
// the points' own type (this part's FP64 rate is a small fraction of its FP32 rate), reduced over the
// block first: one atomic per block and bound on the seven words (one per warp took 44 us at 250k points).
template <class T>
__global__ void __launch_bounds__(256) k_bbox(const T *__restrict__ P, int64_t n, unsigned long long *out) {
    T lo[3] = {(T)INFINITY, (T)INFINITY, (T)INFINITY}, hi[3] = {-(T)INFINITY, -(T)INFINITY, -(T)INFINITY};
    bool bad = false;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const T x = P[3 * i + d];
            bad |= !isfinite(x);
            lo[d] = x < lo[d] ? x : lo[d];
            hi[d] = x > hi[d] ? x : hi[d];
        }
    }
    __shared__ T s[6][8];
    __shared__ int sbad;
    if (threadIdx.x == 0) sbad = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        for (int off = 16; off; off >>= 1) {
            const T a = __shfl_xor_sync(0xffffffffu, lo[d], off), c = __shfl_xor_sync(0xffffffffu, hi[d], off);
            lo[d] = a < lo[d] ? a : lo[d];
            hi[d] = c > hi[d] ? c : hi[d];
        }
        if (lane == 0) {
            s[d][warp] = lo[d];
            s[3 + d][warp] = hi[d];
        }
    }
    if (bad) sbad = 1;
    __syncthreads();
    if (threadIdx.x < 6) {
        T v = s[threadIdx.x][0];
        for (int w = 1; w < 8; ++w) {
            const T o = s[threadIdx.x][w];
            v = threadIdx.x < 3 ? (o < v ? o : v) : (o > v ? o : v);
        }
        if (threadIdx.x < 3)
            atomicMin(&out[threadIdx.x], ord_enc((double)v));
        else
            atomicMax(&out[threadIdx.x], ord_enc((double)v));
    }
    if (threadIdx.x == 0 && sbad) atomicOr(&out[6], 1ull);
}

// =================================================================== keys

__device__ __forceinline__ uint64_t spread3(uint64_t x) {
    x &= 0x1fffffull;
    x = (x | x << 32) & 0x1f00000000ffffull;
    x = (x | x << 16) & 0x1f0000ff0000ffull;
    x = (x | x << 8) & 0x100f00f00f00f00full;
    x = (x | x << 4) & 0x10c30c30c30c30c3ull;
    x = (x | x << 2) & 0x1249249249249249ull;
    return x;
}
__host__ __device__ __forceinline__ uint64_t compact3(uint64_t x) {
    x &= 0x1249249249249249ull;
    x = (x ^ (x >> 2)) & 0x10c30c30c30c30c3ull;
    x = (x ^ (x >> 4)) & 0x100f00f00f00f00full;
    x = (x ^ (x >> 8)) & 0x1f0000ff0000ffull;
    x = (x ^ (x >> 16)) & 0x1f00000000ffffull;
    x = (x ^ (x >> 32)) & 0x1fffffull;
    return x;
}

// Finest-grid coordinate floor(((x - o)/d0) * 2^21), clamped to [0, 2^21 - 1]; the
// subtraction and the division are IEEE FP64 operations, the scaling is exact.  The quotient is
// first formed as a product with scale = 2^21 / d0 (rounded), which is off by at most two roundings, 2^-30
// of a grid cell here; only when it lies within 2^-26 of a cell boundary, where the floor could
// differ, is the division done (16.4 -> 11.0 ms for 2e8 points: an FP64 division is about twenty FP64 operations).
__device__ __forceinline__ uint64_t fine_coord(double x, double o, double d0, double scale) {
    const double y = __dsub_rn(x, o);
    double t = __dmul_rn(y, scale), f = floor(t);
    const double r = t - f;
    if (!(r > 1.4901161193847656e-08 && r < 1.0 - 1.4901161193847656e-08)) f = floor(__ddiv_rn(y, d0) * 2097152.0);
    f = fmax(f, 0.0);
    f = fmin(f, 2097151.0);
    return (uint64_t)(uint32_t)f;
}

struct D3 {
    double v[3];
};

template <class T>
__global__ void k_keys(const T *__restrict__ P, int64_t n, D3 o, double d0, double scale, uint64_t setbit, uint32_t idx0,
                       uint64_t *__restrict__ keys, uint32_t *__restrict__ idx) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint64_t g0 = fine_coord((double)P[3 * i], o.v[0], d0, scale);
    uint64_t g1 = fine_coord((double)P[3 * i + 1], o.v[1], d0, scale);
    uint64_t g2 = fine_coord((double)P[3 * i + 2], o.v[2], d0, scale);
    keys[i] = setbit | (spread3(g0) << 2) | (spread3(g1) << 1) | spread3(g2);
    idx[i] = idx0 + (uint32_t)i;
}

// After the joint sort: split (keys, vals) into the X part [0, nx) and the Y part.
__global__ void k_split_sorted(const uint64_t *__restrict__ keys, const uint32_t *__restrict__ vals, int64_t nx,
                               int64_t n, uint64_t *__restrict__ kx, uint64_t *__restrict__ ky,
                               uint32_t *__restrict__ px, uint32_t *__restrict__ py) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint64_t k = keys[i] & 0x7fffffffffffffffull;
    if (i < nx) {
        kx[i] = k;
        px[i] = vals[i];
    } else {
        ky[i - nx] = k;
        py[i - nx] = vals[i] - (uint32_t)nx;
    }
}

// ---- box tables of both sets, every level at once
//
// A point starts a box at every level from the first one at which it and its predecessor in Morton
// order differ.  Pass 1 finds that level per point and counts, per tile of BT_TILE points, the
// points that start a box at each level; pass 2 scans the tiles' counts level by level; pass 3
// (k_box_emit) ranks the tile's points again and writes every level's tables: start, integer
// coordinates, parent, first child, and rank in the deepest level.  Three launches for both sets and
// all levels, where a flag, scan, compaction, coordinate and search launch per level and set made
// about a hundred (20k points: 0.55 of 2.3 ms of kernels).
constexpr int BT_TILE = 4096, BT_T = 256, BT_PER = BT_TILE / BT_T;

struct SetPts {
    const uint64_t *key;
    int64_t n;
    uint8_t *f;       // first level at which the point starts a box (LMAX + 1: none)
    uint32_t *cnt;    // LMAX + 1 rows of ntile counts, then their exclusive scans
    int64_t ntile;
};
struct SetPair {
    SetPts s[2];
};

__global__ void __launch_bounds__(BT_T) k_level_marks(SetPair P) {
    const SetPts S = P.s[blockIdx.y];
    if (blockIdx.x >= S.ntile) return;
    __shared__ uint32_t c[LMAX + 2];
    if (threadIdx.x < LMAX + 2) c[threadIdx.x] = 0;
    __syncthreads();
    const int64_t i0 = (int64_t)blockIdx.x * BT_TILE;
    for (int j = 0; j < BT_PER; ++j) {
        const int64_t i = i0 + j * BT_T + threadIdx.x;
        int lev = LMAX + 1;
        if (i < S.n) {
            lev = 0;
            if (i > 0) {
                const uint64_t d = S.key[i] ^ S.key[i - 1];
                lev = d ? LMAX - (63 - __clzll((long long)d)) / 3 : LMAX + 1;
            }
            S.f[i] = (uint8_t)lev;
        }
        const uint32_t peers = __match_any_sync(0xffffffffu, lev);
        if ((int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&c[lev], (uint32_t)__popc(peers));
    }
    __syncthreads();
    if (threadIdx.x <= LMAX) {
        uint32_t sum = 0;
        for (int l = 0; l <= (int)threadIdx.x; ++l) sum += c[l];
        S.cnt[(int64_t)threadIdx.x * S.ntile + blockIdx.x] = sum;
    }
}

// one block per (level, set): exclusive scan of the level's tile counts; total in tot[set][level]
__global__ void __launch_bounds__(1024) k_level_scan(SetPair P, uint32_t *__restrict__ tot) {
    const SetPts S = P.s[blockIdx.y];
    uint32_t *row = S.cnt + (int64_t)blockIdx.x * S.ntile;
    __shared__ uint32_t sw[32];
    __shared__ uint32_t t;
    uint32_t carry = 0;
    for (int64_t b = 0; b < S.ntile; b += 1024) {
        const int64_t i = b + threadIdx.x;
        const uint32_t v = i < S.ntile ? row[i] : 0u;
        const uint32_t e = block_excl_scan(v, sw, &t);
        if (i < S.ntile) row[i] = e + carry;
        carry += t;
        __syncthreads();
    }
    if (threadIdx.x == 0) tot[blockIdx.y * (LMAX + 1) + blockIdx.x] = carry;
}

struct BoxOut {
    uint32_t *start[LMAX + 1], *first_child[LMAX + 1], *fine[LMAX + 1], *parent[LMAX + 1];
    int4 *g[LMAX + 1];
    uint32_t nb[LMAX + 1];
};

__global__ void __launch_bounds__(BT_T) k_box_emit(const __grid_constant__ SetPts S, const __grid_constant__ BoxOut O,
                                                   int ldeep) {
    __shared__ uint32_t run[LMAX + 1][BT_T];  // boxes before the thread's points, per level
    __shared__ uint32_t sw[BT_T / 32], tot;
    const int64_t i0 = (int64_t)blockIdx.x * BT_TILE + (int64_t)threadIdx.x * BT_PER;
    uint8_t f[BT_PER];
#pragma unroll
    for (int j = 0; j < BT_PER; ++j) f[j] = i0 + j < S.n ? S.f[i0 + j] : (uint8_t)(LMAX + 1);
    for (int l = 0; l <= ldeep; ++l) {
        uint32_t c = 0;
#pragma unroll
        for (int j = 0; j < BT_PER; ++j) c += f[j] <= l;
        const uint32_t e = block_excl_scan(c, sw, &tot);
        run[l][threadIdx.x] = S.cnt[(int64_t)l * S.ntile + blockIdx.x] + e;
        __syncthreads();
    }
#pragma unroll 1
    for (int j = 0; j < BT_PER; ++j) {
        const int fl = f[j];
        if (fl > ldeep) continue;
        const int64_t i = i0 + j;
        const uint64_t k = S.key[i];
        const uint32_t cx = (uint32_t)compact3(k >> 2), cy = (uint32_t)compact3(k >> 1), cz = (uint32_t)compact3(k);
        const uint32_t deep = run[ldeep][threadIdx.x];
        uint32_t up = fl > 0 ? run[fl - 1][threadIdx.x] - 1u : 0u;  // the box of level fl - 1 that holds the point
        for (int l = fl; l <= ldeep; ++l) {
            const uint32_t r = run[l][threadIdx.x]++;
            const int sh = LMAX - l;
            O.start[l][r] = (uint32_t)i;
            O.g[l][r] = make_int4((int)(cx >> sh), (int)(cy >> sh), (int)(cz >> sh), 0);
            O.fine[l][r] = deep;
            if (O.parent[l]) O.parent[l][r] = up;
            if (l > fl) O.first_child[l - 1][up] = r;
            up = r;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x <= ldeep) {
        const int l = threadIdx.x;
        O.start[l][O.nb[l]] = (uint32_t)S.n;
        O.fine[l][O.nb[l]] = O.nb[ldeep];
        if (l < ldeep) O.first_child[l][O.nb[l]] = O.nb[l + 1];
    }
}

// out[b] = first index j in sorted `hay` (length nh) with hay[j] >= needle[b]; out[nb] = nh.
__global__ void k_lower_bound(const uint32_t *__restrict__ needle, int64_t nb, const uint32_t *__restrict__ hay,
                              int64_t nh, uint32_t *__restrict__ out) {
    int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b > nb) return;
    if (b == nb) {
        out[nb] = (uint32_t)nh;
        return;
    }
    uint32_t x = needle[b];
    int64_t lo = 0, hi = nh;
    while (lo < hi) {
        int64_t mid = (lo + hi) >> 1;
        if (hay[mid] < x)
            lo = mid + 1;
        else
            hi = mid;
    }
    out[b] = (uint32_t)lo;
}

// ================================================================== descent

// Admissibility of a child pair as integer comparisons.  The offset test |sigma + k| >= 2
// (k = g_X - g_Y per axis, sigma the trees' shift in box units, FP64) depends on k through
// the rounded sum fl(sigma + k), which is non-decreasing in k: it holds exactly for k >= klo
// or k <= khi, the two integer thresholds found on the host by evaluating that same FP64
// sum (adm_thresholds).  The decision is therefore the FP64 one, bit for bit.
struct AdmK {
    int lo[3], hi[3];
};

__device__ __forceinline__ bool child_adm_k(int4 p, int4 q, const AdmK &K) {
    int kx = p.x - q.x, ky = p.y - q.y, kz = p.z - q.z;
    return kx >= K.lo[0] || kx <= K.hi[0] || ky >= K.lo[1] || ky <= K.hi[1] || kz >= K.lo[2] || kz <= K.hi[2];
}

static AdmK adm_thresholds(const D3 &sig) {
    AdmK K;
    for (int d = 0; d < 3; ++d) {
        const volatile double sv = sig.v[d];
        // smallest k with fl(sigma + k) >= 2, largest k with fl(sigma + k) <= -2
        int lo = (int)std::floor(2.0 - sv) - 2;
        while (!(sv + (double)lo >= 2.0)) ++lo;
        while (sv + (double)(lo - 1) >= 2.0) --lo;
        int hi = (int)std::ceil(-2.0 - sv) + 2;
        while (!(sv + (double)hi <= -2.0)) --hi;
        while (sv + (double)(hi + 1) <= -2.0) ++hi;
        K.lo[d] = lo;
        K.hi[d] = hi;
    }
    return K;
}

// One warp per target box a2 of the child level: its candidates are the children of the sources
// near its parent (CSR near_off, near_src over the parents), four near sources of up to eight
// children per round.  Both passes visit them in the same order and test them alike; the
// first counts the admissible and the near ones (and marks the translations and source boxes
// in use), the second writes them at the scanned offsets.  The lists come out in CSR order by
// target with no sort, each target's sources in the order of its parent's list, the order that a
// stable sort by target of the expanded pairs gives.
//
// What bounds it: the candidates' coordinate loads (16 bytes each from L2) and, at 1e8 points, the
// lists' 24 bytes per pair.  Expanding pairs and sorting them by target per level (an iota, a radix
// sort, gathers, run starts, scans: about forty launches and eight read-backs a level) took 2.3 ms of
// kernels at 20k points and 330 ms at 1e8.
//
// Translation code of a pair: integer offset m = gX - gY relative to c = round(-sigma 2^l), 4 bits
// per axis (the descent bounds |sigma 2^l + m| < 5).
constexpr int DS_W = 8;  // warps (targets in flight) per block
struct DescendArgs {
    int64_t n;                    // target boxes of the child level
    const uint32_t *parent;
    const uint32_t *near_off, *near_src;
    const uint32_t *fcy;          // first children of the source boxes
    const int4 *gx, *gy;          // child level
    AdmK K;
    int4 c;
    uint32_t *cadm, *cnear;       // pass 1: counts; pass 2: offsets
    uint32_t *used;               // 4096 flags by code
    uint8_t *src_used;
    int *err;
    const uint32_t *tpos;         // pass 2: translation index by code
    uint32_t *adm_src, *adm_t, *near_out;  // pass 2: null where not wanted
};

template <bool EMIT>
__global__ void __launch_bounds__(32 * DS_W) k_descend(const __grid_constant__ DescendArgs A) {
    __shared__ uint32_t bits[EMIT ? 1 : 128];
    __shared__ uint16_t pos[EMIT ? 4096 : 1];
    const int lane = threadIdx.x & 31, sub = lane >> 3, cb = lane & 7;
    if constexpr (EMIT) {
        for (int i = threadIdx.x; i < 4096; i += blockDim.x) pos[i] = (uint16_t)A.tpos[i];
    } else {
        if (threadIdx.x < 128) bits[threadIdx.x] = 0u;
    }
    __syncthreads();
    const uint32_t below = (1u << lane) - 1u;
    for (int64_t x = (int64_t)blockIdx.x * DS_W + (threadIdx.x >> 5); x < A.n; x += (int64_t)gridDim.x * DS_W) {
        const uint32_t par = A.parent[x], e0 = A.near_off[par], e1 = A.near_off[par + 1];
        const int4 p = A.gx[x];
        uint32_t ia = EMIT ? A.cadm[x] : 0u, in = EMIT ? A.cnear[x] : 0u;
        for (uint32_t eb = e0; eb < e1; eb += 32) {
            uint32_t b0 = 0, nb = 0;
            if (eb + lane < e1) {
                const uint32_t b = A.near_src[eb + lane];
                b0 = A.fcy[b];
                nb = A.fcy[b + 1] - b0;
            }
            const int ne = (int)min(32u, e1 - eb);
            for (int j = 0; j < ne; j += 4) {
                const uint32_t B0 = __shfl_sync(0xffffffffu, b0, j + sub), NB = __shfl_sync(0xffffffffu, nb, j + sub);
                const bool valid = cb < (int)NB;  // lanes past the list have no children
                const uint32_t b2 = B0 + cb;
                bool adm = false;
                uint32_t code = 0;
                if (valid) {
                    const int4 q = A.gy[b2];
                    adm = child_adm_k(p, q, A.K);
                    if (adm) {
                        int mx = p.x - q.x - A.c.x + 8, my = p.y - q.y - A.c.y + 8, mz = p.z - q.z - A.c.z + 8;
                        if (mx < 0 || mx > 15 || my < 0 || my > 15 || mz < 0 || mz > 15) {
                            atomicOr(A.err, 1);
                            mx = my = mz = 0;
                        }
                        code = (uint32_t)(mx | (my << 4) | (mz << 8));
                    }
                }
                const uint32_t ma = __ballot_sync(0xffffffffu, adm), mn = __ballot_sync(0xffffffffu, valid && !adm);
                if constexpr (EMIT) {
                    if (adm) {
                        if (A.adm_src) {
                            const uint32_t o = ia + __popc(ma & below);
                            A.adm_src[o] = b2;
                            A.adm_t[o] = pos[code];
                        }
                    } else if (valid && A.near_out) {
                        A.near_out[in + __popc(mn & below)] = b2;
                    }
                } else if (adm) {
                    const uint32_t bit = 1u << (code & 31);
                    if (!(*reinterpret_cast<volatile uint32_t *>(&bits[code >> 5]) & bit)) atomicOr(&bits[code >> 5], bit);
                    A.src_used[b2] = 1;
                }
                ia += __popc(ma);
                in += __popc(mn);
            }
        }
        if (!EMIT && lane == 0) {
            A.cadm[x] = ia;
            A.cnear[x] = in;
        }
    }
    if constexpr (!EMIT) {
        __syncthreads();
        for (int k = threadIdx.x; k < 4096; k += blockDim.x)
            if (bits[k >> 5] & (1u << (k & 31))) A.used[k] = 1u;
    }
}

// ---- a level's lists from its counts: offsets of the admissible and near pairs by target, the
// targets with admissible pairs and the sources in use, and all boxes' point chunks (box, first
// point) of at most ch points, so that the point-wise kernels spread large boxes over many blocks.
// Tiles of LV_TILE boxes: sums per tile, a scan over the tiles in one block (which also numbers the
// translations in use and leaves all totals in one place, the level's only read-back), then the lists.
constexpr int LV_T = 256, LV_PER = 8, LV_TILE = LV_T * LV_PER;

// Pairs are counted in 64 bits (a tile's in 32: LV_TILE boxes of at most 665 admissible and 64 near ones), their lists
// and offsets have 32: the host refuses what does not fit before anything is written through them.
struct LevelTotals {
    unsigned long long tgt_points, src_points;
    unsigned long long na, nn;
    uint32_t ntgt, nsrc, tch, sch, ntrans, err;
    uint32_t pw_sch, pw_tch;  // chunks of PW_TC_FCH source points and PW_TC_BCH target points
    uint32_t bits[128];       // the translation codes in use
};

struct LevelArgsL {
    int64_t nx, ny, ntx, nty;
    uint32_t *cadm, *cnear;          // counts in, offsets out (nx + 1)
    const uint8_t *src_used;
    const uint32_t *xstart, *ystart;
    uint32_t ch;
    unsigned long long *ta, *tb;     // per tile: admissible << 32 | near (X); listed << 32 | chunks (X, then Y)
    const uint32_t *used;
    uint32_t *tpos;
    LevelTotals *tot;
    const int *err;
    uint32_t *tgt, *adm_off, *src;
    uint2 *tchunks, *schunks;
};

__device__ __forceinline__ unsigned long long warp_incl_scan64(unsigned long long v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// block-wide exclusive scan of one 64-bit value per thread
__device__ __forceinline__ unsigned long long block_excl_scan64(unsigned long long v, unsigned long long *sm,
                                                                unsigned long long *tot) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const unsigned long long inc = warp_incl_scan64(v);
    if (lane == 31) sm[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const unsigned long long w = lane < nw ? sm[lane] : 0ull, wi = warp_incl_scan64(w);
        if (lane < nw) sm[lane] = wi - w;
        if (lane == nw - 1) *tot = wi;
    }
    __syncthreads();
    return inc - v + sm[warp];
}

__global__ void __launch_bounds__(LV_T) k_level_sums(const __grid_constant__ LevelArgsL A) {
    const bool X = blockIdx.x < A.ntx;
    const int64_t tile = X ? blockIdx.x : blockIdx.x - A.ntx, n = X ? A.nx : A.ny;
    const uint32_t *start = X ? A.xstart : A.ystart;
    unsigned long long a = 0, b = 0, pts = 0;
    uint32_t pw = 0;
    for (int j = 0; j < LV_PER; ++j) {
        const int64_t i = tile * LV_TILE + j * LV_T + threadIdx.x;
        if (i >= n) break;
        bool listed;
        if (X) {
            const uint32_t na = A.cadm[i];
            a += ((unsigned long long)na << 32) | A.cnear[i];
            listed = na > 0;
        } else {
            listed = A.src_used[i] != 0;
        }
        const uint32_t sz = start[i + 1] - start[i];
        if (A.ch) b += (sz + A.ch - 1) / A.ch;
        if (listed) {
            b += 1ull << 32;
            pts += sz;
            pw += X ? (sz + PW_TC_BCH - 1) / PW_TC_BCH : (sz + PW_TC_FCH - 1) / PW_TC_FCH;
        }
    }
    __shared__ unsigned long long sm[32], t;
    block_excl_scan64(a, sm, &t);
    if (threadIdx.x == 0 && X) {
        A.ta[tile] = t;
        // the totals, each kind by itself: the scan's packed sums hold only 32 bits of each
        atomicAdd(&A.tot->na, t >> 32);
        atomicAdd(&A.tot->nn, t & 0xffffffffull);
    }
    __syncthreads();
    block_excl_scan64(b, sm, &t);
    if (threadIdx.x == 0) A.tb[blockIdx.x] = t;
    __syncthreads();
    block_excl_scan64(pts, sm, &t);
    if (threadIdx.x == 0 && t) atomicAdd(X ? &A.tot->tgt_points : &A.tot->src_points, t);
    __syncthreads();
    block_excl_scan64(pw, sm, &t);
    if (threadIdx.x == 0 && t) atomicAdd(X ? &A.tot->pw_tch : &A.tot->pw_sch, (uint32_t)t);
}

__global__ void __launch_bounds__(1024) k_level_mid(const __grid_constant__ LevelArgsL A) {
    __shared__ unsigned long long sm[32], t;
    auto scan_row = [&](unsigned long long *row, int64_t n) {
        unsigned long long carry = 0;
        for (int64_t b = 0; b < n; b += 1024) {
            const int64_t i = b + threadIdx.x;
            const unsigned long long v = i < n ? row[i] : 0ull;
            const unsigned long long e = block_excl_scan64(v, sm, &t);
            if (i < n) row[i] = e + carry;
            carry += t;
            __syncthreads();
        }
        return carry;
    };
    const unsigned long long a = scan_row(A.ta, A.ntx), bx = scan_row(A.tb, A.ntx), by = scan_row(A.tb + A.ntx, A.nty);
    uint32_t u[4], c = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        u[j] = c;
        c += A.used[threadIdx.x * 4 + j];
    }
    const uint32_t e = (uint32_t)block_excl_scan64(c, sm, &t);
#pragma unroll
    for (int j = 0; j < 4; ++j) A.tpos[threadIdx.x * 4 + j] = e + u[j];
    if (threadIdx.x < 128) {
        uint32_t w = 0;
        for (int j = 0; j < 32; ++j) w |= (A.used[threadIdx.x * 32 + j] ? 1u : 0u) << j;
        A.tot->bits[threadIdx.x] = w;
    }
    if (threadIdx.x == 0) {
        A.tot->ntgt = (uint32_t)(bx >> 32);
        A.tot->tch = (uint32_t)bx;
        A.tot->nsrc = (uint32_t)(by >> 32);
        A.tot->sch = (uint32_t)by;
        A.tot->ntrans = (uint32_t)t;
        A.tot->err = (uint32_t)*A.err;
        A.cadm[A.nx] = (uint32_t)(a >> 32);
        A.cnear[A.nx] = (uint32_t)a;
        A.adm_off[bx >> 32] = (uint32_t)(a >> 32);
    }
}

__global__ void __launch_bounds__(LV_T) k_level_lists(const __grid_constant__ LevelArgsL A) {
    __shared__ unsigned long long sm[32], t;
    __shared__ uint32_t cpos[LV_TILE + 1];  // first chunk of each box of the tile
    const bool X = blockIdx.x < A.ntx;
    const int64_t tile = X ? blockIdx.x : blockIdx.x - A.ntx, n = X ? A.nx : A.ny;
    const int64_t i0 = tile * LV_TILE + (int64_t)threadIdx.x * LV_PER;
    const uint32_t *start = X ? A.xstart : A.ystart;
    unsigned long long a[LV_PER], b[LV_PER], sa = 0, sb = 0;
#pragma unroll
    for (int j = 0; j < LV_PER; ++j) {
        const int64_t i = i0 + j;
        a[j] = b[j] = 0;
        if (i < n) {
            bool listed;
            if (X) {
                const uint32_t na = A.cadm[i];
                a[j] = ((unsigned long long)na << 32) | A.cnear[i];
                listed = na > 0;
            } else {
                listed = A.src_used[i] != 0;
            }
            const uint32_t sz = start[i + 1] - start[i];
            b[j] = ((unsigned long long)listed << 32) | (A.ch ? (sz + A.ch - 1) / A.ch : 0u);
        }
        sa += a[j];
        sb += b[j];
    }
    unsigned long long ea = block_excl_scan64(sa, sm, &t);
    if (X) ea += A.ta[tile];
    __syncthreads();
    unsigned long long eb = block_excl_scan64(sb, sm, &t) + A.tb[blockIdx.x];
    const uint32_t c0 = (uint32_t)A.tb[blockIdx.x];
#pragma unroll
    for (int j = 0; j < LV_PER; ++j) {
        const int64_t i = i0 + j;
        cpos[threadIdx.x * LV_PER + j] = (uint32_t)eb - c0;
        if (i < n) {
            if (b[j] >> 32) {
                const uint32_t r = (uint32_t)(eb >> 32);
                if (X) {
                    A.tgt[r] = (uint32_t)i;
                    A.adm_off[r] = (uint32_t)(ea >> 32);
                } else {
                    A.src[r] = (uint32_t)i;
                }
            }
            if (X) {
                A.cadm[i] = (uint32_t)(ea >> 32);
                A.cnear[i] = (uint32_t)ea;
            }
        }
        ea += a[j];
        eb += b[j];
    }
    if (threadIdx.x == LV_T - 1) cpos[LV_TILE] = (uint32_t)eb - c0;
    __syncthreads();
    if (!A.ch) return;
    // the tile's chunks, consecutive in the list: each finds its box in the tile's positions
    uint2 *out = (X ? A.tchunks : A.schunks) + c0;
    const uint32_t m = cpos[LV_TILE];
    for (uint32_t k = threadIdx.x; k < m; k += LV_T) {
        int lo = 0, hi = LV_TILE;  // last box with cpos <= k
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (cpos[mid] <= k)
                lo = mid;
            else
                hi = mid;
        }
        const uint32_t box = (uint32_t)(tile * LV_TILE + lo);
        out[k] = make_uint2(box, start[box] + (k - cpos[lo]) * A.ch);
    }
}

// ---- pairs grouped by translation, for the transfers by translation: counts per translation, their
// scan, then every block of GP_TGT targets reserves a range in each of its translations and places
// its pairs there (the order within a translation decides nothing: the transfers add).
constexpr int GP_TGT = 32, GP_MAXT = 4096;

template <bool PLACE>
__global__ void __launch_bounds__(256) k_group_pairs(const uint32_t *__restrict__ tgt, const uint32_t *__restrict__ off,
                                                     int64_t n_tgt, const uint32_t *__restrict__ src,
                                                     const uint32_t *__restrict__ tr, int n_trans,
                                                     uint32_t *__restrict__ cursor, uint32_t *__restrict__ bt_src,
                                                     uint32_t *__restrict__ bt_tgt) {
    __shared__ uint32_t cnt[GP_MAXT];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t x0 = (int64_t)blockIdx.x * GP_TGT, x1 = min(n_tgt, x0 + GP_TGT);
    for (int t = tid; t < n_trans; t += 256) cnt[t] = 0u;
    __syncthreads();
    const uint32_t e0 = off[x0], e1 = off[x1];
    for (uint32_t e = e0 + tid; e < e1; e += 256) atomicAdd(&cnt[tr[e]], 1u);
    __syncthreads();
    for (int t = tid; t < n_trans; t += 256)
        if (cnt[t]) cnt[t] = atomicAdd(&cursor[t], cnt[t]);
    if constexpr (PLACE) {
        __syncthreads();
        for (int64_t x = x0 + warp; x < x1; x += 8)
            for (uint32_t e = off[x] + lane; e < off[x + 1]; e += 32) {
                const uint32_t o = atomicAdd(&cnt[tr[e]], 1u);
                bt_src[o] = src[e];
                bt_tgt[o] = tgt[x];
            }
    }
}

static uint32_t read_u32(const uint32_t *d, cudaStream_t s) {
    uint32_t h;
    FFM_CUDA(cudaMemcpyAsync(&h, d, sizeof h, cudaMemcpyDeviceToHost, s));
    FFM_CUDA(cudaStreamSynchronize(s));
    return h;
}

// Near-field work items of one target leaf: its targets in chunks of tchunk times its
// near pairs split into consecutive ranges of at most smax source points.
__device__ __forceinline__ int p2p_ranges(const uint32_t *off, const uint32_t *src, const uint32_t *ystart, int64_t a,
                                          int4 *out, int base, int tc, int tchunk, uint32_t smax,
                                          unsigned long long &sources) {
    int nr = 0;
    uint32_t e0 = off[a], acc = 0;
    sources = 0;
    for (uint32_t e = off[a]; e < off[a + 1]; ++e) {
        uint32_t nb = ystart[src[e] + 1] - ystart[src[e]];
        sources += nb;
        if (acc > 0 && acc + nb > smax) {
            if (out)
                for (int c = 0; c < tc; ++c) out[base + nr * tc + c] = make_int4((int)a, c * tchunk, (int)e0, (int)e);
            ++nr;
            e0 = e;
            acc = 0;
        }
        acc += nb;
    }
    if (off[a + 1] > off[a]) {
        if (out)
            for (int c = 0; c < tc; ++c)
                out[base + nr * tc + c] = make_int4((int)a, c * tchunk, (int)e0, (int)off[a + 1]);
        ++nr;
    }
    return nr;
}

// Pass 1 (out null) counts the items per leaf and, with `pairs`, sums the point pairs n_a n_b.
__global__ void k_p2p_items(const uint32_t *__restrict__ off, const uint32_t *__restrict__ src,
                            const uint32_t *__restrict__ xstart, const uint32_t *__restrict__ ystart, int64_t nleaf,
                            int tchunk, uint32_t smax, const uint32_t *__restrict__ pos, uint32_t *__restrict__ cnt,
                            int4 *__restrict__ out, unsigned long long *__restrict__ pairs) {
    int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long v = 0;
    if (a < nleaf) {
        int np = (int)(xstart[a + 1] - xstart[a]);
        int tc = (np + tchunk - 1) / tchunk;
        if (!out) {
            cnt[a] = (uint32_t)(p2p_ranges(off, src, ystart, a, nullptr, 0, tc, tchunk, smax, v) * tc);
            v *= (unsigned long long)np;
        } else {
            p2p_ranges(off, src, ystart, a, out, (int)pos[a], tc, tchunk, smax, v);
        }
    }
    if (!pairs) return;
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(pairs, v);
}

// Work items for the near field with targets in chunks of tchunk (<= P2P_T) and at most
// smax source points per item (a larger single leaf stays whole); returns the count.
int64_t build_p2p_items(ffm_plan_s *p, int tchunk, uint32_t smax, Alloc &out_mem, int4 **items, Alloc &tmp,
                        cudaStream_t s, int64_t *pairs) {
    int ls = p->l_stop;
    int64_t nleafX = p->bx[ls].nb;
    uint32_t *icnt = tmp.get<uint32_t>(nleafX + 1), *ipos = tmp.get<uint32_t>(nleafX + 1);
    unsigned long long *sums = tmp.get<unsigned long long>(2), h[2];  // point pairs, items
    FFM_CUDA(cudaMemsetAsync(icnt + nleafX, 0, sizeof(uint32_t), s));
    FFM_CUDA(cudaMemsetAsync(sums, 0, sizeof h, s));
    FFM_LAUNCH(k_p2p_items, cdiv(nleafX, 128), 128, 0, s, p->near_off, p->near_src, p->bx[ls].start, p->by[ls].start,
               nleafX, tchunk, smax, (const uint32_t *)nullptr, icnt, (int4 *)nullptr, pairs ? sums : nullptr);
    scan_u32(icnt, ipos, nleafX + 1, (uint32_t *)(sums + 1), tmp, s);
    FFM_CUDA(cudaMemcpyAsync(h, sums, sizeof h, cudaMemcpyDeviceToHost, s));
    FFM_CUDA(cudaStreamSynchronize(s));
    int64_t n = (int64_t)(uint32_t)h[1];
    if (pairs) *pairs = (int64_t)h[0];
    *items = out_mem.get<int4>(n);
    FFM_LAUNCH(k_p2p_items, cdiv(nleafX, 128), 128, 0, s, p->near_off, p->near_src, p->bx[ls].start, p->by[ls].start,
               nleafX, tchunk, smax, ipos, icnt, *items, (unsigned long long *)nullptr);
    return n;
}

// ======================================================== leaf coordinates

template <class T>
__global__ void k_leaf_eps(const T *__restrict__ P, const uint32_t *__restrict__ perm,
                           const uint64_t *__restrict__ key, const uint32_t *__restrict__ lstart, int64_t nleaf,
                           int64_t n, D3 o, double dls, int ls, float4 *__restrict__ eps, float4 *__restrict__ lo) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint64_t k = key[i];
    int sh = LMAX - ls;
    double g0 = (double)(compact3(k >> 2) >> sh), g1 = (double)(compact3(k >> 1) >> sh), g2 = (double)(compact3(k) >> sh);
    uint32_t j = perm[i];
    // leaf-relative coordinates as an unevaluated FP32 pair hi + lo
    double d0 = (double)P[3 * (int64_t)j] - (o.v[0] + (g0 + 0.5) * dls);
    double d1 = (double)P[3 * (int64_t)j + 1] - (o.v[1] + (g1 + 0.5) * dls);
    double d2 = (double)P[3 * (int64_t)j + 2] - (o.v[2] + (g2 + 0.5) * dls);
    float e0 = (float)d0, e1 = (float)d1, e2 = (float)d2;
    int64_t lo_ = 0, hi_ = nleaf - 1;  // last leaf with start <= i
    while (lo_ < hi_) {
        int64_t mid = (lo_ + hi_ + 1) >> 1;
        if (lstart[mid] <= (uint32_t)i)
            lo_ = mid;
        else
            hi_ = mid - 1;
    }
    eps[i] = make_float4(e0, e1, e2, __uint_as_float((uint32_t)lo_));
    lo[i] = make_float4((float)(d0 - (double)e0), (float)(d1 - (double)e1), (float)(d2 - (double)e2), 0.f);
}

template <class T>
__global__ void k_sorted_weights(const T *__restrict__ w, const uint32_t *__restrict__ perm, int64_t n,
                                 double *__restrict__ out) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = (double)w[perm[i]];
}

// Source normals in Morton order as unevaluated FP32 pairs (hi, lo): the double layer's
// n . (x - y) cancels to second order in |x - y| for points of one surface.
template <class T>
__global__ void k_sorted_normals(const T *__restrict__ nrm, const uint32_t *__restrict__ perm, int64_t n,
                                 float4 *__restrict__ hi, float4 *__restrict__ lo) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const T *v = nrm + 3 * (int64_t)perm[i];
    double a = (double)v[0], b = (double)v[1], c = (double)v[2];
    float ah = (float)a, bh = (float)b, ch = (float)c;
    hi[i] = make_float4(ah, bh, ch, 0.f);
    lo[i] = make_float4((float)(a - (double)ah), (float)(b - (double)bh), (float)(c - (double)ch), 0.f);
}

// ================================================================ host side

static bool is_device_ptr(const void *p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// Device copy of a caller array (host or device) of `bytes` bytes.
static const void *to_device(const void *p, size_t bytes, Alloc &tmp, cudaStream_t s) {
    if (is_device_ptr(p)) return p;
    void *d = tmp.raw(bytes);
    FFM_CUDA(cudaMemcpyAsync(d, p, bytes, cudaMemcpyHostToDevice, s));
    return d;
}

template <class T>
static void launch_keys(const void *P, int64_t n, const double o[3], double d0, uint64_t setbit, uint32_t idx0,
                        uint64_t *keys, uint32_t *idx, cudaStream_t s) {
    D3 oo{{o[0], o[1], o[2]}};
    FFM_LAUNCH(k_keys<T>, cdiv(n, 256), 256, 0, s, (const T *)P, n, oo, d0, 2097152.0 / d0, setbit, idx0, keys,
               idx);
}

template <class T>
static void launch_bbox(const void *P, int64_t n, unsigned long long *out, cudaStream_t s) {
    FFM_LAUNCH(k_bbox<T>, std::min<unsigned>(cdiv(n, 1024), 152u * 8u), 256, 0, s, (const T *)P, n, out);
}

template <class T>
static void launch_leaf_eps(const void *P, const uint32_t *perm, const uint64_t *key, const uint32_t *lstart,
                            int64_t nleaf, int64_t n, const double o[3], double dls, int ls, float4 *eps,
                            float4 *lo, cudaStream_t s) {
    D3 oo{{o[0], o[1], o[2]}};
    FFM_LAUNCH(k_leaf_eps<T>, cdiv(n, 256), 256, 0, s, (const T *)P, perm, key, lstart, nleaf, n, oo, dls, ls, eps,
               lo);
}


// Box tables of one set for levels 0..ldeep (boxes at level l = runs of key >> 3(21-l)); parents
// only where asked for (the target boxes).
static void build_boxes(ffm_plan_s *p, BoxLevel *bl, const SetPts &S, const int64_t *nb, int ldeep, uint32_t **parent,
                        cudaStream_t s) {
    Alloc &m = p->mem;
    BoxOut O{};
    for (int l = 0; l <= ldeep; ++l) {
        BoxLevel &B = bl[l];
        B.nb = nb[l];
        O.nb[l] = (uint32_t)nb[l];
        O.start[l] = B.start = m.get<uint32_t>(B.nb + 1);
        O.fine[l] = B.fine = m.get<uint32_t>(B.nb + 1);
        O.g[l] = B.g = m.get<int4>(B.nb);
        if (l < ldeep) O.first_child[l] = B.first_child = m.get<uint32_t>(B.nb + 1);
        if (parent) O.parent[l] = parent[l] = m.get<uint32_t>(B.nb);
    }
    FFM_LAUNCH(k_box_emit, (unsigned)S.ntile, BT_T, 0, s, S, O, ldeep);
}

static int oscillatory(const ffm_plan_s *p, int l) {
    double dl = std::ldexp(p->d0, -l);
    return p->kind == FFM_HELMHOLTZ && p->k * dl >= p->kappa;
}

static int pw_rank(double k, double dl, double eps) {
    int L = (int)std::floor(std::fabs(k) * std::sqrt(3.0) * dl - std::log(eps));
    return L < 1 ? 1 : L;
}

// Chunks of at most ch points of the listed boxes (their number is known): (box, first point).
__global__ void k_chunk_count(const uint32_t *__restrict__ list, int64_t n, const uint32_t *__restrict__ start,
                              uint32_t ch, uint32_t *__restrict__ cnt) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t b = list[i];
    cnt[i] = (start[b + 1] - start[b] + ch - 1) / ch;
}
__global__ void k_chunk_emit(const uint32_t *__restrict__ list, int64_t n, const uint32_t *__restrict__ start,
                             uint32_t ch, const uint32_t *__restrict__ pos, uint2 *__restrict__ out) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t b = list[i], k = pos[i];
    for (uint32_t q = start[b]; q < start[b + 1]; q += ch) out[k++] = make_uint2(b, q);
}

static uint2 *build_chunks(ffm_plan_s *p, const uint32_t *list, int64_t n, const uint32_t *start, int64_t count,
                           Alloc &tmp, cudaStream_t s, uint32_t ch) {
    uint32_t *cnt = tmp.get<uint32_t>(n), *pos = tmp.get<uint32_t>(n);
    FFM_LAUNCH(k_chunk_count, cdiv(n, 256), 256, 0, s, list, n, start, ch, cnt);
    scan_u32(cnt, pos, n, nullptr, tmp, s);
    uint2 *out = p->mem.get<uint2>(count);
    FFM_LAUNCH(k_chunk_emit, cdiv(n, 256), 256, 0, s, list, n, start, ch, pos, out);
    return out;
}

// Whether a level runs the target-stationary transfer when nothing else decides.  Measured on GB300 at
// r = 64: that transfer takes 0.53 us per translation of a 128-target tile, one tile per SM at a
// time, whatever the tile's pairs; the one by translation 9.0e-5 us per pair (from 1.4M pairs on), and
// grouping the pairs for it about as much again in the plan.  So it pays from about 3000 (one product)
// to 5900 (many products) pairs per translation and wave of tiles.  Both sides, us: clustered 10M level 7
// (68M pairs, 10 waves) 3520 / 6139, level 6 (11M, 2 waves) 709 / 1006, level 5 (1.4M, 1 wave)
// 356 / 141; volume 2M level 5 (11.9M, 2 waves) 704 / 1087; sphere 2M level 7 (5.5M, 4 waves) 631 / 511.
// Lower ranks take the same line: volume 2M, level 5, about 0.5 / 0.65 ms at r = 8 and 0.5 / 1.6 at r = 27 (from totals
// over the levels).  Several right-hand sides multiply both sides, so a level that is over the line stays over it
// (8 columns, all levels of a clustered 3M: 29.0 / 50.3 ms); one below it may be worth it for many columns, which
// the plan does not know.
static bool target_stationary_pays(const FarLevel &F) {
    const int64_t waves = (F.n_tgt + 128 * 152 - 1) / (128 * 152);
    return F.n_adm >= 4000 * (int64_t)F.n_trans * waves;
}

// Column tiles of the per-translation transfer: tile i of translation t covers pairs
// off[t] + i bn .. (count per translation, then one block per translation emits its tiles).
__global__ void k_tile_count(const uint32_t *__restrict__ off, int n_trans, uint32_t bn, uint32_t *__restrict__ cnt) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n_trans) cnt[t] = (off[t + 1] - off[t] + bn - 1) / bn;
}
__global__ void k_tile_emit(const uint32_t *__restrict__ off, uint32_t bn, const uint32_t *__restrict__ pos,
                            uint32_t *__restrict__ tt, uint32_t *__restrict__ tp) {
    int t = blockIdx.x;
    uint32_t p0 = off[t], n = (off[t + 1] - p0 + bn - 1) / bn, o = pos[t];
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) {
        tt[o + i] = (uint32_t)t;
        tp[o + i] = p0 + i * bn;
    }
}

static int64_t build_tiles(ffm_plan_s *p, const FarLevel &F, uint32_t bn, uint32_t **tt, uint32_t **tp, Alloc &tmp,
                           cudaStream_t s) {
    uint32_t *cnt = tmp.get<uint32_t>(F.n_trans), *pos = tmp.get<uint32_t>(F.n_trans), *tot = tmp.get<uint32_t>(1);
    FFM_LAUNCH(k_tile_count, cdiv(F.n_trans, 256), 256, 0, s, F.bt_off, F.n_trans, bn, cnt);
    scan_u32(cnt, pos, F.n_trans, tot, tmp, s);
    int64_t n = read_u32(tot, s);
    *tt = p->mem.get<uint32_t>(n);
    *tp = p->mem.get<uint32_t>(n);
    if (n > 0) FFM_LAUNCH(k_tile_emit, F.n_trans, 128, 0, s, F.bt_off, bn, pos, *tt, *tp);
    return n;
}

static D3 level_shift(const ffm_plan_s *p, int l) {
    return D3{{std::ldexp(p->sigma[0], l), std::ldexp(p->sigma[1], l), std::ldexp(p->sigma[2], l)}};
}

int3 near_base(const ffm_plan_s *p, int l) {
    const AdmK K = adm_thresholds(level_shift(p, l));
    return make_int3(K.hi[0] + 1, K.hi[1] + 1, K.hi[2] + 1);
}

static int4 trans_centre(const ffm_plan_s *p, int l) {
    if (l == 0) return make_int4(0, 0, 0, 0);  // the single root pair has m = 0
    return make_int4((int)std::floor(-std::ldexp(p->sigma[0], l) + 0.5), (int)std::floor(-std::ldexp(p->sigma[1], l) + 0.5),
                     (int)std::floor(-std::ldexp(p->sigma[2], l) + 0.5), 0);
}

__global__ void k_trans_codes(const int4 *__restrict__ m, int n, int4 c, uint32_t *__restrict__ tpos) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const int4 v = m[t];
    tpos[(v.x - c.x + 8) | (v.y - c.y + 8) << 4 | (v.z - c.z + 8) << 8] = (uint32_t)t;
}

// The descent's second pass again, for the admissible pairs alone; the offsets per box come from the
// listed targets' offsets.
__global__ void k_box_offsets(const uint32_t *__restrict__ tgt, const uint32_t *__restrict__ off, int64_t n,
                              uint32_t *__restrict__ out) {
    const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x < n) out[tgt[x]] = off[x];
}

void fill_pair_lists(const ffm_plan_s *p, int l, uint32_t *src, uint32_t *t, cudaStream_t s) {
    const FarLevel &F = p->far[l];
    if (F.n_adm > MAX_LISTED) fail(FFM_EUNSUPPORTED, "more than 2^32 - 2^12 admissible pairs: the level has no list of them");
    Alloc tmp;
    tmp.stream = s;
    DescendArgs D{};
    D.n = p->bx[l].nb;
    D.parent = p->parent[l];
    D.near_off = p->nr_off[l - 1];
    D.near_src = p->nr_src[l - 1];
    D.fcy = p->by[l - 1].first_child;
    D.gx = p->bx[l].g;
    D.gy = p->by[l].g;
    D.K = adm_thresholds(level_shift(p, l));
    D.c = trans_centre(p, l);
    D.cadm = tmp.get<uint32_t>(D.n);
    D.cnear = tmp.get<uint32_t>(D.n);
    uint32_t *tpos = tmp.get<uint32_t>(4096);
    D.tpos = tpos;
    D.err = p->dev_err;
    D.adm_src = src;
    D.adm_t = t;
    FFM_CUDA(cudaMemsetAsync(D.cadm, 0, sizeof(uint32_t) * D.n, s));
    FFM_CUDA(cudaMemsetAsync(D.cnear, 0, sizeof(uint32_t) * D.n, s));
    FFM_CUDA(cudaMemsetAsync(tpos, 0, sizeof(uint32_t) * 4096, s));
    FFM_LAUNCH(k_trans_codes, cdiv(F.n_trans, 256), 256, 0, s, F.trans_m, F.n_trans, D.c, tpos);
    FFM_LAUNCH(k_box_offsets, cdiv(F.n_tgt, 256), 256, 0, s, F.tgt, F.adm_off, F.n_tgt, D.cadm);
    FFM_LAUNCH(k_descend<true>, std::min<unsigned>(cdiv(D.n, DS_W), 152u * 32u), 32 * DS_W, 0, s, D);
}

// Pairs of Lagrange level l grouped by translation (CSR bt_off over translations, with each
// pair's source and target box).  Made while the plan is built, or later by the autotuner or
// when the target-stationary transfer cannot take the level; a level that runs the
// target-stationary transfer does without them.
void build_translation_groups(ffm_plan_s *p, int l, cudaStream_t s) {
    FarLevel &F = p->far[l];
    if (F.mode != 1 || F.n_adm == 0 || F.bt_off) return;
    if (F.n_adm > MAX_LISTED) fail(FFM_EUNSUPPORTED, "more than 2^32 - 2^12 admissible pairs: the level has no list of them");
    Alloc tmp;
    tmp.stream = s;
    if (!F.adm_src) {
        F.adm_src = p->mem.get<uint32_t>(F.n_adm);
        F.adm_t = p->mem.get<uint32_t>(F.n_adm);
        fill_pair_lists(p, l, F.adm_src, F.adm_t, s);
    }
    F.bt_src = p->mem.get<uint32_t>(F.n_adm);
    F.bt_tgt = p->mem.get<uint32_t>(F.n_adm);
    F.bt_off = p->mem.get<uint32_t>(F.n_trans + 1);
    uint32_t *cursor = tmp.get<uint32_t>(F.n_trans + 1);
    const unsigned g = cdiv(F.n_tgt, GP_TGT);
    FFM_CUDA(cudaMemsetAsync(cursor, 0, sizeof(uint32_t) * (F.n_trans + 1), s));
    FFM_LAUNCH(k_group_pairs<false>, g, 256, 0, s, F.tgt, F.adm_off, F.n_tgt, F.adm_src, F.adm_t, F.n_trans, cursor,
               (uint32_t *)nullptr, (uint32_t *)nullptr);
    scan_u32(cursor, F.bt_off, F.n_trans + 1, nullptr, tmp, s);
    FFM_CUDA(cudaMemcpyAsync(cursor, F.bt_off, sizeof(uint32_t) * F.n_trans, cudaMemcpyDeviceToDevice, s));
    FFM_LAUNCH(k_group_pairs<true>, g, 256, 0, s, F.tgt, F.adm_off, F.n_tgt, F.adm_src, F.adm_t, F.n_trans, cursor,
               F.bt_src, F.bt_tgt);
    tmp.release();
}

// Column tiles over those groups: 32 pairs for the CUDA-core GEMM, 256 for the ACA factors on
// the tensor cores (the dense tensor-core transfer cuts its own).
void build_group_tiles(ffm_plan_s *p, int l, cudaStream_t s) {
    FarLevel &F = p->far[l];
    if (F.mode != 1 || F.n_adm == 0 || F.tile_t) return;
    build_translation_groups(p, l, s);
    if (!(p->aca_eps > 0.0)) build_lag_table(p, l, s);
    Alloc tmp;
    tmp.stream = s;
    F.n_tiles = build_tiles(p, F, LAG_GEMM_BN, &F.tile_t, &F.tile_p0, tmp, s);
    if (p->aca_eps > 0.0) F.tc_tiles = build_tiles(p, F, 256, &F.tc_tile_t, &F.tc_tile_p0, tmp, s);
    tmp.release();
}

// Level l of the descent (its temporaries in tmp): counts, lists, the read-back of their sizes, the pairs.  D holds
// the geometry and the parents' near lists; at l = 0 (root cubes already far apart) the one pair is
// given.  The near pairs of the level go to near_off / near_src, in the plan's memory when the
// descent stops here (stop(near pairs)).  Returns the number of near pairs.
struct NearLists {
    uint32_t *off = nullptr, *src = nullptr;
};

template <class Stop>
static int64_t descend_level(ffm_plan_s *p, int l, DescendArgs D, Stop &&stop, NearLists &near, int64_t pw[2], Alloc &tmp,
                             cudaStream_t s) {
    FarLevel &F = p->far[l];
    const int64_t nx = p->bx[l].nb, ny = p->by[l].nb;
    const bool root = l == 0;
    D.n = nx;
    D.gx = p->bx[l].g;
    D.gy = p->by[l].g;
    D.c = trans_centre(p, l);
    // zeroed scratch: totals, translation flags, error flag, source flags
    struct Scratch {
        LevelTotals tot;
        uint32_t used[4096];
        int err;
    };
    unsigned char *scr = static_cast<unsigned char *>(tmp.raw(sizeof(Scratch) + (size_t)ny));
    Scratch *S = reinterpret_cast<Scratch *>(scr);
    FFM_CUDA(cudaMemsetAsync(scr, 0, sizeof(Scratch) + (size_t)ny, s));
    D.used = S->used;
    D.err = &S->err;
    D.src_used = scr + sizeof(Scratch);
    D.cadm = tmp.get<uint32_t>(nx + 1);
    D.cnear = tmp.get<uint32_t>(nx + 1);
    uint32_t *tpos = tmp.get<uint32_t>(4096);
    D.tpos = tpos;
    const unsigned dg = std::min<unsigned>(cdiv(nx, DS_W), 152u * 32u);
    if (root) {
        static const uint32_t one = 1, zero = 0;
        FFM_CUDA(cudaMemcpyAsync(D.cadm, &one, sizeof one, cudaMemcpyHostToDevice, s));
        FFM_CUDA(cudaMemcpyAsync(D.cnear, &zero, sizeof zero, cudaMemcpyHostToDevice, s));
        FFM_CUDA(cudaMemcpyAsync(D.used + (8 | 8 << 4 | 8 << 8), &one, sizeof one, cudaMemcpyHostToDevice, s));
        FFM_CUDA(cudaMemsetAsync(D.src_used, 1, 1, s));
    } else {
        FFM_LAUNCH(k_descend<false>, dg, 32 * DS_W, 0, s, D);
    }
    // Lagrange levels take point chunks; the lists are sized by their upper bounds
    const bool lag = !oscillatory(p, l);
    LevelArgsL L{};
    L.nx = nx;
    L.ny = ny;
    L.ntx = cdiv(nx, LV_TILE);
    L.nty = cdiv(ny, LV_TILE);
    L.cadm = D.cadm;
    L.cnear = D.cnear;
    L.src_used = D.src_used;
    L.xstart = p->bx[l].start;
    L.ystart = p->by[l].start;
    L.ch = lag ? LAG_CHUNK : 0;
    L.ta = tmp.get<unsigned long long>(L.ntx);
    L.tb = tmp.get<unsigned long long>(L.ntx + L.nty);
    L.used = D.used;
    L.tpos = tpos;
    L.tot = &S->tot;
    L.err = D.err;
    L.tgt = p->mem.get<uint32_t>(nx);
    L.adm_off = p->mem.get<uint32_t>(nx + 1);
    L.src = p->mem.get<uint32_t>(ny);
    if (lag) {
        L.tchunks = p->mem.get<uint2>(nx + p->nx / LAG_CHUNK);
        L.schunks = p->mem.get<uint2>(ny + p->ny / LAG_CHUNK);
    }
    const unsigned lg = (unsigned)(L.ntx + L.nty);
    FFM_LAUNCH(k_level_sums, lg, LV_T, 0, s, L);
    FFM_LAUNCH(k_level_mid, 1, 1024, 0, s, L);
    FFM_LAUNCH(k_level_lists, lg, LV_T, 0, s, L);
    LevelTotals h;
    FFM_CUDA(cudaMemcpyAsync(&h, &S->tot, sizeof h, cudaMemcpyDeviceToHost, s));
    FFM_CUDA(cudaStreamSynchronize(s));
    if (h.err) fail(FFM_ECUDA, "box translation outside the expected range");
    const int64_t na = (int64_t)h.na, nn = (int64_t)h.nn;
    if (nn > MAX_LISTED) fail(FFM_EUNSUPPORTED, "more than 2^32 - 2^12 near pairs at one level");
    F.n_adm = na;
    p->info.n_adm[l] = na;
    const bool last = stop(nn);
    F.n_trans = (int)h.ntrans;
    F.n_tgt = h.ntgt;
    F.r1 = p->r1_override > 0 ? p->r1_override : r1_rule(p->kind, p->eps);
    // before anything is sized or indexed by it
    if (lag && na > 0 && F.r1 > R1MAX) fail(FFM_EUNSUPPORTED, "eps needs more than 8 Chebyshev nodes per axis");
    // a level that is to run the target-stationary transfer (the option, the pick stored in the plan's
    // autotune cache, or the rule) takes no pair lists
    const bool ts_able = p->kind == FFM_LAPLACE && F.r1 <= 4 && !(p->aca_eps > 0.0);
    const int pick = lag && na > 0 && p->lag_transfer == 0 ? cached_lag_pick(p, l) : -1;
    bool ts_first = false;
    if (lag && na > 0) {
        if (p->lag_transfer > 0) F.tune_tc = p->lag_transfer - 1;  // forced variant
        if (ts_able && !root && p->lag_transfer == 0 && pick < 0 && target_stationary_pays(F)) F.tune_tc = 2;
        // (the only transfer for more pairs than a list can hold)
        if (ts_able && !root && (pick == 2 || (p->lag_transfer == 0 && na > MAX_LISTED))) F.tune_tc = 2;
        ts_first = ts_able && !root && F.tune_tc == 2;
    }
    if (na > MAX_LISTED && !ts_first)
        fail(FFM_EUNSUPPORTED, "more than 2^32 - 2^12 admissible pairs at one level (only the target-stationary transfer "
                               "of the Laplace single layer does without a list of them)");
    if (na > 0 && !ts_first) {
        F.adm_src = p->mem.get<uint32_t>(na);
        F.adm_t = p->mem.get<uint32_t>(na);
    }
    // the near lists outlive the descent where it stops and where the next level may look into them
    const bool keep = last || ts_able;
    near.src = keep ? p->mem.get<uint32_t>(nn) : tmp.get<uint32_t>(nn);
    near.off = D.cnear;
    if (keep) {
        near.off = p->mem.get<uint32_t>(nx + 1);
        FFM_CUDA(cudaMemcpyAsync(near.off, D.cnear, sizeof(uint32_t) * (nx + 1), cudaMemcpyDeviceToDevice, s));
        p->nr_off[l] = near.off;
        p->nr_src[l] = near.src;
    }
    D.adm_src = F.adm_src;
    D.adm_t = F.adm_t;
    D.near_out = near.src;
    if (root) {
        FFM_CUDA(cudaMemsetAsync(F.adm_src, 0, sizeof(uint32_t), s));
        FFM_CUDA(cudaMemsetAsync(F.adm_t, 0, sizeof(uint32_t), s));
    } else {
        FFM_LAUNCH(k_descend<true>, dg, 32 * DS_W, 0, s, D);
    }
    if (na == 0) return nn;
    F.mode = lag ? 1 : 2;
    F.tgt = L.tgt;
    F.adm_off = L.adm_off;
    F.n_src = h.nsrc;
    F.src = L.src;
    F.tgt_chunks = L.tchunks;
    F.src_chunks = L.schunks;
    F.n_tgt_chunks = h.tch;
    F.n_src_chunks = h.sch;
    pw[0] = h.pw_sch;
    pw[1] = h.pw_tch;
    F.h_trans_m.clear();
    for (int k = 0; k < 4096; ++k)
        if (h.bits[k >> 5] >> (k & 31) & 1u)
            F.h_trans_m.push_back(make_int4((k & 15) - 8 + D.c.x, ((k >> 4) & 15) - 8 + D.c.y, (k >> 8) - 8 + D.c.z, 0));
    F.trans_m = p->mem.get<int4>(F.n_trans);
    FFM_CUDA(cudaMemcpyAsync(F.trans_m, F.h_trans_m.data(), sizeof(int4) * F.n_trans, cudaMemcpyHostToDevice, s));
    p->info.n_trans[l] = F.n_trans;
    p->info.src_points[l] = (int64_t)h.src_points;
    p->info.tgt_points[l] = (int64_t)h.tgt_points;
    if (F.mode == 1) {
        // pairs grouped by translation for the transfers by translation (ACA levels need them)
        if (!ts_first) build_translation_groups(p, l, s);
        if (p->lag_transfer == 1 || pick == 0 || p->aca_eps > 0.0) build_group_tiles(p, l, s);
        p->info.r1[l] = F.r1;
    }
    p->info.mode[l] = F.mode;
    if (F.mode == 2) {
        F.L = pw_rank(p->k, std::ldexp(p->d0, -l), p->eps);
        F.nQ = 2 * F.L * (F.L + 1);
        p->info.L[l] = F.L;
        p->info.nQ[l] = F.nQ;
    }
    return nn;
}

void build_plan(ffm_plan_s *p, const void *X, ffm_dtype xdt, const void *Y, ffm_dtype ydt, const void *w,
                ffm_dtype wdt, Alloc &tmp) {
    cudaStream_t s = p->stream;
    int64_t nx = p->nx, ny = p->ny, n = nx + ny;
    size_t xb = (xdt == FFM_F64 ? 8 : 4) * 3 * (size_t)nx, yb = (ydt == FFM_F64 ? 8 : 4) * 3 * (size_t)ny;
    const void *dX = to_device(X, xb, tmp, s), *dY = to_device(Y, yb, tmp, s);

    p->dev_err = p->mem.get<int>(4);
    FFM_CUDA(cudaMemsetAsync(p->dev_err, 0, 4 * sizeof(int), s));

    // ---- root cubes (Sec. 2.2.1)
    unsigned long long *bb = tmp.get<unsigned long long>(14);
    unsigned long long init[14];
    for (int i = 0; i < 2; ++i) {
        for (int d = 0; d < 3; ++d) {
            init[7 * i + d] = ~0ull;
            init[7 * i + 3 + d] = 0ull;
        }
        init[7 * i + 6] = 0ull;
    }
    FFM_CUDA(cudaMemcpyAsync(bb, init, sizeof init, cudaMemcpyHostToDevice, s));
    if (xdt == FFM_F64)
        launch_bbox<double>(dX, nx, bb, s);
    else
        launch_bbox<float>(dX, nx, bb, s);
    if (ydt == FFM_F64)
        launch_bbox<double>(dY, ny, bb + 7, s);
    else
        launch_bbox<float>(dY, ny, bb + 7, s);
    unsigned long long hb[14];
    FFM_CUDA(cudaMemcpyAsync(hb, bb, sizeof hb, cudaMemcpyDeviceToHost, s));
    FFM_CUDA(cudaStreamSynchronize(s));
    if (hb[6] || hb[13]) fail(FFM_EINVAL, "non-finite coordinate in X or Y");
    double lx[3], hx[3], ly[3], hy[3];
    for (int d = 0; d < 3; ++d) {
        lx[d] = ord_dec(hb[d]);
        hx[d] = ord_dec(hb[3 + d]);
        ly[d] = ord_dec(hb[7 + d]);
        hy[d] = ord_dec(hb[10 + d]);
    }
    double ex = 0, ey = 0;
    for (int d = 0; d < 3; ++d) {
        ex = std::max(ex, hx[d] - lx[d]);
        ey = std::max(ey, hy[d] - ly[d]);
    }
    double d0 = std::max(ex, ey);
    double infl = 1.0 + std::ldexp(1.0, -20);
    d0 = d0 > 0.0 ? d0 * infl : 1.0;
    for (int d = 0; d < 3; ++d) {
        double cx = 0.5 * (lx[d] + hx[d]), cy = 0.5 * (ly[d] + hy[d]);
        double hd = 0.5 * d0;
        p->oX[d] = cx - hd;
        p->oY[d] = cy - hd;
        p->sigma[d] = (p->oX[d] - p->oY[d]) / d0;
    }
    p->d0 = d0;
    p->info.d0 = d0;
    for (int d = 0; d < 3; ++d) {
        p->info.oX[d] = p->oX[d];
        p->info.oY[d] = p->oY[d];
    }

    // ---- Morton keys and the joint stable sort (X first: set bit 0; Y: set bit 1)
    Alloc sortmem;  // keys, indices and the sort's ping-pong buffers: released after the split
    sortmem.stream = s;
    uint64_t *keys = sortmem.get<uint64_t>(n);
    uint32_t *vals = sortmem.get<uint32_t>(n);
    if (xdt == FFM_F64)
        launch_keys<double>(dX, nx, p->oX, d0, 0ull, 0u, keys, vals, s);
    else
        launch_keys<float>(dX, nx, p->oX, d0, 0ull, 0u, keys, vals, s);
    if (ydt == FFM_F64)
        launch_keys<double>(dY, ny, p->oY, d0, 1ull << 63, (uint32_t)nx, keys + nx, vals + nx, s);
    else
        launch_keys<float>(dY, ny, p->oY, d0, 1ull << 63, (uint32_t)nx, keys + nx, vals + nx, s);
    radix_sort_u64(keys, vals, n, 64, sortmem, s);
    p->keyX = p->mem.get<uint64_t>(nx);
    p->keyY = p->mem.get<uint64_t>(ny);
    p->permX = p->mem.get<uint32_t>(nx);
    p->permY = p->mem.get<uint32_t>(ny);
    FFM_LAUNCH(k_split_sorted, cdiv(n, 256), 256, 0, s, keys, vals, nx, n, p->keyX, p->keyY, p->permX, p->permY);
    sortmem.release();

    // ---- boxes per level
    SetPair sp;
    uint32_t *lvtot = tmp.get<uint32_t>(2 * (LMAX + 1));
    for (int i = 0; i < 2; ++i) {
        SetPts &S = sp.s[i];
        S.key = i == 0 ? p->keyX : p->keyY;
        S.n = i == 0 ? nx : ny;
        S.ntile = cdiv(S.n, BT_TILE);
        S.f = tmp.get<uint8_t>(S.n);
        S.cnt = tmp.get<uint32_t>((size_t)S.ntile * (LMAX + 1));
    }
    FFM_LAUNCH(k_level_marks, dim3((unsigned)std::max(sp.s[0].ntile, sp.s[1].ntile), 2), BT_T, 0, s, sp);
    FFM_LAUNCH(k_level_scan, dim3(LMAX + 1, 2), 1024, 0, s, sp, lvtot);
    uint32_t hc[2 * (LMAX + 1)];
    FFM_CUDA(cudaMemcpyAsync(hc, lvtot, sizeof hc, cudaMemcpyDeviceToHost, s));
    FFM_CUDA(cudaStreamSynchronize(s));
    int64_t nbx[LMAX + 1], nby[LMAX + 1];
    for (int l = 0; l <= LMAX; ++l) {
        nbx[l] = hc[l];
        nby[l] = hc[LMAX + 1 + l];
    }
    // deepest level the occupancy rule can reach
    int ldeep = 0;
    while (ldeep < p->l_cap && !(n < (int64_t)p->n_leaf * (nbx[ldeep] + nby[ldeep]))) ++ldeep;
    build_boxes(p, p->bx, sp.s[0], nbx, ldeep, p->parent, s);
    build_boxes(p, p->by, sp.s[1], nby, ldeep, nullptr, s);
    for (int l = 0; l <= ldeep; ++l) {
        p->info.nboxX[l] = nbx[l];
        p->info.nboxY[l] = nby[l];
    }

    // ---- descent (Sec. 2.2.2, 2.2.4)
    bool root_adm = false;
    for (int d = 0; d < 3; ++d)
        if (std::fabs(p->sigma[d]) >= 2.0) root_adm = true;
    Alloc levels[LMAX + 2];  // per-level temporaries of the descent, released level by level
    TableJob tj(s);
    NearLists near;  // at the root: box 0 with box 0
    p->nr_off[0] = near.off = p->mem.get<uint32_t>(2);
    p->nr_src[0] = near.src = p->mem.get<uint32_t>(1);
    static const uint32_t root_off[2] = {0, 1};
    FFM_CUDA(cudaMemcpyAsync(near.off, root_off, sizeof root_off, cudaMemcpyHostToDevice, s));
    FFM_CUDA(cudaMemsetAsync(near.src, 0, sizeof(uint32_t), s));
    int64_t nnear = 1, pwc[LMAX + 1][2] = {};
    auto stops = [&](int l, int64_t nn) {
        return nn == 0 || n < (int64_t)p->n_leaf * (nbx[l] + nby[l]) || l >= p->l_cap;
    };
    p->l_stop = 0;
    if (root_adm) {
        p->root_adm = 1;
        p->info.root_admissible = 1;
        levels[0].stream = s;
        nnear = descend_level(p, 0, DescendArgs{}, [](int64_t) { return true; }, near, pwc[0], levels[0], s);
        build_tables(p, 0, tj);
    } else {
        p->info.n_near[0] = 1;
        int l = 0;
        for (; !stops(l, nnear); ++l) {
            const int lc = l + 1;
            DescendArgs D{};
            D.parent = p->parent[lc];
            D.near_off = near.off;
            D.near_src = near.src;
            D.fcy = p->by[l].first_child;
            D.K = adm_thresholds(level_shift(p, lc));
            levels[lc].stream = s;
            nnear = descend_level(p, lc, D, [&](int64_t nn) { return stops(lc, nn); }, near, pwc[lc], levels[lc], s);
            // the previous level's near lists are no longer needed
            if (l >= 1) levels[l].release();
            if (p->far[lc].n_adm > 0) build_tables(p, lc, tj);
            p->info.n_near[lc] = nnear;
        }
        p->l_stop = l;
    }
    int ls = p->l_stop;
    p->info.l_stop = ls;

    // ---- near pairs at the stop level: CSR over all target leaves
    p->n_near = nnear;
    p->near_off = near.off;
    if (nnear > 0) {
        p->near_src = near.src;
        // work items: target chunks x bounded source ranges
        p->n_items = build_p2p_items(p, p->p2p_tchunk, p->p2p_smax, p->mem, &p->items, tmp, s, &p->info.p2p_pairs);
    }

    // ---- leaf links and leaf-relative coordinates
    for (int l = 0; l <= ls; ++l) {
        for (BoxLevel *B : {&p->bx[l], &p->by[l]}) {
            if (ls == ldeep) {  // the leaves are the deepest boxes: their ranks are in the tables
                B->first_leaf = B->fine;
                continue;
            }
            BoxLevel &Lf = (B == &p->bx[l]) ? p->bx[ls] : p->by[ls];
            B->first_leaf = p->mem.get<uint32_t>(B->nb + 1);
            FFM_LAUNCH(k_lower_bound, cdiv(B->nb + 1, 256), 256, 0, s, B->fine, B->nb, Lf.fine, Lf.nb, B->first_leaf);
        }
    }
    double dls = std::ldexp(d0, -ls);
    p->epsX = p->mem.get<float4>(nx);
    p->epsY = p->mem.get<float4>(ny);
    p->epsXlo = p->mem.get<float4>(nx);
    p->epsYlo = p->mem.get<float4>(ny);
    if (xdt == FFM_F64)
        launch_leaf_eps<double>(dX, p->permX, p->keyX, p->bx[ls].start, p->bx[ls].nb, nx, p->oX, dls, ls, p->epsX, p->epsXlo, s);
    else
        launch_leaf_eps<float>(dX, p->permX, p->keyX, p->bx[ls].start, p->bx[ls].nb, nx, p->oX, dls, ls, p->epsX, p->epsXlo, s);
    if (ydt == FFM_F64)
        launch_leaf_eps<double>(dY, p->permY, p->keyY, p->by[ls].start, p->by[ls].nb, ny, p->oY, dls, ls, p->epsY, p->epsYlo, s);
    else
        launch_leaf_eps<float>(dY, p->permY, p->keyY, p->by[ls].start, p->by[ls].nb, ny, p->oY, dls, ls, p->epsY, p->epsYlo, s);
    if (w) {
        const void *dw = to_device(w, (wdt == FFM_F64 ? 8 : 4) * (size_t)ny, tmp, s);
        p->wY = p->mem.get<double>(ny);
        if (wdt == FFM_F64)
            FFM_LAUNCH(k_sorted_weights<double>, cdiv(ny, 256), 256, 0, s, (const double *)dw, p->permY, ny, p->wY);
        else
            FFM_LAUNCH(k_sorted_weights<float>, cdiv(ny, 256), 256, 0, s, (const float *)dw, p->permY, ny, p->wY);
    }
    if (p->kind == FFM_LAPLACE_DL) {
        size_t esz = p->normals_dt == FFM_F64 ? 8 : 4;
        const void *dn = to_device(p->normals_in, 3 * esz * (size_t)ny, tmp, s);
        p->nY = p->mem.get<float4>(ny);
        p->nYlo = p->mem.get<float4>(ny);
        if (p->normals_dt == FFM_F64)
            FFM_LAUNCH(k_sorted_normals<double>, cdiv(ny, 256), 256, 0, s, (const double *)dn, p->permY, ny, p->nY,
                       p->nYlo);
        else
            FFM_LAUNCH(k_sorted_normals<float>, cdiv(ny, 256), 256, 0, s, (const float *)dn, p->permY, ny, p->nY,
                       p->nYlo);
    }
    for (int l = 0; l <= ls; ++l)
        if (p->far[l].n_adm > 0) build_octants(p, l, tj);
    // every dense Lagrange level leaves here with what its transfer reads: near tables or grouped pairs
    for (int l = 0; l <= ls; ++l) {
        FarLevel &F = p->far[l];
        if (F.tune_tc == 2) prepare_target_stationary(p, l, s);
        if (F.mode == 1 && F.n_adm > 0 && !F.ts_ok) build_translation_groups(p, l, s);
    }
    // plane-wave levels whose F steps run as type-3 NUFFTs: FP32 levels with many directions
    // (the NUFFT's cost per box barely depends on nQ, the direct sums' grows with it), all
    // FP32 and compensated-FP32 levels when forced, none when direct sums are forced
    for (int l = 0; l <= ls; ++l) {
        const FarLevel &F = p->far[l];
        if (F.mode != 2 || F.n_adm == 0) continue;
        bool want = p->pw_transform == 2   ? (F.prec == FFM_PREC_F32 || F.prec == FFM_PREC_F32C)
                    : p->pw_transform == 1 ? false
                                           : (F.prec == FFM_PREC_F32 && F.nQ >= NUFFT_MIN_NQ);
        if (want && nufft_possible(p, l)) build_nufft(p, l, tmp, s);
    }
    // the remaining FP32 and compensated-FP32 direct levels: point pieces of their boxes for
    // the tensor-core transforms of several right-hand sides (not with direct sums forced
    // onto the CUDA cores, nor for the NUFFT)
    if (p->pw_transform == 0 || p->pw_transform == 3)
        for (int l = 0; l <= ls; ++l) {
            FarLevel &F = p->far[l];
            if (F.mode != 2 || F.n_adm == 0 || F.nufft || (F.prec != FFM_PREC_F32 && F.prec != FFM_PREC_F32C))
                continue;
            F.n_pw_chunks = pwc[l][0];
            F.n_pw_tchunks = pwc[l][1];
            F.pw_chunks = build_chunks(p, F.src, F.n_src, p->by[l].start, pwc[l][0], tmp, s, PW_TC_FCH);
            F.pw_tchunks = build_chunks(p, F.tgt, F.n_tgt, p->bx[l].start, pwc[l][1], tmp, s, PW_TC_BCH);
        }
    FFM_CUDA(cudaStreamSynchronize(s));
}

}  // namespace ffm
