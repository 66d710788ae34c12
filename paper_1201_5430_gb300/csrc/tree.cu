// Octree construction on the GPU: cube, Morton keys, stable LSD radix sort,
// boxes per level, parent/child ranges, colleague lists and P2P work items.
//
// The paper fixes the data structure only as "octree, neighbor lists" (Sec. 4,
// table of FMM stages) with the standard 189-box M2L stencil (Sec. 5).  The
// construction here is: cube origin = per-axis minimum; side = the smallest
// r_q 2^k >= the largest extent (k an integer), with r_q the core radius r_K
// below rounded up to an 8-bit mantissa, so that the box side of some level lies
// in [r_K, 1.008 r_K) and the core rule below can stop the tree there (without a
// core: the smallest power of two >= the largest extent); q = floor((x - x0) 2^21 /
// side) in FP64 (in a batch with a core every system takes the largest side of the
// batch, origins staying per system),
// clamped to [0, 2^21 - 1]; key = 63-bit interleave with x in bit 0 of each
// triple; stable sort by key (ties keep the caller's order); leaf level
// L = min(L_leaf, L_K, max_level) where L_leaf is the shallowest level with at
// most leaf_max elements per box and L_K the deepest level whose box side is
// >= r_K, the radius beyond which the Gaussian core of Eq. vem1 equals 1 to
// eps/10 (so every far-field pair sees the singular kernel of Eq. 1).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "lhv_internal.cuh"

namespace lhv {

// words of the counts array past the levels' counts (0 ..) and offsets (32 ..)
constexpr int COUNTS_L = 56, COUNTS_NONFINITE = 57, COUNTS_L_CAP = 58;
static_assert(KEY_BITS + 1 < 32 && 32 + KEY_BITS + 1 < COUNTS_L, "a word per level");

// r_K rounded up to an 8-bit mantissa (0 for no core): the unit of the cube side
double core_unit(double rK) {
    if (!(rK > 0.0)) return 0.0;
    int e;
    const double m = std::frexp(rK, &e);  // rK = m 2^e, 0.5 <= m < 1
    return std::ldexp(std::ceil(m * 256.0) / 256.0, e);
}

// ---------------------------------------------------------------------------
// Bit interleave helpers (21 bits per axis into 63 bits)
// ---------------------------------------------------------------------------
__host__ __device__ inline uint64_t spread3(uint64_t v) {
    v &= 0x1fffffull;
    v = (v | (v << 32)) & 0x1f00000000ffffull;
    v = (v | (v << 16)) & 0x1f0000ff0000ffull;
    v = (v | (v << 8)) & 0x100f00f00f00f00full;
    v = (v | (v << 4)) & 0x10c30c30c30c30c3ull;
    v = (v | (v << 2)) & 0x1249249249249249ull;
    return v;
}

__host__ __device__ inline uint64_t compact3(uint64_t v) {
    v &= 0x1249249249249249ull;
    v = (v ^ (v >> 2)) & 0x10c30c30c30c30c3ull;
    v = (v ^ (v >> 4)) & 0x100f00f00f00f00full;
    v = (v ^ (v >> 8)) & 0x1f0000ff0000ffull;
    v = (v ^ (v >> 16)) & 0x1f00000000ffffull;
    v = (v ^ (v >> 32)) & 0x1fffffull;
    return v;
}

__host__ __device__ inline uint64_t morton3(uint64_t qx, uint64_t qy, uint64_t qz) {
    return spread3(qx) | (spread3(qy) << 1) | (spread3(qz) << 2);
}

// ---------------------------------------------------------------------------
// Cube
// ---------------------------------------------------------------------------
template <typename T>
__device__ inline T warp_min(T v) {
    for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// nsys * parts blocks; block b reduces part b % parts of system b / parts, and the last block of
// a system its parts to its cube (an empty system gets the unit cube at the origin); rq > 0:
// the side is the smallest rq 2^k >= the extent, else the smallest power of two.  One launch
// for both: a second one of one block took 8 us.
template <typename T>
__global__ void __launch_bounds__(256) k_bbox(int parts, const int64_t* __restrict__ sysoff,
                                              const vec4_t<T>* __restrict__ x4, const vec4_t<T>* __restrict__ w4,
                                              T* __restrict__ part, SysCube* __restrict__ cubes,
                                              TreeParams* __restrict__ tp, int* __restrict__ tickets, double rq) {
    // min/max in the input type (exact; its conversion to double is exact and monotonic);
    // entries 3..5 hold the negated upper bounds
    __shared__ T s[8][6];
    const int sys = blockIdx.x / parts, q = blockIdx.x % parts, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t o0 = sysoff[sys], len = sysoff[sys + 1] - o0;
    const int64_t beg = o0 + len * q / parts, end = o0 + len * (q + 1) / parts;
    const T inf = (T)INFINITY;
    T lo[6] = {inf, inf, inf, inf, inf, inf};
    int bad = 0;
#pragma unroll 4
    for (int64_t i = beg + threadIdx.x; i < end; i += blockDim.x) {
        vec4_t<T> p = x4[i];
        vec4_t<T> qv = w4 ? w4[i] : p;
        const T c[3] = {p.x, p.y, p.z};
        bad |= !(isfinite(c[0]) && isfinite(c[1]) && isfinite(c[2]));
        bad |= !(isfinite(qv.x) && isfinite(qv.y) && isfinite(qv.z));
        for (int k = 0; k < 3; ++k) {
            lo[k] = fmin(lo[k], c[k]);
            lo[3 + k] = fmin(lo[3 + k], -c[k]);
        }
    }
    if (bad) atomicOr(&tp->nonfinite, 1);
    for (int k = 0; k < 6; ++k) {
        const T v = warp_min(lo[k]);
        if (lane == 0) s[warp][k] = v;
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        T v = s[0][threadIdx.x];
        for (int w = 1; w < 8; ++w) v = fmin(v, s[w][threadIdx.x]);
        __stcg(part + blockIdx.x * 6 + threadIdx.x, v);
    }
    if (!last_block(tickets + sys, parts)) return;
    for (int k = 0; k < 6; ++k) lo[k] = inf;
    for (int b = threadIdx.x; b < parts; b += blockDim.x)
        for (int k = 0; k < 6; ++k) lo[k] = fmin(lo[k], __ldcg(part + (sys * parts + b) * 6 + k));
    for (int k = 0; k < 6; ++k) {
        const T v = warp_min(lo[k]);
        if (lane == 0) s[warp][k] = v;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int k = 0; k < 6; ++k)
        for (int w = 0; w < 8; ++w) lo[k] = w == 0 ? s[0][k] : fmin(lo[k], s[w][k]);
    double ext = 0.0;
    const bool empty = !(lo[0] <= -lo[3]);
    for (int k = 0; k < 3; ++k) {
        cubes[sys].x0[k] = empty ? 0.0 : (double)lo[k];
        if (!empty) ext = fmax(ext, -(double)lo[3 + k] - (double)lo[k]);
    }
    double side = 1.0;
    if (ext > 0.0) {
        const double unit = rq > 0.0 ? rq : 1.0;
        // unit 2^k from the exponents, k one more where ext's mantissa is the larger; by search
        // where an exponent is not that of a normal number
        const long long be = __double_as_longlong(ext), bu = __double_as_longlong(unit);
        const int ee = (int)(be >> 52), eu = (int)(bu >> 52);
        const long long frac = (1ll << 52) - 1;
        const int es = ee + ((be & frac) > (bu & frac) ? 1 : 0);
        if (ee > 0 && eu > 0 && es < 2047 && eu < 2047) {
            side = __longlong_as_double((long long)es << 52 | (bu & frac));
        } else {
            int e;
            frexp(ext / unit, &e);  // a first guess of k, then the exact test on unit 2^k
            int k = e;
            while (ldexp(unit, k) < ext) ++k;
            while (ldexp(unit, k - 1) >= ext) --k;
            side = ldexp(unit, k);
        }
    }
    cubes[sys].side = side;
    if (sys == 0) tp->deepest_shared = -1;
}

// A batch with a core: every system takes the largest side of the batch (origins stay its
// own), so that the one leaf level of the batch, capped by the core rule, gives every system
// leaves of side r_q (with its own side, a system with a larger cube would get leaves of
// 2^j r_q at that level).
__global__ void k_cube_common(SysCube* __restrict__ cubes, int nsys) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    double side = 0.0;
    for (int k = 0; k < nsys; ++k) side = fmax(side, cubes[k].side);
    for (int k = 0; k < nsys; ++k) cubes[k].side = side;
}

__device__ inline int system_of(int64_t i, int nsys, const int64_t* __restrict__ sysoff) {
    int lo = 0, hi = nsys - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (sysoff[mid] <= i) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// ---------------------------------------------------------------------------
// Morton keys and their stable LSD radix sort with the element index, 8-bit digits
// ---------------------------------------------------------------------------
// A pass counts the digits of every tile of SORT_THREADS ITEMS keys (the keys' own kernel does it
// for the first pass), then scatters: a block finds where the tile's items of each digit
// go from the counts of all tiles, hist[tile][digit].  Up to SORT_COLUMNS tiles every block adds the
// column itself (two launches a pass, counts from L2); above, k_radix_scan turns the counts into prefixes first.
constexpr int SORT_THREADS = 256;
constexpr int SORT_WARPS = SORT_THREADS / 32;
constexpr int SORT_COLUMNS = 64;
// Items per thread: a small sort is latency on few blocks, a large one wants long runs per digit.  Tree, 4 v 16
// items, ms: 4096 elements 0.13 v 0.17, 2^18 0.18 v 0.21, 2^20 0.41 v 0.40, 2^22 0.77 v 0.73.
constexpr int64_t SORT_FEW_MAX = 524288;
constexpr int sort_items(int64_t n) { return n <= SORT_FEW_MAX ? 4 : 16; }
constexpr int64_t sort_tiles(int64_t n) { return (n + SORT_THREADS * sort_items(n) - 1) / (SORT_THREADS * sort_items(n)); }
// counts of every tile, then the digits' totals
constexpr int64_t sort_hist_ints(int64_t n) { return (sort_tiles(n) + 1) * 256; }

// Cell floor((p - x0) scale) clamped to [0, qmax], the arithmetic in double.
template <typename T>
__device__ inline unsigned cell_f64(T p, double x0, double scale, double qmax) {
    return (unsigned)fmin(fmax(floor(((double)p - x0) * scale), 0.0), qmax);
}
// Origin and scale of a cube; sh + sl = scale in floats (sh no number where the scale is out of
// their range), pow2: the scale is the power of two sh.
struct CellMap {
    double x0[3], scale;
    float x0f[3], sh, sl;
    bool pow2;
};
__device__ inline unsigned cell_of(double p, const CellMap& m, int k, double qmax) {
    return cell_f64(p, m.x0[k], m.scale, qmax);
}
// The same cell for a float position.  The difference d + e is exact (Knuth's two-sum) and ph + pl its
// product with the scale.  For a power of two the product is exact too, and so is the double
// arithmetic as long as d + e fits its 53 bits, so that the floor is that of ph, one less on a face
// with pl < 0.  Otherwise the distance r to the cell's lower face is known to far less than 2^-16, and nearer
// than that to a face (and where r is no number in between) the double arithmetic decides.
// A warp's FP64 instruction holds the SM for 16 cycles: 2^20 keys took 63 us that way, now 26.
__device__ inline unsigned cell_of(float p, const CellMap& m, int k, double qmax) {
    const float x0 = m.x0f[k], d = p - x0, bv = p - d, av = d + bv, e = (p - av) + (bv - x0);
    const float ph = d * m.sh, f = floorf(ph);
    if (m.pow2 && (e == 0.0f || fabsf(e) >= d * 0x1p-28f)) {
        const float q = f - (ph == f && e < 0.0f ? 1.0f : 0.0f);
        return (unsigned)fminf(fmaxf(q, 0.0f), (float)qmax);
    }
    const float pl = __fmaf_rn(d, m.sh, -ph) + __fmaf_rn(d, m.sl, e * m.sh), r = (ph - f) + pl;
    if (r > 0x1p-16f && r < 1.0f - 0x1p-16f && f >= 0.0f) return (unsigned)f;
    return cell_f64(p, m.x0[k], m.scale, qmax);
}

// Keys of a tile's elements and, for the first pass of their sort, the counts of its digits.
template <typename T, int ITEMS>
__global__ void __launch_bounds__(SORT_THREADS) k_morton(int64_t n, int nsys, int bits,
                                                         const int64_t* __restrict__ sysoff,
                                                         const SysCube* __restrict__ cubes,
                                                         const vec4_t<T>* __restrict__ x4,
                                                         uint64_t* __restrict__ keys, int shift,
                                                         int* __restrict__ hist) {
    struct Sys {
        int id;
        int64_t end;
        CellMap map;
    };
    __shared__ Sys first;
    __shared__ int cnt[256];
    const int64_t base = (int64_t)blockIdx.x * (SORT_THREADS * ITEMS);
    const auto load = [&](Sys& q, int64_t i) {
        q.id = nsys > 1 ? system_of(i, nsys, sysoff) : 0;
        q.end = nsys > 1 ? sysoff[q.id + 1] : n;
        const SysCube cb = cubes[q.id];
        CellMap& m = q.map;
        m.scale = (double)(1 << bits) / cb.side;
        const bool in_range = m.scale > 0x1p-60 && m.scale < 0x1p60;
        m.sh = in_range ? (float)m.scale : NAN;
        m.sl = (float)(m.scale - (double)m.sh);
        m.pow2 = in_range && (__double_as_longlong(m.scale) & ((1ll << 52) - 1)) == 0;
        for (int k = 0; k < 3; ++k) {
            m.x0[k] = cb.x0[k];
            m.x0f[k] = (float)cb.x0[k];
        }
    };
    cnt[threadIdx.x] = 0;
    if (threadIdx.x == 0) load(first, base);
    __syncthreads();
    const double qmax = (double)((1 << bits) - 1);
    Sys cur = first;
    vec4_t<T> at[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) at[j] = x4[min(base + j * SORT_THREADS + threadIdx.x, n - 1)];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const int64_t i = base + j * SORT_THREADS + threadIdx.x;
        if (i >= n) break;
        if (i >= cur.end) load(cur, i);
        const vec4_t<T> p = at[j];
        const unsigned qx = cell_of(p.x, cur.map, 0, qmax);
        const unsigned qy = cell_of(p.y, cur.map, 1, qmax);
        const unsigned qz = cell_of(p.z, cur.map, 2, qmax);
        const uint64_t key = ((uint64_t)cur.id << (3 * bits)) | morton3(qx, qy, qz);
        keys[i] = key;
        atomicAdd(&cnt[(key >> shift) & 255u], 1);
    }
    __syncthreads();
    hist[blockIdx.x * 256 + threadIdx.x] = cnt[threadIdx.x];
}

template <int ITEMS>
__global__ void __launch_bounds__(SORT_THREADS) k_radix_hist(int64_t n, const uint64_t* __restrict__ keys, int shift,
                                                             int* __restrict__ hist) {
    __shared__ int cnt[256];
    cnt[threadIdx.x] = 0;
    const int64_t base = (int64_t)blockIdx.x * (SORT_THREADS * ITEMS) + threadIdx.x;
    uint64_t key[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) key[j] = base + j * SORT_THREADS < n ? keys[base + j * SORT_THREADS] : 0ull;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < ITEMS; ++j)
        if (base + j * SORT_THREADS < n) atomicAdd(&cnt[(key[j] >> shift) & 255u], 1);
    __syncthreads();
    hist[blockIdx.x * 256 + threadIdx.x] = cnt[threadIdx.x];
}

// hist[tile][digit] -> items of the digit in earlier tiles, hist[ntiles][digit] = the digit's total.  A
// block takes eight digits (one 32-byte sector of a row), 32 threads of each a run of the rows.
__global__ void __launch_bounds__(SORT_THREADS) k_radix_scan(int ntiles, int* __restrict__ hist) {
    __shared__ int sum[32][9];
    const int d = threadIdx.x & 7, g = threadIdx.x >> 3, per = (ntiles + 31) / 32;
    const int r0 = min(g * per, ntiles), r1 = min(r0 + per, ntiles);
    int* h = hist + blockIdx.x * 8 + d;
    int t = 0;
#pragma unroll 8
    for (int r = r0; r < r1; ++r) t += h[r * 256];
    sum[g][d] = t;
    __syncthreads();
    int run = 0;
    for (int k = 0; k < g; ++k) run += sum[k][d];
    if (g == 31) h[ntiles * 256] = run + t;
    for (int r = r0; r < r1; r += 8) {
        int v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = r + k < r1 ? h[(r + k) * 256] : 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (r + k < r1) h[(r + k) * 256] = run;
            run += v[k];
        }
    }
}

__device__ int block_exclusive_scan(int v, int* total);

// Stable scatter of one digit (vin null: the indices 0, 1, ...).  Warp w of a block owns 32 ITEMS
// consecutive items: it counts its digits privately in order (rounds of 32 consecutive
// items), the warps' counts are scanned per digit, and the tile is put into digit order in shared
// memory before it is written, so that a digit's items leave as one run.
// 2^20 elements, eight passes: 45 us a pass with a three-launch scan of the counts and scattered
// writes, now 21 us; 4096 elements 28 us (one block of 16 items a thread), now 8.
template <int ITEMS, bool SCANNED>
__global__ void __launch_bounds__(SORT_THREADS) k_radix_scatter(int64_t n, const uint64_t* __restrict__ kin,
                                                               const int* __restrict__ vin,
                                                               uint64_t* __restrict__ kout, int* __restrict__ vout,
                                                               int shift, int ntiles, const int* __restrict__ hist) {
    constexpr int TILE = SORT_THREADS * ITEMS;
    __shared__ int wcnt[SORT_WARPS][256];
    __shared__ int to[256];  // global position of a digit's first item less its position in the tile
    __shared__ uint64_t stage[TILE];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    for (int w = 0; w < SORT_WARPS; ++w) wcnt[w][t] = 0;
    const int64_t tile0 = (int64_t)blockIdx.x * TILE, first = tile0 + (int64_t)warp * (32 * ITEMS);
    const unsigned lt = (1u << lane) - 1u;
    uint64_t key[ITEMS];
    int val[ITEMS], slot[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const int64_t i = first + r * 32 + lane;
        key[r] = i < n ? kin[i] : 0ull;
        val[r] = i < n ? (vin ? vin[i] : (int)i) : 0;
    }
    int before = 0, all = 0;  // items of digit t in earlier tiles, in all
    if (SCANNED) {
        before = hist[blockIdx.x * 256 + t];
        all = hist[ntiles * 256 + t];
    } else {
#pragma unroll 16
        for (int b = 0; b < ntiles; ++b) {
            const int v = hist[b * 256 + t];
            all += v;
            before += b < (int)blockIdx.x ? v : 0;
        }
    }
    // lanes with the same digit, by eight ballots (a match of the lanes runs over their distinct values)
    unsigned peers[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const int d = (int)((key[r] >> shift) & 255u);
        peers[r] = __ballot_sync(0xffffffffu, first + r * 32 + lane < n);
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const unsigned m = __ballot_sync(0xffffffffu, d >> b & 1);
            peers[r] &= d >> b & 1 ? m : ~m;
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const int d = (int)((key[r] >> shift) & 255u);
        const bool in = first + r * 32 + lane < n;
        slot[r] = wcnt[warp][d] + __popc(peers[r] & lt);
        __syncwarp();
        if (in && (peers[r] & lt) == 0) wcnt[warp][d] += __popc(peers[r]);
        __syncwarp();
    }
    __syncthreads();
    {
        int mine = 0;
        for (int w = 0; w < SORT_WARPS; ++w) mine += wcnt[w][t];
        int run = block_exclusive_scan(mine, nullptr);
        to[t] = block_exclusive_scan(all, nullptr) + before - run;
        for (int w = 0; w < SORT_WARPS; ++w) {
            const int c = wcnt[w][t];
            wcnt[w][t] = run;
            run += c;
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r)
        if (first + r * 32 + lane < n) {
            slot[r] += wcnt[warp][(int)((key[r] >> shift) & 255u)];
            stage[slot[r]] = key[r];
        }
    __syncthreads();
    const int len = (int)min((int64_t)TILE, n - tile0);
    int pos[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const int j = r * SORT_THREADS + t;
        if (j < len) {
            const uint64_t k = stage[j];
            pos[r] = to[(int)((k >> shift) & 255u)] + j;
            kout[pos[r]] = k;
        }
    }
    __syncthreads();
    int* sval = reinterpret_cast<int*>(stage);
#pragma unroll
    for (int r = 0; r < ITEMS; ++r)
        if (first + r * 32 + lane < n) sval[slot[r]] = val[r];
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r)
        if (r * SORT_THREADS + t < len) vout[pos[r]] = sval[r * SORT_THREADS + t];
}

// Launches of the two halves above for a sort of n items; return the number of launches.
template <typename T>
int launch_keys(cudaStream_t s, int64_t n, int nsys, int bits, const int64_t* sysoff, const SysCube* cubes,
                const vec4_t<T>* x4, uint64_t* keys, int shift, int* hist) {
    const auto go = [&](auto items) {
        k_morton<T, decltype(items)::value><<<(int)sort_tiles(n), SORT_THREADS, 0, s>>>(n, nsys, bits, sysoff, cubes,
                                                                                        x4, keys, shift, hist);
    };
    switch (sort_items(n)) {
        case 4: go(std::integral_constant<int, 4>{}); break;
        default: go(std::integral_constant<int, 16>{}); break;
    }
    return 1;
}

// Passes first .. 7; the keys go back and forth between kin and kout and end in kin if the number of
// passes is even, the indices start as 0, 1, ... (vin null) or in vin and end in vfin, by way of vtmp.
// counted: hist holds the first pass's counts.
int launch_sort(cudaStream_t s, int64_t n, int first, uint64_t* kin, uint64_t* kout, const int* vin, int* vfin,
                int* vtmp, bool counted, int* hist) {
    const int nt = (int)sort_tiles(n);
    int launches = 0;
    for (int pass = first; pass < 8; ++pass) {
        const int shift = 8 * pass;
        int* vout = (7 - pass) % 2 == 0 ? vfin : vtmp;
        const auto go = [&](auto items) {
            constexpr int I = decltype(items)::value;
            if (!(counted && pass == first)) {
                k_radix_hist<I><<<nt, SORT_THREADS, 0, s>>>(n, kin, shift, hist);
                ++launches;
            }
            if (nt > SORT_COLUMNS) {
                k_radix_scan<<<32, SORT_THREADS, 0, s>>>(nt, hist);
                k_radix_scatter<I, true><<<nt, SORT_THREADS, 0, s>>>(n, kin, vin, kout, vout, shift, nt, hist);
                launches += 2;
            } else {
                k_radix_scatter<I, false><<<nt, SORT_THREADS, 0, s>>>(n, kin, vin, kout, vout, shift, nt, hist);
                ++launches;
            }
        };
        switch (sort_items(n)) {
            case 4: go(std::integral_constant<int, 4>{}); break;
                default: go(std::integral_constant<int, 16>{}); break;
        }
        std::swap(kin, kout);
        vin = vout;
    }
    return launches;
}

// ---------------------------------------------------------------------------
// Exclusive scan of int32 (three passes)
// ---------------------------------------------------------------------------
constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 16;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

__device__ int block_exclusive_scan(int v, int* total) {
    __shared__ int warp_sums[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int nw = blockDim.x >> 5;
        int s = lane < nw ? warp_sums[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        if (lane < nw) warp_sums[lane] = s;
    }
    __syncthreads();
    int excl = x - v + (warp > 0 ? warp_sums[warp - 1] : 0);
    if (total) *total = warp_sums[(blockDim.x >> 5) - 1];
    __syncthreads();
    return excl;
}

__global__ void k_scan_reduce(int64_t n, const int* __restrict__ in, int* __restrict__ sums) {
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
    int s = 0;
    for (int j = 0; j < SCAN_ITEMS; ++j)
        if (base + j < n) s += in[base + j];
    int total;
    block_exclusive_scan(s, &total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// Single block: exclusive scan of the block sums; writes the grand total.
__global__ void k_scan_sums(int nb, int* __restrict__ sums, int* __restrict__ total_out) {
    __shared__ int carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int b0 = 0; b0 < nb; b0 += blockDim.x) {
        int i = b0 + threadIdx.x;
        int v = i < nb ? sums[i] : 0;
        int tot;
        int ex = block_exclusive_scan(v, &tot);
        if (i < nb) sums[i] = carry + ex;
        __syncthreads();
        if (threadIdx.x == 0) carry += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0 && total_out) *total_out = carry;
}

__global__ void k_scan_apply(int64_t n, const int* __restrict__ in, const int* __restrict__ sums,
                             int* __restrict__ out) {
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
    int v[SCAN_ITEMS];
    int s = 0;
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        v[j] = (base + j < n) ? in[base + j] : 0;
        s += v[j];
    }
    int ex = block_exclusive_scan(s, nullptr) + sums[blockIdx.x];
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        if (base + j < n) out[base + j] = ex;
        ex += v[j];
    }
}

// Small arrays (n <= 1024 * SCAN_ITEMS) in one block and one launch.
constexpr int SCAN_ONE_THREADS = 1024;
__global__ void __launch_bounds__(SCAN_ONE_THREADS) k_scan_one(int n, const int* __restrict__ in,
                                                                int* __restrict__ out, int* __restrict__ total_out) {
    const int base = threadIdx.x * SCAN_ITEMS;
    int v[SCAN_ITEMS];
    int s = 0;
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        v[j] = (base + j < n) ? in[base + j] : 0;
        s += v[j];
    }
    int tot;
    int ex = block_exclusive_scan(s, &tot);
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        if (base + j < n) out[base + j] = ex;
        ex += v[j];
    }
    if (threadIdx.x == 0 && total_out) *total_out = tot;
}

void exclusive_scan(Ctx* c, int64_t n, const int* in, int* out, int* sums_tmp, int* total_out) {
    cudaStream_t s = stream_of(c);
    if (n <= (int64_t)SCAN_ONE_THREADS * SCAN_ITEMS) {
        k_scan_one<<<1, SCAN_ONE_THREADS, 0, s>>>((int)n, in, out, total_out);
        count_launch(c);
        check_launch("exclusive_scan");
        return;
    }
    int nb = (int)((n + SCAN_TILE - 1) / SCAN_TILE);
    if (nb < 1) nb = 1;
    k_scan_reduce<<<nb, SCAN_THREADS, 0, s>>>(n, in, sums_tmp);
    count_launch(c);
    k_scan_sums<<<1, 1024, 0, s>>>(nb, sums_tmp, total_out);
    count_launch(c);
    k_scan_apply<<<nb, SCAN_THREADS, 0, s>>>(n, in, sums_tmp, out);
    count_launch(c);
    check_launch("exclusive_scan");
}

int64_t scan_tmp_ints(int64_t n) { return (n + SCAN_TILE - 1) / SCAN_TILE + 1; }

// ---------------------------------------------------------------------------
// Leaf level
// ---------------------------------------------------------------------------
// The deepest level at which leaf_max + 1 consecutive keys share a box, and from it in the last
// block the one leaf level for all systems: the deepest L_leaf any system needs, capped by the core
// rule of the smallest cube (every far pair of every system sees K = 1).
// abort_word (a captured step, whose leaf level is fixed, L_graph): the tree it builds is
// valid while every far pair still sees K = 1 (L_graph <= the core rule's cap of the current
// cube) and the input is finite; otherwise the word tells the step not to write its result.
__global__ void __launch_bounds__(256) k_leaf_level(int64_t n, int leaf_max, int bits,
                                                    const uint64_t* __restrict__ keys, TreeParams* __restrict__ tp,
                                                    const SysCube* __restrict__ cubes, int nsys, double rK,
                                                    int max_level, int L_graph, int* __restrict__ abort_word) {
    __shared__ int s_best;
    if (threadIdx.x == 0) s_best = -1;
    __syncthreads();
    int best = -1;
#pragma unroll 4
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i + leaf_max < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        uint64_t x = keys[i] ^ keys[i + leaf_max];
        int lvl;
        if (x == 0) {
            lvl = bits;
        } else {
            int msb = 63 - __clzll((long long)x);
            lvl = bits - (msb + 3) / 3;  // deepest level at which both keys share a box (< 0: two systems)
        }
        best = max(best, lvl);
    }
    best = __reduce_max_sync(0xffffffffu, best);
    if ((threadIdx.x & 31) == 0 && best >= 0) atomicMax(&s_best, best);
    __syncthreads();
    if (threadIdx.x == 0 && s_best >= 0) atomicMax(&tp->deepest_shared, s_best);
    if (!last_block(&tp->ticket, gridDim.x) || threadIdx.x >= 32) return;
    const int lane = threadIdx.x;
    double min_side = INFINITY;
    for (int s = lane; s < nsys; s += 32) min_side = fmin(min_side, cubes[s].side);
    min_side = warp_min(min_side);
    int L_K = bits;
    if (rK > 0.0) {
        const unsigned ok = __ballot_sync(0xffffffffu, lane <= bits && ldexp(min_side, -lane) >= rK);
        L_K = ok ? 31 - __clz((int)ok) : 0;
    }
    if (lane != 0) return;
    const int L_leaf = min(__ldcg(&tp->deepest_shared) + 1, bits);
    int L_cap = L_K;
    if (max_level > 0) L_cap = min(L_cap, max_level);
    tp->L_cap = L_cap;
    tp->L = min(L_leaf, L_cap);
    if (abort_word && (__ldcg(&tp->nonfinite) || L_cap < L_graph)) atomicOr(abort_word, 1);
}

// ---------------------------------------------------------------------------
// Boxes of all levels in three passes over the sorted keys
// ---------------------------------------------------------------------------
// Element i starts a box at level l iff its key and the previous key differ in
// the level-l prefix key >> 3 (bits - l), i.e. iff l >= start_level(i).
__device__ inline int start_level(const uint64_t* __restrict__ keys, int64_t i, int bits) {
    if (i == 0) return 0;
    const uint64_t x = keys[i] ^ keys[i - 1];
    if (x == 0) return 1 << 20;  // never: same leaf at every level
    const int msb = 63 - __clzll((long long)x);
    return max(0, bits - msb / 3);
}

// Elements a thread takes in the two passes over the sorted keys: few for a small tree, whose few blocks
// would leave the rest of the GPU idle; more for a large one, whose levels' rows of block counts get shorter.
// Whole tree of a cube, ms, 4 v 16: 262,144 elements 0.234 v 0.247, 2^22 0.813 v 0.819, 6,000,000 1.090 v 1.092,
// 2^23 1.409 v 1.403, 2^24 3.28 v 3.24
constexpr int lvl_items(int64_t n) { return n <= 4194304 ? 4 : 16; }
constexpr int lvl_blocks(int64_t n) { return (int)((n + SCAN_THREADS * lvl_items(n) - 1) / (SCAN_THREADS * lvl_items(n))); }

// cnt[l * nblk + block] = starts at level l <= L among the block's elements (L from the device unless
// it is fixed, L_graph >= 0).  The last block scans every level's row in place (a warp per level) and writes counts[l]
// = boxes at level l (0 past L), counts[32 + l] = first real box of level l, [32 + L + 1] = total, and
// at 56 the tree's parameters, so that the host reads counts and leaf level in one copy.
template <int ITEMS>
__global__ void __launch_bounds__(SCAN_THREADS) k_lvl_count(int64_t n, const uint64_t* __restrict__ keys, int bits,
                                                            int L_graph, TreeParams* __restrict__ tp, int nblk,
                                                            int* __restrict__ cnt, int* __restrict__ counts) {
    __shared__ int sc[32];
    const int L = L_graph >= 0 ? L_graph : tp->L;
    if (threadIdx.x < 32) sc[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = ((int64_t)blockIdx.x * SCAN_THREADS + threadIdx.x) * ITEMS;
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const int sl = base + j < n ? start_level(keys, base + j, bits) : (1 << 20);
        if (sl <= L) atomicAdd(&sc[sl], 1);
    }
    __syncthreads();
    if (threadIdx.x <= L) {
        int c = 0;
        for (int l = 0; l <= (int)threadIdx.x; ++l) c += sc[l];
        __stcg(cnt + threadIdx.x * nblk + blockIdx.x, c);
    }
    if (!last_block(&tp->ticket, nblk)) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x < 32) sc[threadIdx.x] = 0;
    __syncthreads();
    for (int l = warp; l <= L; l += SCAN_THREADS / 32) {
        int* row = cnt + (int64_t)l * nblk;
        int carry = 0;
        for (int b0 = 0; b0 < nblk; b0 += 128) {
            int v[4];  // four chunks' loads at once, then their scans
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = b0 + 32 * k + lane < nblk ? __ldcg(row + b0 + 32 * k + lane) : 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                int x = v[k];
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, x, o);
                    if (lane >= o) x += y;
                }
                if (b0 + 32 * k + lane < nblk) row[b0 + 32 * k + lane] = carry + x - v[k];
                carry += __shfl_sync(0xffffffffu, x, 31);
            }
        }
        if (lane == 0) sc[l] = carry;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        const int c = sc[lane];
        int x = c;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        counts[lane] = c;
        if (lane < COUNTS_L - 32) counts[32 + lane] = lane <= L + 1 ? x - c : 0;
        if (lane == 0) {
            counts[COUNTS_L] = L;
            counts[COUNTS_NONFINITE] = __ldcg(&tp->nonfinite);
            counts[COUNTS_L_CAP] = __ldcg(&tp->L_cap);
        }
    }
}

// Box records of every level (global index off[l] + b): key prefix, element range,
// parent (level-local, -1 at level 0) and the first child of each parent.
template <int ITEMS>
__global__ void __launch_bounds__(SCAN_THREADS) k_lvl_apply(int64_t n, const uint64_t* __restrict__ keys, int bits,
                                                            int L, int nblk, const int* __restrict__ cnt,
                                                            LevelTable off, uint64_t* __restrict__ bkey,
                                                            int* __restrict__ bbeg, int* __restrict__ bend,
                                                            int* __restrict__ bpar, int* __restrict__ bcbeg) {
    __shared__ int wsum[SCAN_THREADS / 32][32];  // starts per warp and level
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t base = ((int64_t)blockIdx.x * SCAN_THREADS + threadIdx.x) * ITEMS;
    int sl[ITEMS], prev[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        sl[j] = base + j < n ? start_level(keys, base + j, bits) : (1 << 20);
        prev[j] = 0;
    }
    const auto starts = [&](int l) {
        int t = 0;
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) t += sl[j] <= l;
        return t;
    };
    for (int l = 0; l <= L; ++l) {
        const int t = __reduce_add_sync(0xffffffffu, starts(l));
        if (lane == 0) wsum[warp][l] = t;
    }
    __syncthreads();
    for (int l = 0; l <= L; ++l) {
        const int t = starts(l);
        int run = t;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, run, o);
            if (lane >= o) run += y;
        }
        run += cnt[(int64_t)l * nblk + blockIdx.x] - t;
        for (int w = 0; w < warp; ++w) run += wsum[w][l];
        const int o = off.off[l], ou = l > 0 ? off.off[l - 1] : 0;
        const int shift = 3 * (bits - l);
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            const int64_t i = base + j;
            if (i >= n) break;
            if (sl[j] <= l) {
                const int b = run;
                bkey[o + b] = keys[i] >> shift;
                bbeg[o + b] = (int)i;
                if (b > 0) bend[o + b - 1] = (int)i;
                const int par = l > 0 ? prev[j] - 1 : -1;  // the level l-1 box holding element i
                bpar[o + b] = par;
                if (l > 0 && sl[j] <= l - 1) bcbeg[ou + par] = b;  // i starts the parent too: first child
                ++run;
            }
            prev[j] = run;  // inclusive count of level-l starts up to element i
            if (i == n - 1) bend[o + run - 1] = (int)n;
        }
    }
}

// Box arrays hold level l at [off[l], off[l] + count[l]); count (device, from k_lvl_count)
// can be smaller than the level's slot range when the offsets are capacities (the layout
// of a captured step), so every kernel over boxes skips the unused slots.

// The real boxes of levels 0..L, numbered rb = loff[l] + b (loff: the exclusive scan of the
// counts, device), and their slots gb = off[l] + b.
__device__ inline int real_level(const int* __restrict__ loff, int L, int rb) {
    int l = 0;
    while (l < L && rb >= loff[l + 1]) ++l;
    return l;
}

// children ranges: end of parent p = first child of p + 1 (or the level's box count);
// leaves have none.  P2P work items: leaf b is split into ceil(count / P2P_TILE) tiles, tcnt[b] (the
// leaf slots past the leaf count hold no leaf and get none).
__global__ void k_lvl_children(LevelTable lt, const int* __restrict__ count, const int* __restrict__ loff,
                               const int* __restrict__ bbeg, const int* __restrict__ bend, int* __restrict__ bcbeg,
                               int* __restrict__ bcend, int* __restrict__ tcnt) {
    const int nreal = loff[lt.L + 1], nl = count[lt.L], cap = lt.off[lt.L + 1] - lt.off[lt.L];
    const int stride = gridDim.x * blockDim.x, t = blockIdx.x * blockDim.x + threadIdx.x;
    for (int b = nl + t; b < cap; b += stride) tcnt[b] = 0;
    for (int rb = t; rb < nreal; rb += stride) {
        const int l = real_level(loff, lt.L, rb);
        const int p = rb - loff[l], nb = count[l], gb = lt.off[l] + p;
        if (l == lt.L) {
            bcbeg[gb] = 0;
            bcend[gb] = 0;
            tcnt[p] = (bend[gb] - bbeg[gb] + P2P_TILE - 1) / P2P_TILE;
            continue;
        }
        bcend[gb] = p + 1 < nb ? bcbeg[gb + 1] : count[l + 1];
    }
}

// 27 colleagues of every box of the levels up to lmax (binary search among its level's keys);
// the system id above the level's 3*level Morton bits is kept.  One thread per
// (box, slot), slot = ((dx + 1) 3 + (dy + 1)) 3 + (dz + 1).
__global__ void k_colleagues_all(LevelTable lt, int lmax, const int* __restrict__ count,
                                 const int* __restrict__ loff, const uint64_t* __restrict__ bkey_all,
                                 int* __restrict__ col_all) {
    const int64_t nreal = loff[lmax + 1];
    for (int64_t it = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; it < nreal * 27;
         it += (int64_t)gridDim.x * blockDim.x) {
        const int rb = (int)(it / 27), slot = (int)(it - (int64_t)rb * 27);
        const int dx = slot / 9 - 1, dy = (slot / 3) % 3 - 1, dz = slot % 3 - 1;
        const int level = real_level(loff, lt.L, rb);
        const int o = lt.off[level], nb = count[level], b = rb - loff[level];
        const uint64_t* bkey = bkey_all + o;
        const int64_t dim = 1ll << level;
        const uint64_t mask = (level > 0) ? ((~0ull) >> (64 - 3 * level)) : 0ull;
        const uint64_t full = bkey[b];
        const uint64_t sysk = (level > 0) ? ((full >> (3 * level)) << (3 * level)) : full;
        const uint64_t key = full & mask;
        const int64_t x = (int64_t)compact3(key) + dx, y = (int64_t)compact3(key >> 1) + dy,
                      z = (int64_t)compact3(key >> 2) + dz;
        int found = -1;
        if (x >= 0 && y >= 0 && z >= 0 && x < dim && y < dim && z < dim) {
            const uint64_t k2 = sysk | morton3((uint64_t)x, (uint64_t)y, (uint64_t)z);
            int lo = 0, hi = nb - 1;
            while (lo <= hi) {
                const int mid = (lo + hi) >> 1;
                const uint64_t km = bkey[mid];
                if (km == k2) {
                    found = mid;
                    break;
                }
                if (km < k2) lo = mid + 1; else hi = mid - 1;
            }
        }
        col_all[(int64_t)o * 27 + (int64_t)b * 27 + slot] = found;
    }
}

// The colleagues of the leaves from their parents': the box in a slot is the child, of the octant that the
// slot asks for, of one colleague of the parent.  A search of the level takes a chain of log2(boxes)
// dependent reads, this one five: sphere surface of 2^20, 69,700 leaves, 61 us for all levels by search, 38 us
// with the leaves this way.
__global__ void k_colleagues_leaf(LevelTable lt, const int* __restrict__ count, const uint64_t* __restrict__ bkey,
                                  const int* __restrict__ bpar, const int* __restrict__ bcbeg,
                                  const int* __restrict__ bcend, int* __restrict__ col) {
    const int o = lt.off[lt.L], po = lt.off[lt.L - 1];
    const int64_t total = (int64_t)count[lt.L] * 27;
    for (int64_t it = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; it < total;
         it += (int64_t)gridDim.x * blockDim.x) {
        const int b = (int)(it / 27), slot = (int)(it - (int64_t)b * 27);
        const int oct = (int)(bkey[o + b] & 7ull);
        // cell of the slot in units of leaves from the parent's corner: -1 .. 2 per axis
        const int cx = (oct & 1) + slot / 9 - 1, cy = (oct >> 1 & 1) + slot / 3 % 3 - 1, cz = (oct >> 2) + slot % 3 - 1;
        const int q = ((cx >> 1) + 1) * 9 + ((cy >> 1) + 1) * 3 + (cz >> 1) + 1;
        const uint64_t want = (uint64_t)((cx & 1) | (cy & 1) << 1 | (cz & 1) << 2);
        const int pc = col[((int64_t)po + bpar[o + b]) * 27 + q];
        int found = -1;
        if (pc >= 0) {
            const int c1 = bcend[po + pc];
            for (int c = bcbeg[po + pc]; c < c1; ++c)
                if ((bkey[o + c] & 7ull) == want) {
                    found = c;
                    break;
                }
        }
        col[((int64_t)o + b) * 27 + slot] = found;
    }
}

// The P2P work items (leaf, first element) at first[b], the scan of k_lvl_children's counts.
// Also the geometry of every leaf, (centre, 1 / side), for P2M and L2P: in FP64 once per leaf (a warp's
// FP64 instruction takes 16 cycles of the SM), not once per element.
__global__ void k_tile_fill(int nb, const int* __restrict__ nleaf, const int* __restrict__ bbeg,
                            const int* __restrict__ bend, const int* __restrict__ first, int2* __restrict__ tiles,
                            int level, const uint64_t* __restrict__ bkey, const SysCube* __restrict__ cubes,
                            dbl4* __restrict__ geom) {
    const int nl = min(nb, *nleaf);
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nl; b += gridDim.x * blockDim.x) {
        // key: Morton bits interleaved x, y, z from bit 0; the system id above bit 3 level
        const uint64_t key = bkey[b];
        const SysCube cb = cubes[level > 0 ? (key >> (3 * level)) : key];
        const uint64_t q = level > 0 ? key & ((~0ull) >> (64 - 3 * level)) : 0ull;
        const double h = ldexp(cb.side, -level);
        dbl4 g;
        g.x = cb.x0[0] + ((double)compact3(q) + 0.5) * h;
        g.y = cb.x0[1] + ((double)compact3(q >> 1) + 0.5) * h;
        g.z = cb.x0[2] + ((double)compact3(q >> 2) + 0.5) * h;
        g.w = 1.0 / h;
        geom[b] = g;
        int nt = (bend[b] - bbeg[b] + P2P_TILE - 1) / P2P_TILE;
        for (int j = 0; j < nt; ++j) tiles[first[b] + j] = make_int2(b, bbeg[b] + j * P2P_TILE);
    }
}

template <typename T>
__global__ void k_gather(int64_t n, const int* __restrict__ perm, const vec4_t<T>* __restrict__ x4,
                         const vec4_t<T>* __restrict__ w4, vec4_t<T>* __restrict__ xs, vec4_t<T>* __restrict__ ws) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        int j = perm[i];
        vec4_t<T> a = x4[j], b = w4[j];
        a.w = 0;
        b.w = 0;
        xs[i] = a;
        ws[i] = b;
    }
}

// ---------------------------------------------------------------------------
// Host orchestration
// ---------------------------------------------------------------------------
template <typename T>
void gather_sorted(Ctx* c, int64_t n, const int* perm, const vec4_t<T>* x4, const vec4_t<T>* w4, vec4_t<T>* xs,
                   vec4_t<T>* ws) {
    if (n <= 0) return;
    k_gather<T><<<grid_for(n, 256), 256, 0, stream_of(c)>>>(n, perm, x4, w4, xs, ws);
    count_launch(c);
    check_launch("gather");
}

int key_bits_for(int nsys) {
    int sysbits = 0;
    while ((1 << sysbits) < nsys) ++sysbits;
    return std::min(KEY_BITS, (63 - sysbits) / 3);
}

constexpr int SORT_BELOW_CAP = 5;
constexpr int COLLEAGUES_BY_PARENT = 8192;

template <typename T>
int build_tree(Ctx* c, int64_t n, int nsys, const int64_t* sysoff, const vec4_t<T>* x4, const vec4_t<T>* w4,
               TreeBufs& tb, Levels& lv, TreeParams& hp, Error& err) {
    cudaStream_t s = stream_of(c);
    const int leaf_max = ctx_leaf_max(c);
    const int64_t nn = n;
    const int bits = key_bits_for(nsys);

    // capacities that depend on n only
    ensure(c, tb.keys_a, nn * 8);
    ensure(c, tb.keys_b, nn * 8);
    ensure(c, tb.idx, nn * 4);
    ensure(c, tb.perm, nn * 4);
    ensure(c, tb.flags, nn * 4);
    ensure(c, tb.boxof, nn * 4);
    ensure(c, tb.scan_tmp, (scan_tmp_ints(nn) + 64) * 4);
    ensure(c, tb.params, sizeof(TreeParams) + (int64_t)nsys * 4);
    ensure(c, tb.counts, 64 * 4);
    ensure(c, tb.cubes, (int64_t)nsys * sizeof(SysCube));
    ensure(c, tb.sysoff, (int64_t)(nsys + 1) * 8);
    // a captured step uploads its system offsets before the capture, and again before a replay that
    // follows another tree
    const int L_graph = ctx_graph_level(c);
    const bool graph = L_graph >= 0;
    if (!graph) {
        cuda_check(cudaMemcpyAsync(tb.sysoff.ptr, sysoff, (nsys + 1) * 8, cudaMemcpyHostToDevice, s),
                   "system offsets");
        tb.offsets.assign(sysoff, sysoff + nsys + 1);
    }

    TreeParams* tp = tb.params.as<TreeParams>();
    int* counts = tb.counts.as<int>();
    cuda_check(cudaMemsetAsync(tp, 0, sizeof(TreeParams) + (int64_t)nsys * 4, s), "memset params");

    // cubes (the radix histogram buffer holds the bounding-box partials first)
    const int parts = std::max(1, std::min(1024 / nsys, (int)((nn / nsys + 1023) / 1024)));
    ensure(c, tb.hist, std::max<int64_t>(sort_hist_ints(nn) * 4, (int64_t)nsys * parts * 6 * 8));
    const int64_t* dsysoff = tb.sysoff.as<int64_t>();
    SysCube* cubes = tb.cubes.as<SysCube>();
    k_bbox<T><<<nsys * parts, 256, 0, s>>>(parts, dsysoff, x4, w4, tb.hist.as<T>(), cubes, tp,
                                           reinterpret_cast<int*>(tp + 1), core_unit(ctx_rK(c)));
    count_launch(c);
    if (nsys > 1 && ctx_rK(c) > 0.0) {
        k_cube_common<<<1, 32, 0, s>>>(cubes, nsys);
        count_launch(c);
    }

    // Keys, their stable LSD radix sort of 8-bit digits, then the leaf level.  A tree never goes below
    // L_cap = min(L_K, the level cap); ordering the keys by their prefix down to a level
    // S >= L_cap gives the same boxes at every level <= S and the same leaf level (keys that
    // differ within the prefix give the same shared level either way, and keys that share
    // their level-S box give a shared level >= S, beyond L_cap, either way).  S is the
    // previous tree's L_cap + SORT_BELOW_CAP (all levels for a context's first tree); if the new L_cap
    // exceeds it, the sort is completed (a stable sort of the prefix-sorted keys is the
    // stable sort) and the leaf level recomputed.  S is set a few levels below the previous
    // cap (SORT_BELOW_CAP), which also orders each leaf's elements spatially.
    // Keys end in keys_a, indices in perm.
    uint64_t* const keys = tb.keys_a.as<uint64_t>();
    int* const perm = tb.perm.as<int>();
    int* hist = tb.hist.as<int>();
    // all levels at once: counts per (level, block of elements), their scan, the records
    const int nblk = lvl_blocks(nn);
    const bool few = lvl_items(nn) == 4;
    Buf& lcnt = ctx_tmp(c, 0);
    ensure(c, lcnt, (int64_t)(KEY_BITS + 1) * nblk * 4);
    auto leaf_level = [&]() {
        k_leaf_level<<<grid_for(nn, 256, 152 * 4), 256, 0, s>>>(nn, leaf_max, bits, keys, tp, cubes, nsys, ctx_rK(c),
                                                                ctx_max_level(c), L_graph,
                                                                graph ? ctx_abort_word(c) : nullptr);
        count_launch(c);
        (few ? k_lvl_count<4> : k_lvl_count<16>)<<<nblk, SCAN_THREADS, 0, s>>>(nn, keys, bits, L_graph, tp, nblk,
                                                                              lcnt.as<int>(), counts);
        count_launch(c);
        check_launch("leaf level");
    };
    // a captured step's fixed leaf level needs the boxes of levels <= L_graph only: the keys ordered
    // down to S = L_graph + SORT_BELOW_CAP levels give exactly those, whatever the cap does
    int S = graph ? std::min(bits, L_graph + SORT_BELOW_CAP) : ctx_sort_levels(c);
    if (S <= 0 || S > bits) S = bits;
    const int first_pass = 3 * (bits - S) / 8;  // lower digits order nothing the tree uses
    {
        uint64_t* k0 = (8 - first_pass) % 2 == 0 ? keys : tb.keys_b.as<uint64_t>();
        uint64_t* k1 = k0 == keys ? tb.keys_b.as<uint64_t>() : keys;
        int launches = launch_keys<T>(s, nn, nsys, bits, dsysoff, cubes, x4, k0, 8 * first_pass, hist);
        launches += launch_sort(s, nn, first_pass, k0, k1, nullptr, perm, tb.idx.as<int>(), true, hist);
        while (launches-- > 0) count_launch(c);
        check_launch("keys, sort");
    }
    leaf_level();
    // host offsets of the box arrays: the actual counts (read back), or in a captured step the
    // capacities, which need no read; the kernels below take the counts from the device
    int hcounts[64] = {0};
    if (!graph) {
        auto read_counts = [&]() {
            cuda_check(cudaMemcpyAsync(hcounts, counts, sizeof(hcounts), cudaMemcpyDeviceToHost, s), "read counts");
            cuda_check(cudaStreamSynchronize(s), "sync counts");
            hp.L = hcounts[COUNTS_L];
            hp.L_cap = hcounts[COUNTS_L_CAP];
            hp.nonfinite = hcounts[COUNTS_NONFINITE];
        };
        read_counts();
        if (first_pass > 0 && hp.L_cap > S && !hp.nonfinite) {
            int launches = launch_sort(s, nn, 0, keys, tb.keys_b.as<uint64_t>(), perm, perm, tb.idx.as<int>(), false,
                                       hist);
            while (launches-- > 0) count_launch(c);
            check_launch("sort");
            cuda_check(cudaMemsetAsync(&tp->deepest_shared, 0xff, sizeof(int), s), "reset shared level");  // -1, as k_bbox sets it
            leaf_level();
            read_counts();
        }
        // the next tree orders its keys down to SORT_BELOW_CAP levels below the cap: the leaves
        // only need one, the rest keeps consecutive elements of a leaf (the near-field warp tiles)
        // spatially compact
        ctx_sort_levels(c) = std::min(bits, hp.L_cap + SORT_BELOW_CAP);
        if (hp.nonfinite) {
            err = {LHV_ENONFINITE, "non-finite position or strength"};
            return LHV_ENONFINITE;
        }
    }
    const int L = graph ? L_graph : hp.L;
    lv.L = L;
    lv.n = nn;
    hp.bits = bits;
    hp.nsys = nsys;

    // capacity of every level: boxes per level <= min(n, nsys 8^l)
    lv.cap_off[0] = 0;
    for (int l = 0; l <= L; ++l) {
        int64_t cap = nn;
        if (3 * l < 40) cap = std::min<int64_t>(nn, (int64_t)nsys << (3 * l));
        lv.cap_off[l + 1] = lv.cap_off[l] + (int)cap;
    }
    const int64_t tot_cap = lv.cap_off[L + 1];
    ensure(c, tb.bkey, tot_cap * 8);
    ensure(c, tb.bbeg, tot_cap * 4);
    ensure(c, tb.bend, tot_cap * 4);
    ensure(c, tb.bparent, tot_cap * 4);
    ensure(c, tb.bcbeg, tot_cap * 4);
    ensure(c, tb.bcend, tot_cap * 4);

    int* loff = counts + 32;  // off[0 .. L+1] of the actual counts, on the device
    lv.off[0] = 0;
    if (graph) {
        for (int l = 0; l < MAX_LEVELS; ++l) {
            lv.nbox[l] = (l <= L) ? lv.cap_off[l + 1] - lv.cap_off[l] : 0;
            lv.off[l + 1] = lv.off[l] + lv.nbox[l];
        }
    } else {
        for (int l = 0; l < MAX_LEVELS; ++l) {
            lv.nbox[l] = (l <= L) ? hcounts[l] : 0;
            lv.off[l + 1] = lv.off[l] + lv.nbox[l];
        }
        for (int l = 0; l < MAX_LEVELS; ++l) lv.real[l] = lv.nbox[l];
        lv.leaves = lv.nbox[L];
    }
    LevelTable lt{};
    lt.L = L;
    for (int l = 0; l <= L + 1 && l <= MAX_LEVELS; ++l) lt.off[l] = lv.off[l];
    lt.off[L + 2 <= MAX_LEVELS + 1 ? L + 2 : MAX_LEVELS + 1] = lv.off[L + 1];
    (few ? k_lvl_apply<4> : k_lvl_apply<16>)<<<nblk, SCAN_THREADS, 0, s>>>(
        nn, keys, bits, L, nblk, lcnt.as<int>(), lt, tb.bkey.as<uint64_t>(), tb.bbeg.as<int>(), tb.bend.as<int>(),
        tb.bparent.as<int>(), tb.bcbeg.as<int>());
    count_launch(c);
    check_launch("levels");
    const int64_t nbt = lv.off[L + 1];
    const int nl = lv.nbox[L], o = lv.off[L];
    int* tcnt = tb.flags.as<int>();
    k_lvl_children<<<grid_for(nbt, 256), 256, 0, s>>>(lt, counts, loff, tb.bbeg.as<int>(), tb.bend.as<int>(),
                                                      tb.bcbeg.as<int>(), tb.bcend.as<int>(), tcnt);
    count_launch(c);
    ensure(c, tb.bcol, nbt * 27 * 4);
    // a few thousand boxes are searched in one launch, of more the leaves (most of them) take the short way
    const bool by_parent = L >= 1 && nl >= COLLEAGUES_BY_PARENT;
    k_colleagues_all<<<grid_for((by_parent ? o : nbt) * 27, 128), 128, 0, s>>>(
        lt, by_parent ? L - 1 : L, counts, loff, tb.bkey.as<uint64_t>(), tb.bcol.as<int>());
    count_launch(c);
    if (by_parent) {
        k_colleagues_leaf<<<grid_for((int64_t)nl * 27, 128), 128, 0, s>>>(lt, counts, tb.bkey.as<uint64_t>(),
                                                                          tb.bparent.as<int>(), tb.bcbeg.as<int>(),
                                                                          tb.bcend.as<int>(), tb.bcol.as<int>());
        count_launch(c);
    }
    check_launch("children, colleagues");

    // P2P work items over the leaves
    int* first = tb.boxof.as<int>();
    ensure(c, tb.tile_count, 16);
    exclusive_scan(c, nl, tcnt, first, tb.scan_tmp.as<int>(), tb.tile_count.as<int>());
    ensure(c, tb.tiles, (nl + nn / P2P_TILE + 1) * 8);
    ensure(c, tb.geom, (int64_t)nl * sizeof(dbl4));
    k_tile_fill<<<grid_for(nl, 256), 256, 0, s>>>(nl, counts + L, tb.bbeg.as<int>() + o, tb.bend.as<int>() + o, first,
                                                  tb.tiles.as<int2>(), L, tb.bkey.as<uint64_t>() + o, cubes,
                                                  tb.geom.as<dbl4>());
    count_launch(c);
    check_launch("tiles");
    return LHV_OK;
}


// Rows [off[l], off[l] + count[l]) of levels l0..l1 (row_len elements each, row r at
// data + (r - row0) row_len) set to `value`: the rows of real boxes only, whatever the
// slot layout.
template <typename T>
__global__ void k_fill_level_rows(LevelTable lt, const int* __restrict__ count, int l0, int l1, int64_t row_len,
                                  int64_t row0, T* __restrict__ data, T value) {
    for (int l = l0; l <= l1; ++l) {
        const int64_t n = (int64_t)count[l] * row_len;
        T* base = data + ((int64_t)lt.off[l] - row0) * row_len;
        for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
            base[e] = value;
    }
}

template <typename T>
void fill_level_rows(Ctx* c, const Levels& lv, const int* dcount, int l0, int l1, int64_t row_len, int64_t row0,
                     T* data, T value) {
    if (l1 < l0) return;
    LevelTable lt{};
    lt.L = lv.L;
    for (int l = 0; l <= lv.L + 1 && l <= MAX_LEVELS + 1; ++l) lt.off[l] = lv.off[l];
    int64_t cap = 0;
    for (int l = l0; l <= l1; ++l) cap = std::max<int64_t>(cap, (int64_t)lv.nbox[l] * row_len);
    k_fill_level_rows<T><<<grid_for(cap, 256, 152 * 16), 256, 0, stream_of(c)>>>(lt, dcount, l0, l1, row_len, row0,
                                                                                   data, value);
    count_launch(c);
    check_launch("fill rows");
}

template void fill_level_rows<float>(Ctx*, const Levels&, const int*, int, int, int64_t, int64_t, float*, float);
template void fill_level_rows<double>(Ctx*, const Levels&, const int*, int, int, int64_t, int64_t, double*, double);
template void fill_level_rows<int>(Ctx*, const Levels&, const int*, int, int, int64_t, int64_t, int*, int);

template int build_tree<float>(Ctx*, int64_t, int, const int64_t*, const float4*, const float4*, TreeBufs&, Levels&,
                               TreeParams&, Error&);
template int build_tree<double>(Ctx*, int64_t, int, const int64_t*, const dbl4*, const dbl4*, TreeBufs&, Levels&,
                                TreeParams&, Error&);
template void gather_sorted<float>(Ctx*, int64_t, const int*, const float4*, const float4*, float4*, float4*);
template void gather_sorted<double>(Ctx*, int64_t, const int*, const dbl4*, const dbl4*, dbl4*, dbl4*);

}  // namespace lhv

// ---------------------------------------------------------------------------
// Cube, Morton keys and sort without allocation (lhv_morton_sort_noalloc)
// ---------------------------------------------------------------------------
// The same kernels as the first part of build_tree for one system, with every
// temporary array in one fixed file-scope device array instead of context
// buffers.  The caller's output arrays are one side of the sort's ping-pong.
namespace lhv {
namespace {

constexpr int64_t NOALLOC_MAX_N = LHV_NOALLOC_MAX_N;
constexpr int NOALLOC_MAX_PARTS = 1024;
// the most sort tiles: at the largest n, or where a thread's items change
constexpr int64_t NOALLOC_HIST_INTS = std::max(sort_hist_ints(NOALLOC_MAX_N), sort_hist_ints(SORT_FEW_MAX));

constexpr int64_t align256(int64_t b) { return (b + 255) / 256 * 256; }
// scratch regions (byte offsets)
constexpr int64_t NA_KEYS = 0;                                                   // uint64[max n]
constexpr int64_t NA_IDX = NA_KEYS + align256(NOALLOC_MAX_N * 8);                // int32[max n]
constexpr int64_t NA_HIST = NA_IDX + align256(NOALLOC_MAX_N * 4);                // int32[256 * (tiles + 1)]
constexpr int64_t NA_PART = NA_HIST + align256(NOALLOC_HIST_INTS * 4);                // float[parts][6]
constexpr int64_t NA_SYSOFF = NA_PART + align256((int64_t)NOALLOC_MAX_PARTS * 6 * 4);  // int64[2]
constexpr int64_t NA_CUBE = NA_SYSOFF + 256;                                     // SysCube
constexpr int64_t NA_PARAMS = NA_CUBE + align256(sizeof(SysCube));               // TreeParams
constexpr int64_t NA_TICKET = NA_PARAMS + align256(sizeof(TreeParams));          // int32[1]
constexpr int64_t NA_BYTES = NA_TICKET + 256;

static __device__ __align__(256) unsigned char g_noalloc_scratch[NA_BYTES];

// Address of g_noalloc_scratch per device, looked up by the first call on that device.
constexpr int NOALLOC_MAX_DEVICES = 64;
unsigned char* g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {};

// The only state that must start at zero: the non-finite flag (all of
// TreeParams is cleared) and the block counter; also writes the system offsets {0, n}.
__global__ void k_noalloc_init(int64_t n, int64_t* __restrict__ sysoff, TreeParams* __restrict__ tp,
                               int* __restrict__ ticket) {
    if (threadIdx.x == 0) {
        sysoff[0] = 0;
        sysoff[1] = n;
        *tp = TreeParams{};
        *ticket = 0;
    }
}

}  // namespace
}  // namespace lhv

extern "C" int lhv_morton_sort_noalloc(int64_t n, const float* x4, const float* w4, uint64_t* keys, int32_t* perm,
                                       void* cuda_stream) {
    using namespace lhv;
    if (n < 0) return LHV_EINVAL;
    if (n > NOALLOC_MAX_N) return LHV_ETOOBIG;
    if (n == 0) return LHV_OK;
    if (!x4 || !keys || !perm) return LHV_EINVAL;
    if ((reinterpret_cast<uintptr_t>(x4) | reinterpret_cast<uintptr_t>(w4)) % 16 != 0 ||
        reinterpret_cast<uintptr_t>(keys) % 8 != 0 || reinterpret_cast<uintptr_t>(perm) % 4 != 0)
        return LHV_EINVAL;
    // An error left pending by the caller's earlier work would be read back (and cleared)
    // by the launch check below and reported as this call's; refuse instead, leaving it
    // in place for the caller.
    if (cudaPeekAtLastError() != cudaSuccess) return LHV_ECUDA;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return LHV_ECUDA;
    if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) return LHV_EUNSUPPORTED;
    if (!g_noalloc_ptr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) {
            cudaGetLastError();
            return LHV_ECUDA;
        }
        g_noalloc_ptr[dev] = static_cast<unsigned char*>(p);
    }
    unsigned char* base = g_noalloc_ptr[dev];
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    int64_t* sysoff = reinterpret_cast<int64_t*>(base + NA_SYSOFF);
    SysCube* cube = reinterpret_cast<SysCube*>(base + NA_CUBE);
    TreeParams* tp = reinterpret_cast<TreeParams*>(base + NA_PARAMS);
    float* part = reinterpret_cast<float*>(base + NA_PART);
    int* hist = reinterpret_cast<int*>(base + NA_HIST);
    int* ticket = reinterpret_cast<int*>(base + NA_TICKET);
    const float4* x = reinterpret_cast<const float4*>(x4);
    const float4* w = reinterpret_cast<const float4*>(w4);

    const int bits = key_bits_for(1);
    const int parts = std::max(1, std::min(NOALLOC_MAX_PARTS, (int)((n + 4095) / 4096)));
    k_noalloc_init<<<1, 32, 0, s>>>(n, sysoff, tp, ticket);
    k_bbox<float><<<parts, 256, 0, s>>>(parts, sysoff, x, w, part, cube, tp, ticket, 0.0);
    // 8 passes of 8 bits; the even count leaves the keys in the caller's array
    launch_keys<float>(s, n, 1, bits, sysoff, cube, x, keys, 0, hist);
    launch_sort(s, n, 0, keys, reinterpret_cast<uint64_t*>(base + NA_KEYS), nullptr, perm,
                reinterpret_cast<int*>(base + NA_IDX), true, hist);
    if (cudaGetLastError() != cudaSuccess) return LHV_ECUDA;
    TreeParams hp{};
    if (cudaMemcpyAsync(&hp, tp, sizeof(TreeParams), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess) {
        cudaGetLastError();
        return LHV_ECUDA;
    }
    return hp.nonfinite ? LHV_ENONFINITE : LHV_OK;
}
