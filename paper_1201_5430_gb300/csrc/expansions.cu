// P2M (Sec. 4.3), M2M and L2L with conversion (Sec. 4.4), L2P (Sec. 4.5).
//
// All coefficient vectors are in the scaled real layout described in
// operators.cu; the operator tables come from there, and every dense map runs
// through the grouped GEMM of group_gemm.cu.  Per-element work builds
// the normalised regular solid harmonics Q_n^m(rho) = rho^n sqrt((n-m)!/(n+m)!)
// P_n^m(cos theta) e^{i m phi} on the fly by their three-term recurrences, with
// rho = (x - box centre) / h, so no element ever stores p^2 values.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "lhv_group.cuh"
#include "lhv_internal.cuh"

namespace lhv {

namespace {

// Coefficients of the recurrences of Q_n^m for n, m < p (they depend on (n, m)
// only), formed once per context in double precision (lhv::build_qtab) and copied to shared memory by
// each block (p = 12: 312 reals; formed by every block they took it 7,000 cycles of the FP64 pipe):
//   Q_m^m     = cm[m] (x + i y) Q_{m-1}^{m-1},        cm[m] = -sqrt((2m - 1) / (2m)),
//   Q_{m+1}^m = c1[m] z Q_m^m,                        c1[m] = sqrt(2m + 1),
//   Q_n^m     = A[m][n] z Q_{n-1}^m - B[m][n] r^2 Q_{n-2}^m,
//     A = (2n - 1) / sqrt((n + m)(n - m)),  B = sqrt((n + m - 1)(n - m - 1) / ((n + m)(n - m))).
// The table takes qtab_reals(p) reals of the block's dynamic shared memory.
template <typename T>
struct QTab {
    T *A, *B, *cm, *c1;
    int p;
};

__host__ __device__ inline int qtab_reals(int p) { return 2 * p * p + 2 * p; }

template <typename T>
__device__ inline QTab<T> load_qtab(T* base, const T* __restrict__ src, int p) {
    for (int i = threadIdx.x; i < qtab_reals(p); i += blockDim.x) base[i] = src[i];
    return QTab<T>{base, base + p * p, base + 2 * p * p, base + 2 * p * p + p, p};
}

// Walks every (n, m), 0 <= m <= n < p, of the recurrence of Q_n^m at (x, y, z)
// and calls f(n, m, Re Q, Im Q).  State is O(1).  par = 0 or 1 keeps the orders m of that
// parity only (the diagonal Q_m^m is still advanced through every m).
template <typename T, typename F>
__device__ inline void for_each_Q(int p, T x, T y, T z, const QTab<T>& q, F&& f, int par = -1) {
    const T r2 = x * x + y * y + z * z;
    T dre = 1, dim = 0;  // Q_m^m
    for (int m = 0; m < p; ++m) {
        if (m > 0) {
            const T c = q.cm[m];
            T nre = c * (x * dre - y * dim);
            T nim = c * (x * dim + y * dre);
            dre = nre;
            dim = nim;
        }
        if (par >= 0 && (m & 1) != par) continue;
        f(m, m, dre, dim);
        if (m + 1 >= p) continue;
        const T c1 = q.c1[m] * z;
        T pre = dre, pim = dim;             // Q_{n-2}
        T qre = c1 * dre, qim = c1 * dim;   // Q_{n-1} = Q_{m+1}^m
        f(m + 1, m, qre, qim);
        for (int n = m + 2; n < p; ++n) {
            const T a = q.A[m * q.p + n] * z;
            const T b = q.B[m * q.p + n] * r2;
            T nre = a * qre - b * pre;
            T nim = a * qim - b * pim;
            pre = qre;
            pim = qim;
            qre = nre;
            qim = nim;
            f(n, m, qre, qim);
        }
    }
}

// The same walk for N points at once: f(n, m, sum of w Re Q, sum of w Im Q).  A table entry is read
// once for the N points, and their chains interleave.
template <int N, typename T, typename F>
__device__ inline void for_each_Q_sum(int p, const T (&x)[N], const T (&y)[N], const T (&z)[N], const T (&w)[N],
                                      const QTab<T>& q, F&& f, int par) {
    T r2[N], dre[N], dim[N];  // Q_m^m w
#pragma unroll
    for (int i = 0; i < N; ++i) {
        r2[i] = x[i] * x[i] + y[i] * y[i] + z[i] * z[i];
        dre[i] = w[i];
        dim[i] = 0;
    }
    const auto put = [&](int n, int m, const T(&re)[N], const T(&im)[N]) {
        T a = re[0], b = im[0];
#pragma unroll
        for (int i = 1; i < N; ++i) {
            a += re[i];
            b += im[i];
        }
        f(n, m, a, b);
    };
    for (int m = 0; m < p; ++m) {
        if (m > 0) {
            const T c = q.cm[m];
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const T nre = c * (x[i] * dre[i] - y[i] * dim[i]);
                dim[i] = c * (x[i] * dim[i] + y[i] * dre[i]);
                dre[i] = nre;
            }
        }
        if ((m & 1) != par) continue;
        put(m, m, dre, dim);
        if (m + 1 >= p) continue;
        T pre[N], pim[N], qre[N], qim[N];  // Q_{n-2}, Q_{n-1}
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const T c1 = q.c1[m] * z[i];
            pre[i] = dre[i];
            pim[i] = dim[i];
            qre[i] = c1 * dre[i];
            qim[i] = c1 * dim[i];
        }
        put(m + 1, m, qre, qim);
        for (int n = m + 2; n < p; ++n) {
            const T A = q.A[m * q.p + n], B = q.B[m * q.p + n];
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const T a = A * z[i], b = B * r2[i];
                const T nre = a * qre[i] - b * pre[i];
                const T nim = a * qim[i] - b * pim[i];
                pre[i] = qre[i];
                pim[i] = qim[i];
                qre[i] = nre;
                qim[i] = nim;
            }
            put(n, m, qre, qim);
        }
    }
}

// out[r] = sum of the sparse map's row r over `in` (shared memory, in[cols] = 0), f(r, sum): the warps of
// a block take the slices in turn.
template <typename T, typename F>
__device__ inline void sparse_rows(const SellView<T>& m, const T* in, int warp, int nwarps, F&& f) {
    const int lane = threadIdx.x & 31;
    for (int q = warp; 32 * q < m.rows; q += nwarps) {
        const int b = m.sptr[q], e = m.sptr[q + 1];
        T acc = 0;
#pragma unroll 4
        for (int i = b + lane; i < e; i += 32) {
            const SellEntry<T> n = m.ent[i];
            acc += n.val * in[n.col];
        }
        const int r = 32 * q + lane;
        if (r < m.rows) f(r, acc);
    }
}

// ---------------------------------------------------------------------------
// P2M, part 1 (per leaf): W_k = sum_e w_{e,k} g_hat(rho_e), where
// g_hat_n^m = nu_n^m R_n^{-m}(-rho) = i^m conj(Q_n^m(rho)), rho = (x - c)/h.
// Part 2 is the grouped GEMM  M_hat = (1/h) [G_x G_y G_z] [W_x; W_y; W_z]
// with G_k the scaled real form of Eq. eve4 for w = i_k.
// ---------------------------------------------------------------------------
// Blocks of 128 threads over chunks of up to 128 elements, or of 64 threads over 32 where the mean leaf
// is small: a block's shared memory then holds the rows of 32 elements, and an SM 11 blocks instead
// of two (p = 12).  P2M of the sphere surface of 2^20 (15 elements a leaf) 1.86 -> 0.48 ms, of the ring
// of 32,768 (10) 0.140 -> 0.060; of the leapfrog pair (440), where an entry of the harmonics is
// now read once for its three strengths, 2.12 -> 1.45 ms at p = 16.
constexpr int P2M_THREADS = 128, P2M_SMALL = 64;
constexpr int P2M_SMALL_LEAF = 48;  // mean elements per leaf up to which the small blocks are taken
constexpr int p2m_max_out(int threads) { return (24 * 24 + threads - 1) / threads; }  // (n, m) entries per thread, p <= 24

// Row stride of the staged harmonics: odd, so that the lanes of a warp, each writing entry k of
// its own element's row, fall in 32 different shared-memory banks (a stride of p^2 = 256 put all
// 32 in one bank).
__host__ __device__ inline int p2m_row_stride(int P) { return P | 1; }

// Shared memory of k_p2m_w and the elements per chunk: the largest chunk (`most`, at least 32,
// halved) whose rows, strengths and recurrence table fit in 80 KB (two blocks per SM).
template <typename T>
size_t p2m_smem(int p, int most, int& chunk) {
    const size_t row = (size_t)p2m_row_stride(p * p) + 4;
    chunk = most;
    while (chunk > 32 && sizeof(T) * (chunk * row + qtab_reals(p)) > 80 * 1024) chunk /= 2;
    return sizeof(T) * (chunk * row + qtab_reals(p));
}

// Gauss points of a segment that one walk of the harmonics takes.  One at a time, every point added to the
// element's row in shared memory: P2M of the filament ring of 2^18 (p = 16, eight points) 1.21 ms; four at a
// time (two in FP64, by registers) 0.59.
template <typename T> constexpr int SEG_POINTS = sizeof(T) == 4 ? 4 : 2;

// Work items are the tiles of at most P2P_TILE consecutive elements of one leaf
// (the near-field tiles), so a crowded leaf is spread over several blocks; each
// block adds its partial W into the leaf's (zeroed) W with atomics.
// NC = 3: W of the vortex elements (rows of 3P per leaf); NC = 1: the scalar reference
// case, monopoles q: the scaled S coefficients of Eq. rsbf5, (1/h) sum_e q_e g_hat(rho_e),
// written straight into the leaf's multipole row (ldw reals per leaf).
// SEG (NC = 3): the element is a filament node owning the segment x -> x + l with
// circulation Gamma, ws = (l, Gamma): W gets (Gamma l / (8 pi h)) sum_j w_j g_hat(rho_j) at
// the Gauss-Legendre points x + l (1 + xi_j) / 2 (Eqs. vf5, vf6).
template <typename T, int NC, bool SEG, int THREADS>
__global__ void __launch_bounds__(THREADS) k_p2m_w(const int* __restrict__ ntiles_dev,
                                                     const int2* __restrict__ tiles, const dbl4* __restrict__ geom,
                                                     const T* __restrict__ qtab, const int* __restrict__ bend,
                                                     const vec4_t<T>* __restrict__ xs,
                                                     const vec4_t<T>* __restrict__ ws, const T* __restrict__ qs,
                                                     T* __restrict__ Wout, int64_t ldw, int p, int chunk,
                                                     GaussRule rule = GaussRule{}) {
    extern __shared__ __align__(32) unsigned char smem_raw[];
    static_assert(THREADS % 64 == 0, "warps pair up by the parity of m");
    constexpr int MAX_OUT = p2m_max_out(THREADS);
    const int P = p * p, gs = p2m_row_stride(P);
    const int par = (threadIdx.x >> 5) & 1;  // parity of the orders m this warp's harmonics take
    constexpr int WS = NC == 3 ? 4 : 1;      // reals per strength: one vector read
    T* wk = reinterpret_cast<T*>(smem_raw);  // [chunk][WS]: strength / h
    T* gh = wk + (size_t)chunk * WS;         // [chunk][gs]: the harmonics of an element in a row
    const int ntiles = *ntiles_dev;
    const QTab<T> qt = load_qtab(gh + (size_t)chunk * gs, qtab, p);  // visible after the tile loop's first barrier
    // a block takes a contiguous range of tiles; the tiles of a leaf are consecutive, so the
    // partial W of a leaf is summed over its tiles in registers and added once per leaf
    const int t_lo = (int)((int64_t)ntiles * blockIdx.x / gridDim.x);
    const int t_hi = (int)((int64_t)ntiles * (blockIdx.x + 1) / gridDim.x);
    T acc[MAX_OUT][NC];  // entries j = threadIdx.x + q THREADS of the current leaf's NC rows of W
#pragma unroll
    for (int q = 0; q < MAX_OUT; ++q)
#pragma unroll
        for (int k = 0; k < NC; ++k) acc[q][k] = 0;
    auto flush = [&](int leaf) {
        T* Wb = Wout + (int64_t)leaf * ldw;
#pragma unroll
        for (int q = 0; q < MAX_OUT; ++q) {
            const int j = threadIdx.x + q * THREADS;
#pragma unroll
            for (int k = 0; k < NC; ++k) {
                if (j < P) atomicAdd(Wb + k * P + j, acc[q][k]);
                acc[q][k] = 0;
            }
        }
    };
    int cur = -1;
    for (int t = t_lo; t < t_hi; ++t) {
        const int2 tw = tiles[t];
        const int b = tw.x;
        if (b != cur) {
            if (cur >= 0) flush(cur);
            cur = b;
        }
        const dbl4 bg = geom[b];
        const T invh = (T)bg.w;
        const int e0 = tw.y, e1 = min(bend[b], tw.y + P2P_TILE);
        for (int c0 = e0; c0 < e1; c0 += chunk) {
            const int ne = min(chunk, e1 - c0);
            __syncthreads();
            // two warps per 32 elements: the even-numbered one takes the orders m of even
            // parity, its neighbour the odd ones (disjoint entries of the row; the parity is
            // uniform across a warp, so its lanes do not diverge)
            for (int e = (threadIdx.x >> 6) * 32 + (threadIdx.x & 31); e < ne; e += blockDim.x >> 1) {
                vec4_t<T> xv = xs[c0 + e];
                if (par == 0) {
                    if constexpr (NC == 3) {
                        const vec4_t<T> wv = ws[c0 + e];
                        // M_hat carries 1/h (P2M scaling); a segment's strength is Gamma l / (8 pi)
                        const T sc = SEG ? wv.w * (T)(0.039788735772973833942) * invh : invh;  // 1/(8 pi)
                        wk[e * 4 + 0] = wv.x * sc;
                        wk[e * 4 + 1] = wv.y * sc;
                        wk[e * 4 + 2] = wv.z * sc;
                    } else {
                        wk[e] = qs[c0 + e] * invh;
                    }
                }
                T* g = gh + (size_t)e * gs;
                // i^m conj(Q) to the element's row, or added to it
                auto put = [&](int n, int m, T qr, T qi, bool add) {
                    T re, im;
                    switch (m & 3) {
                        case 0: re = qr; im = -qi; break;
                        case 1: re = qi; im = qr; break;
                        case 2: re = -qr; im = qi; break;
                        default: re = -qi; im = -qr; break;
                    }
                    const int k0 = m == 0 ? n * n : n * n + 2 * m - 1;
                    g[k0] = add ? g[k0] + re : re;
                    if (m > 0) g[k0 + 1] = add ? g[k0 + 1] + im : im;
                };
                if constexpr (SEG) {
                    // the Gauss points of the segment (Eq. vf6) SEG_POINTS at a time, in FP64 up to their rounding
                    const vec4_t<T> wv = ws[c0 + e];
                    const double ox = ((double)xv.x - bg.x) * bg.w, oy = ((double)xv.y - bg.y) * bg.w,
                                 oz = ((double)xv.z - bg.z) * bg.w;
                    const double lx = (double)wv.x * bg.w, ly = (double)wv.y * bg.w, lz = (double)wv.z * bg.w;
                    constexpr int N = SEG_POINTS<T>;
                    for (int j0 = 0; j0 < rule.nq; j0 += N) {
                        T rx[N], ry[N], rz[N], wq[N];
#pragma unroll
                        for (int i = 0; i < N; ++i) {  // past the last point: the last again, of weight zero
                            const int j = min(j0 + i, rule.nq - 1);
                            const double t = 0.5 * (1.0 + rule.xi[j]);
                            rx[i] = (T)fma(t, lx, ox);
                            ry[i] = (T)fma(t, ly, oy);
                            rz[i] = (T)fma(t, lz, oz);
                            wq[i] = j0 + i < rule.nq ? (T)rule.w[j] : (T)0;
                        }
                        for_each_Q_sum<N>(p, rx, ry, rz, wq, qt,
                                          [&](int n, int m, T qr, T qi) { put(n, m, qr, qi, j0 > 0); }, par);
                    }
                } else {
                    const T rx = (T)(((double)xv.x - bg.x) * bg.w), ry = (T)(((double)xv.y - bg.y) * bg.w),
                            rz = (T)(((double)xv.z - bg.z) * bg.w);
                    for_each_Q<T>(p, rx, ry, rz, qt, [&](int n, int m, T qr, T qi) { put(n, m, qr, qi, false); }, par);
                }
            }
            __syncthreads();
            // an entry of the harmonics serves the NC strengths of its element
#pragma unroll
            for (int q = 0; q < MAX_OUT; ++q) {
                const int j = threadIdx.x + q * THREADS;
                if (j >= P) break;
                T s[NC];
#pragma unroll
                for (int k = 0; k < NC; ++k) s[k] = 0;
#pragma unroll 4
                for (int e = 0; e < ne; ++e) {
                    const T g = gh[(size_t)e * gs + j];
                    if constexpr (NC == 3) {
                        const vec4_t<T> w = *reinterpret_cast<const vec4_t<T>*>(wk + e * 4);
                        s[0] += w.x * g;
                        s[1] += w.y * g;
                        s[2] += w.z * g;
                    } else {
                        s[0] += wk[e] * g;
                    }
                }
#pragma unroll
                for (int k = 0; k < NC; ++k) acc[q][k] += s[k];
            }
        }
    }
    if (cur >= 0) flush(cur);
}

// P2M, part 2 (per leaf): M_hat = G W with G the sparse P2M map of Eq. eve4; one block per leaf, W
// staged in shared memory.
constexpr int P2M_APPLY_THREADS = 96;
template <typename T>
__global__ void __launch_bounds__(P2M_APPLY_THREADS) k_p2m_apply(const int* __restrict__ nleaf_dev,
                                                                const T* __restrict__ W, int P, SellView<T> g,
                                                                T* __restrict__ mult, int64_t ld) {
    extern __shared__ __align__(32) unsigned char smem_raw[];
    T* w = reinterpret_cast<T*>(smem_raw);  // [3P], then a zero
    const int nleaf = *nleaf_dev;
    if (threadIdx.x == 0) w[3 * P] = 0;
    for (int b = blockIdx.x; b < nleaf; b += gridDim.x) {
        __syncthreads();
        for (int i = threadIdx.x; i < 3 * P; i += blockDim.x) w[i] = W[(int64_t)b * 3 * P + i];
        __syncthreads();
        T* out = mult + (int64_t)b * ld;
        sparse_rows(g, w, threadIdx.x >> 5, P2M_APPLY_THREADS / 32, [&](int r, T v) { out[r] = v; });
    }
}

// ---------------------------------------------------------------------------
// L2P (per tile of a leaf; the 12 coefficient vectors cf = E L_hat of v_k (Eq. evf3)
// and u_lk = D_{i_l} v_k (Eq. dt3) come from the leaf's local expansion through the
// sparse map E, in shared memory):
//   v_k = (1/h) c_k . b(rho),   u_lk = (1/h^2) c_{3+3l+k} . b(rho),
//   s_k = sum_l w_l u_lk (Eq. evf6),
// b = real form of R_hat = nu R:  b[n^2] = R_hat_n^0,  2 Re R_hat_n^m,  -2 Im R_hat_n^m,
// R_hat_n^m = (-1)^n i^m Q_n^m.
// ---------------------------------------------------------------------------
constexpr int L2P_THREADS = 128;

// Vector j = r / P of row r = j P + i (r < 12 P) of the L2P map without a division a row: the upper half of r per, per =
// floor((2^32 - 1) / P) + 1, exact for 2 <= P <= 24^2.  At P = 1 that reciprocal is 2^32, past its 32 bits, and j = r.
__device__ inline unsigned row_reciprocal(int P) { return P > 1 ? 0xffffffffu / (unsigned)P + 1u : 0u; }
__device__ inline int row_vector(int r, int P, unsigned per) { return P > 1 ? (int)__umulhi((unsigned)r, per) : r; }

// GRAD: the 12 vectors of v and grad v, else the 3 of v (sfar unused)
template <typename T, int THREADS, bool GRAD>
__global__ void __launch_bounds__(THREADS) k_l2p_eval(const int* __restrict__ ntiles_dev,
                                                        const int2* __restrict__ tiles, const dbl4* __restrict__ geom,
                                                        const T* __restrict__ qtab, const int* __restrict__ bend,
                                                        const vec4_t<T>* __restrict__ xs,
                                                        const vec4_t<T>* __restrict__ ws, const T* __restrict__ loc,
                                                        int64_t ld, SellView<T> e, vec4_t<T>* __restrict__ vfar,
                                                        vec4_t<T>* __restrict__ sfar, int p) {
    constexpr int NV = GRAD ? 12 : 3, CS = GRAD ? 12 : 4;  // vectors, and their stride in shared memory
    extern __shared__ __align__(32) unsigned char smem_raw[];
    const int P = p * p;
    T* cf = reinterpret_cast<T*>(smem_raw);  // [P][CS]
    T* lh = cf + CS * P;                     // [2P] the leaf's local expansion, then a zero
    const int ntiles = *ntiles_dev;
    if (threadIdx.x == 0) lh[2 * P] = 0;
    const unsigned per = row_reciprocal(P);
    const QTab<T> qt = load_qtab(lh + 2 * P + 4, qtab, p);  // visible after the tile loop's first barrier
    // a block takes a contiguous range of tiles; the tiles of a leaf are consecutive, so the
    // leaf's coefficient vectors are staged once per leaf, not once per tile
    const int t_lo = (int)((int64_t)ntiles * blockIdx.x / gridDim.x);
    const int t_hi = (int)((int64_t)ntiles * (blockIdx.x + 1) / gridDim.x);
    int staged = -1;
    for (int t = t_lo; t < t_hi; ++t) {
        const int2 tw = tiles[t];
        const int b = tw.x;
        const dbl4 bg = geom[b];
        if (b != staged) {
            __syncthreads();
            for (int i = threadIdx.x; i < 2 * P; i += blockDim.x) lh[i] = loc[(int64_t)b * ld + i];
            __syncthreads();
            sparse_rows(e, lh, threadIdx.x >> 5, THREADS / 32, [&](int r, T v) {  // r = j P + i: vector j, entry i
                const int j = row_vector(r, P, per), i = r - j * P;
                cf[i * CS + j] = v;
            });
            __syncthreads();
            staged = b;
        }
        const T invh = (T)bg.w;
        const int e1 = min(bend[b], tw.y + P2P_TILE);
        for (int e = tw.y + threadIdx.x; e < e1; e += blockDim.x) {
            const vec4_t<T> xv = xs[e];
            const T rx = (T)(((double)xv.x - bg.x) * bg.w), ry = (T)(((double)xv.y - bg.y) * bg.w),
                    rz = (T)(((double)xv.z - bg.z) * bg.w);
            T acc[NV];
#pragma unroll
            for (int j = 0; j < NV; ++j) acc[j] = 0;
            for_each_Q<T>(p, rx, ry, rz, qt, [&](int n, int m, T qr, T qi) {
                T re, im;  // (-1)^n i^m Q
                switch (m & 3) {
                    case 0: re = qr; im = qi; break;
                    case 1: re = -qi; im = qr; break;
                    case 2: re = -qr; im = -qi; break;
                    default: re = qi; im = -qr; break;
                }
                if (n & 1) {
                    re = -re;
                    im = -im;
                }
                if (m == 0) {
                    const T* c = cf + (n * n) * CS;
#pragma unroll
                    for (int j = 0; j < NV; ++j) acc[j] += c[j] * re;
                } else {
                    const T* c1 = cf + (n * n + 2 * m - 1) * CS;
                    const T* c2 = c1 + CS;
                    const T b1 = 2 * re, b2 = -2 * im;
#pragma unroll
                    for (int j = 0; j < NV; ++j) acc[j] += c1[j] * b1 + c2[j] * b2;
                }
            });
            vec4_t<T> v;
            v.x = acc[0] * invh;
            v.y = acc[1] * invh;
            v.z = acc[2] * invh;
            v.w = 0;
            vfar[e] = v;
            if constexpr (GRAD) {
                const vec4_t<T> wv = ws[e];
                const T invh2 = invh * invh;
                vec4_t<T> s;
                s.x = (wv.x * acc[3] + wv.y * acc[6] + wv.z * acc[9]) * invh2;
                s.y = (wv.x * acc[4] + wv.y * acc[7] + wv.z * acc[10]) * invh2;
                s.z = (wv.x * acc[5] + wv.y * acc[8] + wv.z * acc[11]) * invh2;
                s.w = 0;
                sfar[e] = s;
            }
        }
    }
}


// Scalar reference case: phi = L_hat . b(rho) (no factor: R coefficients carry h^n / nu)
// and grad phi_k = (1/h) c_k . b(rho), with c_k the velocity rows of the L2P map (Eq. evf3)
// applied to (L_hat, 0): with chi = 0, v = grad phi (Eq. 4).  Lanes of the output: grad phi
// in x, y, z, phi in w.
template <typename T, int THREADS>
__global__ void __launch_bounds__(THREADS) k_l2p_scalar(const int* __restrict__ ntiles_dev,
                                                          const int2* __restrict__ tiles, const dbl4* __restrict__ geom,
                                                        const T* __restrict__ qtab, const int* __restrict__ bend,
                                                          const vec4_t<T>* __restrict__ xs, const T* __restrict__ loc,
                                                          int64_t ld, SellView<T> e, vec4_t<T>* __restrict__ pgfar,
                                                          int p) {
    extern __shared__ __align__(32) unsigned char smem_raw[];
    const int P = p * p;
    T* cf = reinterpret_cast<T*>(smem_raw);  // [P][4]
    T* lh = cf + 4 * P;                      // [2P] (L_hat, 0), then a zero
    const int ntiles = *ntiles_dev;
    if (threadIdx.x == 0) lh[2 * P] = 0;
    const unsigned per = row_reciprocal(P);
    const QTab<T> qt = load_qtab(lh + 2 * P + 4, qtab, p);
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int2 tw = tiles[t];
        const int b = tw.x;
        const dbl4 bg = geom[b];
        __syncthreads();
        for (int i = threadIdx.x; i < 2 * P; i += blockDim.x) lh[i] = i < P ? loc[(int64_t)b * ld + i] : (T)0;
        __syncthreads();
        // vector j = 0: phi itself, 1..3: rows of v_x, v_y, v_z
        for (int i = threadIdx.x; i < P; i += blockDim.x) cf[i * 4] = lh[i];
        sparse_rows(e, lh, threadIdx.x >> 5, THREADS / 32, [&](int r, T v) {
            const int j = row_vector(r, P, per), i = r - j * P;
            cf[i * 4 + 1 + j] = v;
        });
        __syncthreads();
        const T invh = (T)bg.w;
        const int e1 = min(bend[b], tw.y + P2P_TILE);
        for (int el = tw.y + threadIdx.x; el < e1; el += blockDim.x) {
            const vec4_t<T> xv = xs[el];
            const T rx = (T)(((double)xv.x - bg.x) * bg.w), ry = (T)(((double)xv.y - bg.y) * bg.w),
                    rz = (T)(((double)xv.z - bg.z) * bg.w);
            T acc[4] = {0, 0, 0, 0};
            for_each_Q<T>(p, rx, ry, rz, qt, [&](int n, int m, T qr, T qi) {
                T re, im;  // (-1)^n i^m Q
                switch (m & 3) {
                    case 0: re = qr; im = qi; break;
                    case 1: re = -qi; im = qr; break;
                    case 2: re = -qr; im = -qi; break;
                    default: re = qi; im = -qr; break;
                }
                if (n & 1) {
                    re = -re;
                    im = -im;
                }
                if (m == 0) {
                    const T* c = cf + (n * n) * 4;
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[j] += c[j] * re;
                } else {
                    const T* c1 = cf + (n * n + 2 * m - 1) * 4;
                    const T* c2 = c1 + 4;
                    const T b1 = 2 * re, b2 = -2 * im;
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[j] += c1[j] * b1 + c2[j] * b2;
                }
            });
            vec4_t<T> o;
            o.x = acc[1] * invh;
            o.y = acc[2] * invh;
            o.z = acc[3] * invh;
            o.w = acc[0];
            pgfar[el] = o;
        }
    }
}

}  // namespace

template <typename T>
void build_qtab(Ctx* c, int p, Buf& dst) {
    std::vector<T> h((size_t)qtab_reals(p), (T)0);
    T *A = h.data(), *B = A + p * p, *cm = B + p * p, *c1 = cm + p;
    for (int m = 0; m < p; ++m) {
        for (int n = m + 2; n < p; ++n) {
            const double d = (double)((n + m) * (n - m));
            A[m * p + n] = (T)((2 * n - 1) / std::sqrt(d));
            B[m * p + n] = (T)std::sqrt((double)((n + m - 1) * (n - m - 1)) / d);
        }
        cm[m] = m > 0 ? (T)-std::sqrt((2.0 * m - 1.0) / (2.0 * m)) : (T)0;
        c1[m] = (T)std::sqrt(2.0 * m + 1.0);
    }
    upload(c, dst, h.data(), (int64_t)(h.size() * sizeof(T)), "recurrence table");
}

// Blocks of a persistent kernel: as many as are resident at once, at most `items`.
template <typename K>
static int resident_grid(K kernel, int threads, size_t smem, int64_t items) {
    int per_sm = 1, sms = 152, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
    return (int)std::max<int64_t>(1, std::min<int64_t>(items, (int64_t)sms * std::max(per_sm, 1)));
}

// W of the leaves (rows of ldw reals, zeroed) by blocks that suit their mean size.
template <typename T, int NC, bool SEG>
static void launch_p2m_w(Ctx* c, const TreeBufs& tb, const Levels& lv, int p, const T* qtab, const vec4_t<T>* xs, const vec4_t<T>* ws,
                         const T* qs, T* W, int64_t ldw, const GaussRule& rule) {
    const int L = lv.L, o = lv.off[L];
    auto launch = [&](auto threads, int most) {
        constexpr int TH = decltype(threads)::value;
        int chunk;
        const size_t smem = p2m_smem<T>(p, most, chunk);
        auto kernel = k_p2m_w<T, NC, SEG, TH>;
        cuda_check(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem), "p2m attr");
        kernel<<<tile_grid(kernel, TH, smem, lv), TH, smem, stream_of(c)>>>(
            tb.tile_count.as<int>(), tb.tiles.as<int2>(), tb.geom.as<dbl4>(), qtab, tb.bend.as<int>() + o, xs, ws, qs, W, ldw, p, chunk, rule);
        count_launch(c);
        check_launch("p2m w");
    };
    if (lv.n <= (int64_t)lv.leaves * P2M_SMALL_LEAF) launch(std::integral_constant<int, P2M_SMALL>{}, 32);
    else launch(std::integral_constant<int, P2M_THREADS>{}, 128);
}

template <typename T>
static void launch_p2m_apply(Ctx* c, const Plan<T>& pl, const TreeBufs& tb, const Levels& lv, const T* W, T* mult) {
    const int L = lv.L, P = pl.p[L] * pl.p[L];
    const size_t smem = sizeof(T) * (3 * P + 1);
    k_p2m_apply<T><<<resident_grid(k_p2m_apply<T>, P2M_APPLY_THREADS, smem, lv.nbox[L]), P2M_APPLY_THREADS, smem,
                     stream_of(c)>>>(tb.counts.as<int>() + L, W, P, pl.p2m_sp, mult + (int64_t)lv.off[L] * pl.ld, pl.ld);
    count_launch(c);
    check_launch("p2m apply");
}

// Blocks of a kernel whose blocks take contiguous ranges of the near-field tiles: one tile a block
// where that is less than eight a resident block (their unevenness would set the time: L2P of
// the FP64 ring of 32,768, 1.8 tiles a resident block, 1.10 ms against 0.92), 16 blocks an SM where a
// leaf holds several tiles (P2M, L2P of the leapfrog pair, 440 elements a leaf: 1.8, 1.86 ms with the
// resident blocks, 1.45, 1.74 with 16), else those resident at once (sphere surface, 15 a leaf:
// 0.48, 1.32 ms against 0.54, 1.59 with 16, before the sparse maps were packed).
constexpr int BIG_LEAF = 64;
template <typename K>
static int tile_grid(K kernel, int threads, size_t smem, const Levels& lv) {
    const int64_t tiles = lv.nbox[lv.L] + lv.n / P2P_TILE + 1;
    const int resident = resident_grid(kernel, threads, smem, tiles);
    if (lv.leaves + lv.n / P2P_TILE < 8 * (int64_t)resident) return grid_for(tiles, 1, 8 * resident);
    if (lv.n > (int64_t)lv.leaves * BIG_LEAF) return grid_for(tiles, 1, 152 * 16);
    return resident;
}

// Threads of an L2P block of three or four vectors for the mean leaf: f(integral_constant).  Narrow
// blocks put more leaves on an SM (scalar cube, 32 a leaf: 0.29 ms against 0.35 with 128 threads); with
// twelve vectors the sparse map takes half of the work and wants the wide block (sphere
// surface 1.18 with 64 against 1.06, cloud of 24 a leaf 0.087 against 0.080).
template <typename F>
static void l2p_threads(const Levels& lv, F&& f) {
    const int64_t nl = lv.leaves;
    if (lv.n <= nl * 32) f(std::integral_constant<int, 32>{});
    else if (lv.n <= nl * 64) f(std::integral_constant<int, 64>{});
    else f(std::integral_constant<int, L2P_THREADS>{});
}

template <typename T>
void run_p2m(Ctx* c, const Plan<T>& pl, const TreeBufs& tb, const Levels& lv, const vec4_t<T>* xs,
             const vec4_t<T>* ws, T* W, T* mult) {
    const int L = lv.L, P = pl.p[L] * pl.p[L];
    fill_level_rows<T>(c, lv, tb.counts.as<int>(), L, L, 3 * P, lv.off[L], W, (T)0);  // W of the real leaves
    launch_p2m_w<T, 3, false>(c, tb, lv, pl.p[L], pl.qtab, xs, ws, nullptr, W, 3 * P, GaussRule{});
    launch_p2m_apply<T>(c, pl, tb, lv, W, mult);
}

// chunk width of the list of M2M and L2L: the MMA's where L2L may run on the tensor cores, else set by the
// widest input
template <typename T>
static int oct_nc(const Plan<T>& pl) {
    if (pl.l2l_tiles) return TC_PAIRS;
    int pmax = 1;
    for (int l = 2; l <= pl.L; ++l) pmax = std::max(pmax, pl.p[l]);
    return std::min(16, gemm_nc<T>(2 * pmax * pmax));  // levels hold few boxes: many short items
}

// One level of L2L on the tensor cores (LHV_TF32X3, one p a multiple of 4), true if it ran there.  The
// grouped GEMM streams 250 KB of operator for every 16 boxes (p = 12), here one block T for 128; L2L, ms: sphere
// surface of 2^20 1.38 -> 0.19, offset rings of 2^21 (p = 16) 0.55 -> 0.15, 16 blob systems 0.26 -> 0.079, a
// filament's eleven levels 0.75 -> 0.32, ring of 32,768 0.12 -> 0.084.  A level of few boxes (b boxes with b p^4
// up to OCT_TC_MIN) stays with the grouped GEMM, which splits its sums over the idle SMs: about 12 us at p = 12, 17
// at p = 16, where the MMA's one pass over T and its epilogue take 29 and 36.
//
// M2M stays with the grouped GEMM at every level.  Against the exact map of the same inputs the split products put
// 1.06e-7 on a level's multipoles of a sphere surface (p = 8 to 16) where FP32 puts 5.1e-8 (scalar case 6.5e-8 and
// 4.8e-8), whether or not the cross products of all K come first; L2L's locals come out nearer than FP32's,
// 6.0e-8 against 0.6 to 1.2e-7.  On the tensor cores M2M of the sphere surface of 2^20 took 0.24 ms, here 1.50.
constexpr int64_t OCT_TC_MIN = 16000000;
template <typename T>
static bool l2l_tc(Ctx* c, const Plan<T>& pl, const Grouped& gp, const GemmArgs<T>& a) {
    if constexpr (sizeof(T) == 4) {
        const int64_t P = pl.p[pl.L] * pl.p[pl.L];
        if (pl.l2l_tiles && a.pairs_hint * P * P > OCT_TC_MIN) {
            run_tc_trans(c, TRANS_L2L, gp, a.g0, a.g1, pl.p[pl.L], pl.scalar, pl.l2l_tiles, a.in, a.out, a.ldin,
                         ctx_err_flag(c));
            return true;
        }
    }
    return false;
}

template <typename T>
void run_m2m(Ctx* c, const Plan<T>& pl, const TreeBufs& tb, const Levels& lv, Grouped& gp, T* mult) {
    const int L = lv.L;
    if (L < 3) return;
    // parents of the levels 2 .. L-1 accumulate atomically
    fill_level_rows<T>(c, lv, tb.counts.as<int>(), 2, L - 1, pl.ld, 0, mult, (T)0);
    oct_list(c, tb, lv, gp, oct_nc(pl));
    for (int l = L - 1; l >= 2; --l) {
        const int Pout = pl.p[l] * pl.p[l], Pin = pl.p[l + 1] * pl.p[l + 1];
        GemmArgs<T> a{};
        a.g0 = (l + 1 - 3) * 8;
        a.g1 = a.g0 + 8;
        a.ops = pl.m2m[l];
        a.ops_mod = 8;
        a.R = pl.rows(Pout);  // scalar case: the translation block alone, no chi
        a.C = pl.rows(Pin);
        a.psplit = pl.split_out(Pout);
        a.psplit_c = pl.split_out(Pin);
        a.in = mult;
        a.ldin = pl.ld;
        a.out = mult;
        a.ldout = pl.ld;
        a.mode = GEMM_ATOMIC;
        a.scale = (T)1;
        a.pairs_hint = lv.real[l + 1];
        a.between = BETWEEN_LEVELS;
        run_group_gemm<T>(c, gp, a);
    }
}

template <typename T>
void run_l2l(Ctx* c, const Plan<T>& pl, const Levels& lv, const Grouped& gp, T* loc) {
    const int L = lv.L;
    if (L < 3) return;
    for (int l = 2; l < L; ++l) {
        const int Pout = pl.p[l + 1] * pl.p[l + 1], Pin = pl.p[l] * pl.p[l];
        GemmArgs<T> a{};
        a.g0 = (l + 1 - 3) * 8;
        a.g1 = a.g0 + 8;
        a.ops = pl.l2l[l + 1];
        a.ops_mod = 8;
        a.R = pl.rows(Pout);
        a.C = pl.rows(Pin);
        a.psplit = pl.split_out(Pout);
        a.psplit_c = pl.split_out(Pin);
        a.in = loc;
        a.ldin = pl.ld;
        a.out = loc;
        a.ldout = pl.ld;
        a.mode = GEMM_ATOMIC;  // one parent per child: the plain sum, issued without waiting for the old value
        a.scale = (T)1;
        a.pairs_hint = lv.real[l + 1];
        a.between = BETWEEN_LEVELS | BETWEEN_SWAPPED;
        if (!l2l_tc(c, pl, gp, a)) run_group_gemm<T>(c, gp, a);
    }
}

template <typename T>
void run_l2p(Ctx* c, const Plan<T>& pl, const TreeBufs& tb, const Levels& lv, const vec4_t<T>* xs,
             const vec4_t<T>* ws, const T* loc, vec4_t<T>* vfar, vec4_t<T>* sfar) {
    const int L = lv.L, o = lv.off[L], p = pl.p[L], P = p * p;
    auto launch = [&](auto threads, auto grad) {
        constexpr int TH = decltype(threads)::value;
        constexpr bool GRAD = decltype(grad)::value;
        const size_t smem = sizeof(T) * ((GRAD ? 14 : 6) * P + 4 + qtab_reals(p));
        auto kernel = k_l2p_eval<T, TH, GRAD>;
        cuda_check(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem), "l2p attr");
        kernel<<<tile_grid(kernel, TH, smem, lv), TH, smem, stream_of(c)>>>(
            tb.tile_count.as<int>(), tb.tiles.as<int2>(), tb.geom.as<dbl4>(), pl.qtab, tb.bend.as<int>() + o, xs, ws, loc + (int64_t)o * pl.ld, pl.ld, pl.l2p_sp, vfar, sfar, p);
        count_launch(c);
        check_launch("l2p");
    };
    if (sfar) launch(std::integral_constant<int, L2P_THREADS>{}, std::true_type{});
    else l2p_threads(lv, [&](auto th) { launch(th, std::false_type{}); });
}


// Filament segments (Sec. 5.3): W by Gauss-Legendre quadrature along each node's segment,
// then the P2M map of Eq. eve4 as for vortex elements (Eqs. vf5-vf7).
template <typename T>
void run_p2m_segments(Ctx* c, const Plan<T>& pl, const TreeBufs& tb, const Levels& lv, const vec4_t<T>* xs,
                      const vec4_t<T>* seg, const GaussRule& rule, T* W, T* mult) {
    const int L = lv.L, P = pl.p[L] * pl.p[L];
    fill_level_rows<T>(c, lv, tb.counts.as<int>(), L, L, 3 * P, lv.off[L], W, (T)0);
    launch_p2m_w<T, 3, true>(c, tb, lv, pl.p[L], pl.qtab, xs, seg, nullptr, W, 3 * P, rule);
    launch_p2m_apply<T>(c, pl, tb, lv, W, mult);
}

// Scalar reference case: P2M of the monopoles straight into the leaf multipoles.
template <typename T>
void run_p2m_scalar(Ctx* c, const Plan<T>& pl, const TreeBufs& tb, const Levels& lv, const vec4_t<T>* xs,
                    const T* qs, T* mult) {
    const int L = lv.L;
    fill_level_rows<T>(c, lv, tb.counts.as<int>(), L, L, pl.ld, 0, mult, (T)0);
    launch_p2m_w<T, 1, false>(c, tb, lv, pl.p[L], pl.qtab, xs, nullptr, qs, mult + (int64_t)lv.off[L] * pl.ld, pl.ld,
                              GaussRule{});
}

template <typename T>
void run_l2p_scalar(Ctx* c, const Plan<T>& pl, const TreeBufs& tb, const Levels& lv, const vec4_t<T>* xs,
                    const T* loc, vec4_t<T>* pgfar) {
    const int L = lv.L, o = lv.off[L], p = pl.p[L], P = p * p;
    const size_t smem = sizeof(T) * (6 * P + 4 + qtab_reals(p));
    l2p_threads(lv, [&](auto threads) {
        constexpr int TH = decltype(threads)::value;
        auto kernel = k_l2p_scalar<T, TH>;
        cuda_check(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem), "l2p attr");
        kernel<<<tile_grid(kernel, TH, smem, lv), TH, smem, stream_of(c)>>>(
            tb.tile_count.as<int>(), tb.tiles.as<int2>(), tb.geom.as<dbl4>(), pl.qtab, tb.bend.as<int>() + o, xs, loc + (int64_t)o * pl.ld, pl.ld, pl.l2p_sp, pgfar, p);
        count_launch(c);
        check_launch("l2p scalar");
    });
}

#define LHV_INST(T)                                                                                              \
    template void build_qtab<T>(Ctx*, int, Buf&);                                                                \
    template void run_p2m<T>(Ctx*, const Plan<T>&, const TreeBufs&, const Levels&, const vec4_t<T>*,            \
                             const vec4_t<T>*, T*, T*);                                                         \
    template void run_m2m<T>(Ctx*, const Plan<T>&, const TreeBufs&, const Levels&, Grouped&, T*);              \
    template void run_l2l<T>(Ctx*, const Plan<T>&, const Levels&, const Grouped&, T*);                          \
    template void run_l2p<T>(Ctx*, const Plan<T>&, const TreeBufs&, const Levels&, const vec4_t<T>*,            \
                             const vec4_t<T>*, const T*, vec4_t<T>*, vec4_t<T>*);                      \
    template void run_p2m_scalar<T>(Ctx*, const Plan<T>&, const TreeBufs&, const Levels&, const vec4_t<T>*,     \
                                    const T*, T*);                                                               \
    template void run_p2m_segments<T>(Ctx*, const Plan<T>&, const TreeBufs&, const Levels&, const vec4_t<T>*,   \
                                      const vec4_t<T>*, const GaussRule&, T*, T*);                               \
    template void run_l2p_scalar<T>(Ctx*, const Plan<T>&, const TreeBufs&, const Levels&, const vec4_t<T>*,     \
                                    const T*, vec4_t<T>*);
LHV_INST(float)
LHV_INST(double)
#undef LHV_INST

}  // namespace lhv
