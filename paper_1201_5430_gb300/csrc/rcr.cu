// M2L by rotation - coaxial translation - back rotation (RCR, Sec. 4.4, Eq. rcr1) for the
// two-potential form: FP32 or FP64 products on the CUDA cores, tables built in FP64.
//
// A translation by t = target - source centre runs in the frame whose z axis is t.  With
// Q a rotation taking i_z to t/|t| (r = Q r'), each potential's coefficients are rotated
// degree by degree (the 2n+1 reals of degree n mix only among themselves), translated
// along z by |t| (the coaxial (S|R) map of Eq. mr3 keeps every order m apart), converted
// by the coaxial form of Eq. drt10 (Eq. rcr1: phi~ = phi^ + i|t|(m/n) chi^, chi~ = chi^ -
// |t|/(n+1) chi^_{n+1}) and rotated back with Q^T.
//
// Q = Rz(phi) Ry(theta) with (theta, phi) the polar angles of t, so the forward rotation of
// the coefficients is Y(theta) Z(phi) and the back rotation Z(-phi) Y(-theta):
//   Z: a turn about z multiplies c_n^m by a phase e^{+-i m phi}: a 2 x 2 rotation of (Re, Im)
//      of each order, the same for every degree;
//   Y: a turn about y commutes with the reflection y -> -y, so the 2n+1 real functions of
//      degree n split into an even class (m = 0; Re of even m; Im of odd m; n + 1 of them)
//      and an odd class (the other n), and Y is block diagonal in them: (n+1)^2 + n^2
//      multiply-adds per degree instead of (2n+1)^2.
// The coaxial translation is the same real matrix A_m for phi and chi, Re and Im; the
// conversion is then an elementwise pass.  Per pair about 2 x 2 x (2/3) p^3 for the
// rotations and (2/3) 2 p^3 for the coaxial products, against 3 p^4 for the fused table.
//
// Tables.  In the scaled real basis (see operators.cu) the coefficients are, up to one
// constant per degree, those of the unit-normalised harmonics, so the blocks have entries
// of order one.  Every rotation block is found from its definition, f(R r') = sum_j x'_j
// g_j(r'):  X_{j'j} = <g_j o R, g_j'> / <g_j', g_j'>  over the unit sphere, by a quadrature
// exact for products of two harmonics of degree < p (p Gauss-Legendre nodes in cos(theta),
// 2p equispaced azimuths), in FP64; the structure (2 x 2 phases, even / odd classes) is
// then read out and every entry outside it checked to be zero.  The coaxial block A_m of
// each distinct |t| (24) is read out of the fused table ([[T, C12 T], [0, C22 T]],
// operators.cu) of t = |t| i_z, and its conversion blocks C12 T, C22 T are checked against
// the conversion coefficients used here (scaled basis, box side 1):
//   phi~ = phi^ + i tau chi^,  tau = |t| m / n;   chi~_n = chi^_n - sigma chi^_{n+1},
//   sigma = |t| sqrt((n + 1 - m)(n + 1 + m)) / (n + 1)   (the chi^_p term dropped).
//
// Products: the resident CTAs walk contiguous ranges of chunks of the grouped pair list (pairs
// bucketed by offset slot, m2l_prepare), hold the slot's tables in shared memory, gather NC source
// multipoles into A and run
//   A -transposed-> C -Z-> B -Y-> C -coaxial-> B -conversion-> C -Y-> B -Z-> C -transposed-> B -> locals
// on [row][pair] buffers, the Y and coaxial stages as register-tiled products (4 output rows x 4 pairs
// per thread, one row x 2 pairs in FP64).  The next chunk's gather is issued after the first Z stage.  Where a box's row is a
// multiple of 16 bytes (FP64; FP32 of even p from 4 on) the gather copies 16 bytes at a time to [pair][row] and a
// pair's result leaves as one bulk addition; the index work of 4-byte copies and of one
// atomicAdd per coefficient was a third of the kernel's instructions.  Products at p = 12, FP32, ms with 4-byte
// copies and atomicAdd (odd p still) / so: cloud of 100,003, 0.64 M pairs 1.45 / 1.19; ring of 2^18,
// 0.50 M pairs 1.14 / 0.94; FP64 ring of 2^15 9.15 / 9.11 (4 x 4 tiles).  What bounds it: issue slots and the
// shared-memory pipe, each at about 60 % (two 16-byte reads for 16 multiply-adds), and the seven
// barriers a chunk with 16 warps an SM; 384 and 512 threads a CTA were slower (1.23, 1.47).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <map>
#include <utility>
#include <vector>

#include "lhv_group.cuh"
#include "lhv_internal.cuh"
#include "tc_common.cuh"

namespace lhv {

namespace {

constexpr int RB_THREADS = 256;
constexpr int RB_BATCH = 8;  // quadrature points per pass of the rotation builder
constexpr int RA_THREADS = 256;
constexpr int SMEM_MAX = 227 * 1024;     // dynamic shared memory of one CTA
constexpr int SMEM_PER_SM = 228 * 1024;  // of one SM (1 KB of it reserved per resident CTA)
constexpr double PI = 3.14159265358979323846;

__host__ __device__ inline int pad4(int k) { return (k + 3) & ~3; }

// members of the classes of degree n, by local index j (0 .. 2n) of the real layout
// (j = 0: m = 0; j = 2m - 1, 2m: Re, Im of order m)
__host__ __device__ inline int even_member(int i) { return i == 0 ? 0 : 2 * i - 1 + (i & 1); }  // i = 0 .. n
__host__ __device__ inline int odd_member(int i) { return 2 * i + 1 + (i & 1); }                 // i = 0 .. n-1
__host__ __device__ inline bool is_even(int j) {
    if (j == 0) return true;
    const int m = (j + 1) / 2, im = (j & 1) == 0;
    return ((m & 1) != 0) == (im != 0);
}

// floats of the Y blocks of degrees < n (even block [n+1][pad4(n+1)], odd [n][pad4(n)])
__host__ __device__ inline int y_off(int n) {
    int o = 0;
    for (int k = 0; k < n; ++k) o += (k + 1) * pad4(k + 1) + k * pad4(k);
    return o;
}
__host__ __device__ inline int coax_off(int p, int m) {
    int o = 0;
    for (int k = 0; k < m; ++k) o += (p - k) * pad4(p - k);
    return o;
}

struct RotJob {
    double q[9];  // row-major rotation R: u' = R u
    int r_basis;  // 1: R basis, 0: S basis
    int pad;
};

__device__ inline double2 cmul(double2 a, double2 b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }

// Scaled real basis functions of degree < p at the unit vector u, into g[n*n + j]:
// j = 0: the m = 0 function; j = 2m - 1, 2m: the functions multiplying Re and Im of the
// order-m coefficient.  Up to a constant per degree, R_n^m nu_n^m = i^m Q_n^m and
// S_n^m / nu_n^m = (-i)^m Q_n^m on the unit sphere (Q_n^m the normalised solid harmonic
// of operators.cu), and a real function sum_m c_n^m F_n^m is c^0 F^0 + sum_{m>0}
// (2 Re c^m Re F^m - 2 Im c^m Im F^m).
__device__ void real_basis(double x, double y, double z, int p, bool r_basis, double* g) {
    double2 qmm = make_double2(1.0, 0.0);
    for (int m = 0; m < p; ++m) {
        if (m > 0) {
            const double c = -sqrt((2.0 * m - 1.0) / (2.0 * m));
            qmm = cmul(make_double2(c * x, c * y), qmm);
        }
        // i^m (R) or (-i)^m (S)
        const int k = r_basis ? (m & 3) : ((4 - (m & 3)) & 3);
        double2 q1 = qmm, q2 = make_double2(0.0, 0.0);
        for (int n = m; n < p; ++n) {
            double2 q;
            if (n == m) {
                q = qmm;
            } else if (n == m + 1) {
                const double s = sqrt(2.0 * m + 1.0) * z;
                q = make_double2(s * qmm.x, s * qmm.y);
            } else {
                const double a = (2.0 * n - 1.0) / sqrt((double)(n + m) * (n - m));
                const double b = sqrt((double)(n + m - 1) * (n - m - 1) / ((double)(n + m) * (n - m)));
                q = make_double2(a * z * q1.x - b * q2.x, a * z * q1.y - b * q2.y);
            }
            if (n > m) {
                q2 = q1;
                q1 = q;
            }
            double2 f;
            switch (k) {
                case 0: f = q; break;
                case 1: f = make_double2(-q.y, q.x); break;
                case 2: f = make_double2(-q.x, -q.y); break;
                default: f = make_double2(q.y, -q.x); break;
            }
            if (m == 0) {
                g[n * n] = f.x;
            } else {
                g[n * n + 2 * m - 1] = 2.0 * f.x;
                g[n * n + 2 * m] = -2.0 * f.y;
            }
        }
    }
}

// One CTA per job: the dense rotation blocks of degrees < p, out[job][base_n + j' (2n+1) + j]
// = X_{j'j} (FP64), base_n = sum_{k<n} (2k+1)^2.
__global__ void __launch_bounds__(RB_THREADS) k_rcr_rotations(const RotJob* __restrict__ jobs, int p,
                                                              const double* __restrict__ xq,
                                                              const double* __restrict__ wq,
                                                              double* __restrict__ out) {
    extern __shared__ __align__(16) double rb_smem[];
    const int P = p * p;
    const int NE = p * (4 * p * p - 1) / 3;  // sum of (2n+1)^2
    double* acc = rb_smem;                   // [NE]
    double* nrm = acc + NE;                  // [P]
    double* G = nrm + P;                     // [RB_BATCH][2][P]
    double* wt = G + RB_BATCH * 2 * P;       // [RB_BATCH]
    const RotJob jb = jobs[blockIdx.x];
    const int tid = threadIdx.x;
    for (int e = tid; e < NE; e += RB_THREADS) acc[e] = 0.0;
    for (int e = tid; e < P; e += RB_THREADS) nrm[e] = 0.0;
    const int NA = 2 * p, NP = p * NA;
    for (int b0 = 0; b0 < NP; b0 += RB_BATCH) {
        __syncthreads();
        if (tid < 2 * RB_BATCH) {
            const int b = tid >> 1, rot = tid & 1, pt = b0 + b;
            double* g = G + (b * 2 + rot) * P;
            if (pt < NP) {
                const int k = pt / NA, l = pt - k * NA;
                const double ct = xq[k], st = sqrt(fmax(0.0, 1.0 - ct * ct));
                const double ph = PI * (2.0 * l + 1.0) / NA;
                double ux = st * cos(ph), uy = st * sin(ph), uz = ct;
                if (rot) {
                    const double vx = jb.q[0] * ux + jb.q[1] * uy + jb.q[2] * uz;
                    const double vy = jb.q[3] * ux + jb.q[4] * uy + jb.q[5] * uz;
                    const double vz = jb.q[6] * ux + jb.q[7] * uy + jb.q[8] * uz;
                    ux = vx;
                    uy = vy;
                    uz = vz;
                } else {
                    wt[b] = wq[k];
                }
                real_basis(ux, uy, uz, p, jb.r_basis != 0, g);
            } else {
                for (int j = 0; j < P; ++j) g[j] = 0.0;
                if (!rot) wt[b] = 0.0;
            }
        }
        __syncthreads();
        int n = 0, base = 0;
        for (int e = tid; e < NE; e += RB_THREADS) {
            while (e >= base + (2 * n + 1) * (2 * n + 1)) {
                base += (2 * n + 1) * (2 * n + 1);
                ++n;
            }
            const int w = 2 * n + 1, el = e - base, jp = el / w, j = el - jp * w;
            double s = 0.0;
#pragma unroll
            for (int b = 0; b < RB_BATCH; ++b) s += wt[b] * G[(b * 2 + 1) * P + n * n + j] * G[b * 2 * P + n * n + jp];
            acc[e] += s;
        }
        for (int j = tid; j < P; j += RB_THREADS) {
            double s = 0.0;
#pragma unroll
            for (int b = 0; b < RB_BATCH; ++b) s += wt[b] * G[b * 2 * P + j] * G[b * 2 * P + j];
            nrm[j] += s;
        }
    }
    __syncthreads();
    double* dst = out + (int64_t)blockIdx.x * NE;
    int n = 0, base = 0;
    for (int e = tid; e < NE; e += RB_THREADS) {
        while (e >= base + (2 * n + 1) * (2 * n + 1)) {
            base += (2 * n + 1) * (2 * n + 1);
            ++n;
        }
        const int w = 2 * n + 1, jp = (e - base) / w;
        dst[e] = acc[e] / nrm[n * n + jp];
    }
}

__device__ inline void atomic_max_pos(float* a, float v) {
    atomicMax(reinterpret_cast<int*>(a), __float_as_int(v));  // non-negative floats order as ints
}

// One CTA per slot: the slot's table [Yf | Yb | Zf | Zb] (reals) from the dense blocks of its
// four jobs (job_of[4 s + 0]: Y(theta), S basis; + 1: Y(-theta), R basis; + 2: Z(phi), S basis;
// + 3: Z(-phi), R basis); *resid = the largest entry outside the structure.
template <typename T>
__global__ void k_rcr_pack(const double* __restrict__ dense, const int* __restrict__ job_of, int p, int per_slot,
                           T* __restrict__ out, float* __restrict__ resid) {
    const int NE = p * (4 * p * p - 1) / 3;
    const int ysz = y_off(p);
    T* dst = out + (int64_t)blockIdx.x * per_slot;
    float worst = 0.f;
    for (int which = 0; which < 2; ++which) {  // Y blocks
        const double* X = dense + (int64_t)job_of[blockIdx.x * 4 + which] * NE;
        T* d = dst + which * ysz;
        for (int n = 0; n < p; ++n) {
            const int w = 2 * n + 1, base = n * (4 * n * n - 1) / 3;
            const double* Xn = X + base;
            const int ne = n + 1, no = n, Pe = pad4(ne), Po = pad4(no);
            T* de = d + y_off(n);
            T* dod = de + ne * Pe;
            for (int e = threadIdx.x; e < w * w; e += blockDim.x) {
                const int jp = e / w, j = e - jp * w;
                if (is_even(jp) != is_even(j)) worst = fmaxf(worst, (float)fabs(Xn[e]));
            }
            for (int e = threadIdx.x; e < ne * Pe; e += blockDim.x) {
                const int i = e / Pe, o = e - i * Pe;
                de[e] = o < ne ? (T)Xn[even_member(o) * w + even_member(i)] : (T)0;
            }
            for (int e = threadIdx.x; e < no * Po; e += blockDim.x) {
                const int i = e / Po, o = e - i * Po;
                dod[e] = o < no ? (T)Xn[odd_member(o) * w + odd_member(i)] : (T)0;
            }
        }
    }
    for (int which = 0; which < 2; ++which) {  // Z: [m][4] = (Re<-Re, Re<-Im, Im<-Re, Im<-Im)
        const double* X = dense + (int64_t)job_of[blockIdx.x * 4 + 2 + which] * NE;
        T* d = dst + 2 * ysz + which * 4 * p;
        for (int n = 0; n < p; ++n) {
            const int w = 2 * n + 1, base = n * (4 * n * n - 1) / 3;
            const double* Xn = X + base;
            for (int e = threadIdx.x; e < w * w; e += blockDim.x) {
                const int jp = e / w, j = e - jp * w;
                const int mp = (jp + 1) / 2, m = (j + 1) / 2;
                if (mp != m) {
                    worst = fmaxf(worst, (float)fabs(Xn[e]));
                } else if (m == 0) {
                    worst = fmaxf(worst, (float)fabs(Xn[e] - 1.0));
                } else {
                    // the same 2 x 2 block at every degree: compare with degree p - 1
                    const int N = p - 1, W = 2 * N + 1, bN = N * (4 * N * N - 1) / 3;
                    const int jpN = 2 * m - 1 + ((jp + 1) & 1), jN = 2 * m - 1 + ((j + 1) & 1);
                    worst = fmaxf(worst, (float)fabs(Xn[e] - X[bN + jpN * W + jN]));
                }
            }
        }
        for (int e = threadIdx.x; e < 4 * p; e += blockDim.x) {
            const int m = e / 4, k = e & 3;
            T v = 0;
            if (m > 0) {
                const int N = p - 1, W = 2 * N + 1, bN = N * (4 * N * N - 1) / 3;
                const int jp = 2 * m - 1 + (k >> 1), j = 2 * m - 1 + (k & 1);
                v = (T)X[bN + jp * W + j];
            }
            d[e] = v;
        }
    }
    if (worst > 0.f) atomic_max_pos(resid, worst);
}

// One CTA per distance: [A blocks | tau, sigma] of the coaxial translation at |t| = dist.
// A_m: [input n - m][output n' - m padded to 4]; ts[(n' p + m) 2 + {0, 1}] = tau, sigma.
// *resid = the largest mismatch of the fused table's conversion blocks against them.
template <typename T>
__global__ void k_rcr_coax(const double* __restrict__ fused, const double* __restrict__ dist, int p, int per_dist,
                           T* __restrict__ out, float* __restrict__ resid) {
    const int P = p * p, ld = 2 * P;
    const double* F = fused + (int64_t)blockIdx.x * ld * ld;
    const double t = dist[blockIdx.x];
    T* dst = out + (int64_t)blockIdx.x * per_dist;
    T* ts = dst + coax_off(p, p);
    float worst = 0.f;
    auto tau = [&](int n2, int m) { return n2 > 0 ? t * m / n2 : 0.0; };
    auto sigma = [&](int n2, int m) {
        return n2 + 1 < p ? t * sqrt((double)(n2 + 1 - m) * (n2 + 1 + m)) / (n2 + 1) : 0.0;
    };
    for (int m = 0; m < p; ++m) {
        const int k = p - m, K = pad4(k), mo = m ? 2 * m - 1 : 0;
        T* blk = dst + coax_off(p, m);
        for (int e = threadIdx.x; e < k * K; e += blockDim.x) {
            const int i = e / K, o = e - i * K;
            T v = 0;
            if (o < k) {
                const int n = m + i, n2 = m + o;
                const double a = F[(int64_t)(n * n + mo) * ld + n2 * n2 + mo];
                v = (T)a;
                // check: the phi <- Im chi block is -tau A, the chi <- chi block A - sigma A(n2 + 1)
                const double an = n2 + 1 < p ? F[(int64_t)(n * n + mo) * ld + (n2 + 1) * (n2 + 1) + mo] : 0.0;
                const double b = m ? F[(int64_t)(P + n * n + 2 * m) * ld + n2 * n2 + mo] : 0.0;
                const double c = F[(int64_t)(P + n * n + mo) * ld + P + n2 * n2 + mo];
                const double scale = 1.0 + fabs(a) + fabs(an);
                worst = fmaxf(worst, (float)(fabs(b + tau(n2, m) * a) / scale));
                worst = fmaxf(worst, (float)(fabs(c - (a - sigma(n2, m) * an)) / scale));
            }
            blk[e] = v;
        }
    }
    for (int e = threadIdx.x; e < 2 * P; e += blockDim.x) {
        const int q = e >> 1, n2 = q / p, m = q - n2 * p;
        ts[e] = m <= n2 ? (T)((e & 1) ? sigma(n2, m) : tau(n2, m)) : (T)0;
    }
    if (worst > 0.f) atomic_max_pos(resid, worst);
}

// four pairs of one row: one 16-byte (FP32) or two (FP64) shared-memory accesses
template <typename T> struct alignas(16) Quad {
    T x, y, z, w;
};

template <typename T>
__device__ __forceinline__ Quad<T> make_quad(T x, T y, T z, T w) {
    return Quad<T>{x, y, z, w};
}

template <typename T>
struct RcrArgs {
    const int4* chunks;
    const int2* pairs;
    const int* nchunks;  // device: total chunks (choff[ngroups])
    const T* rot;    // per slot: [Yf | Yb | Zf | Zb]
    const T* coax;   // per distance: [A blocks | tau, sigma]
    const int* dist_of;
    const T* in;
    T* out;
    int64_t ld;
    int p;
    int slot_floats, coax_floats;
    int nrg_y, nrg_cx;   // register-tile row groups of the Y / coaxial stages
    int wide;            // rcr_wide, and a box's row in global memory starts on 16 bytes
};

// Rows and pairs of a thread's register tile in the Y and coaxial stages.  FP32 wants reuse: two 16-byte
// reads feed 16 multiply-adds.  In FP64 a warp's multiply-add holds its quarter of the SM for 64 cycles and
// the reads are free; what counts is that the few items of a chunk of eight pairs (p = 12) load the
// quarters evenly and no row is padded.  Products of the ring of 32,768 in FP64, ms: 4 x 4 tiles 9.1,
// 2 x 4 6.9, 2 x 2 5.8, 1 x 4 5.8, 2 x 1 5.4, 1 x 2 5.2 (its multiply-adds alone: 3.9).
template <typename T> struct RcrTile {
    static constexpr int R = 4, C = 4;
};
template <> struct RcrTile<double> {
    static constexpr int R = 1, C = 2;
};
// consecutive values, read and written 16 bytes at a time
template <typename T, int N> struct alignas(N * sizeof(T) < 16 ? N * sizeof(T) : 16) Run {
    T v[N];
};

template <typename T, int R, int C>
__device__ __forceinline__ void fma_tile(T (&acc)[R][C], Run<T, R> x, Run<T, C> v) {
#pragma unroll
    for (int j = 0; j < R; ++j)
#pragma unroll
        for (int k = 0; k < C; ++k) acc[j][k] = fma(x.v[j], v.v[k], acc[j][k]);
}

// Work item k of a stage for this thread: items are dealt in rounds of RA_THREADS, in
// alternating direction (the row groups come longest first, so every thread gets a mix).
__device__ __forceinline__ int stage_item(int k) {
    return k * RA_THREADS + ((k & 1) ? RA_THREADS - 1 - (int)threadIdx.x : (int)threadIdx.x);
}

// S -> D by the Y blocks: rows q P + n^2 + member(i) of each class of each degree.
template <typename T, int NCP, int NC>
__device__ __forceinline__ void y_stage(const RcrArgs<T>& a, const int* rg_y, const int* yo, const T* Y,
                                        const T* S, T* D) {
    constexpr int TR = RcrTile<T>::R, TC = RcrTile<T>::C, NCG = NC / TC;
    const int P = a.p * a.p, total = a.nrg_y * NCG;
    for (int k = 0; k * RA_THREADS < total; ++k) {
        const int it = stage_item(k);
        if (it >= total) continue;
        const int rg = it / NCG, cg = it - rg * NCG;
        const int code = rg_y[rg], q = code & 1, odd = (code >> 1) & 1, n = (code >> 2) & 31, og = code >> 7;
        const int sz = odd ? n : n + 1, W = pad4(sz);
        const T* x = Y + yo[n] + (odd ? (n + 1) * pad4(n + 1) : 0) + og * TR;
        const T* s = S + (q * P + n * n) * NCP + cg * TC;
        T acc[TR][TC] = {};
        if (odd) {
#pragma unroll 4
            for (int i = 0; i < sz; ++i)
                fma_tile(acc, *reinterpret_cast<const Run<T, TR>*>(x + i * W),
                         *reinterpret_cast<const Run<T, TC>*>(s + odd_member(i) * NCP));
        } else {
#pragma unroll 4
            for (int i = 0; i < sz; ++i)
                fma_tile(acc, *reinterpret_cast<const Run<T, TR>*>(x + i * W),
                         *reinterpret_cast<const Run<T, TC>*>(s + even_member(i) * NCP));
        }
        T* d = D + (q * P + n * n) * NCP + cg * TC;
#pragma unroll
        for (int j = 0; j < TR; ++j) {
            const int o = og * TR + j;
            if (o < sz) {
                Run<T, TC> v;
#pragma unroll
                for (int c = 0; c < TC; ++c) v.v[c] = acc[j][c];
                *reinterpret_cast<Run<T, TC>*>(d + (odd ? odd_member(o) : even_member(o)) * NCP) = v;
            }
        }
    }
}

// S (rotated S-basis multipoles) -> D (rotated R-basis locals): the coaxial translation A_m
// of each order, the same for phi and chi, Re and Im.
template <typename T, int NCP, int NC>
__device__ __forceinline__ void coax_stage(const RcrArgs<T>& a, const int* rg_cx, const int* co, const T* CX,
                                           const T* S, T* D) {
    constexpr int TR = RcrTile<T>::R, TC = RcrTile<T>::C, NCG = NC / TC;
    const int p = a.p, P = p * p, total = a.nrg_cx * NCG;
    for (int kk = 0; kk * RA_THREADS < total; ++kk) {
        const int it = stage_item(kk);
        if (it >= total) continue;
        const int rg = it / NCG, cg = it - rg * NCG;
        const int code = rg_cx[rg], q = code & 1, r = (code >> 1) & 1, m = (code >> 2) & 31, og = code >> 7;
        const int k = p - m, K = pad4(k), mo = m ? 2 * m - 1 : 0;
        const T* blk = CX + co[m] + og * TR;
        const T* s = S + (q * P + mo + r) * NCP + cg * TC;
        T acc[TR][TC] = {};
#pragma unroll 4
        for (int i = 0; i < k; ++i) {
            const int n = m + i;
            fma_tile(acc, *reinterpret_cast<const Run<T, TR>*>(blk + i * K),
                     *reinterpret_cast<const Run<T, TC>*>(s + n * n * NCP));
        }
#pragma unroll
        for (int j = 0; j < TR; ++j) {
            const int n2 = m + og * TR + j;
            if (n2 < p) {
                Run<T, TC> v;
#pragma unroll
                for (int c = 0; c < TC; ++c) v.v[c] = acc[j][c];
                *reinterpret_cast<Run<T, TC>*>(D + (q * P + n2 * n2 + mo + r) * NCP + cg * TC) = v;
            }
        }
    }
}

// S -> D: the phases Z (per order m: the 2 x 2 map of (Re, Im) at z + 4 m) of both
// potentials, per (potential, n, m) and 4 pairs.
template <typename T, int NCP, int NCG>
__device__ __forceinline__ void z_stage(int p, const int* units, const T* Zt, const T* S, T* D) {
    const int P = p * p, nu = p * (p + 1) / 2;
    for (int e = threadIdx.x; e < 2 * nu * NCG; e += RA_THREADS) {
        const int u = e / NCG, cg = e - u * NCG, q = u >= nu, info = units[u - q * nu];
        const int n = info & 31, m = info >> 5;
        const int re = q * P + n * n + (m ? 2 * m - 1 : 0);
        const Quad<T> x = *reinterpret_cast<const Quad<T>*>(S + re * NCP + cg * 4);
        if (m == 0) {
            *reinterpret_cast<Quad<T>*>(D + re * NCP + cg * 4) = x;
        } else {
            const Quad<T> y = *reinterpret_cast<const Quad<T>*>(S + (re + 1) * NCP + cg * 4);
            const Quad<T> z = *reinterpret_cast<const Quad<T>*>(Zt + 4 * m);
            *reinterpret_cast<Quad<T>*>(D + re * NCP + cg * 4) =
                make_quad<T>(fma(z.x, x.x, z.y * y.x), fma(z.x, x.y, z.y * y.y), fma(z.x, x.z, z.y * y.z),
                            fma(z.x, x.w, z.y * y.w));
            *reinterpret_cast<Quad<T>*>(D + (re + 1) * NCP + cg * 4) =
                make_quad<T>(fma(z.z, x.x, z.w * y.x), fma(z.z, x.y, z.w * y.y), fma(z.z, x.z, z.w * y.z),
                            fma(z.z, x.w, z.w * y.w));
        }
    }
}

// Element e of an R x NC block of [row][pair] data, lanes of a warp on 8 rows x 4 pairs:
// conflict-free in shared memory (NCP = 4 mod 8) and 32-byte runs of one pair's row in
// global memory.
template <int NC>
__device__ __forceinline__ void block_elem(int e, int& row, int& col) {
    constexpr int NCT = NC / 4;
    const int tile = e >> 5, ct = tile % NCT, rt = tile / NCT;
    row = rt * 8 + (e & 7);
    col = ct * 4 + ((e >> 3) & 3);
}

// Gathers the source multipoles of a chunk into A (asynchronous 4-byte copies; columns of
// absent pairs are zero).
template <typename T, int NC, int NCP>
__device__ __forceinline__ void gather_async(const RcrArgs<T>& a, int p0, int np, T* A) {
    const int R = 2 * a.p * a.p, R8 = (R + 7) & ~7;
    for (int e = threadIdx.x; e < R8 * NC; e += RA_THREADS) {
        int row, col;
        block_elem<NC>(e, row, col);
        if (row >= R) continue;
        T* dst = A + row * NCP + col;
        if (col < np) {
            const int src = a.pairs[p0 + col].x;
            const T* g = a.in + (int64_t)src * a.ld + row;
            const unsigned sa = (unsigned)__cvta_generic_to_shared(dst);
            asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(sa), "l"(g), "n"((int)sizeof(T)) : "memory");
        } else {
            *dst = (T)0;
        }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
}

// The same where rcr_wide allows it: A as [pair][row], in 16-byte pieces, a row one piece
// longer than R so that one piece of consecutive pairs spreads over the banks.
template <typename T, int NC>
__device__ __forceinline__ void gather_wide(const RcrArgs<T>& a, int p0, int np, T* A) {
    constexpr int VE = 16 / (int)sizeof(T);
    const int R = 2 * a.p * a.p, pieces = R / VE;
    for (int e = threadIdx.x; e < pieces * NC; e += RA_THREADS) {
        const int col = e / pieces, q = e - col * pieces;
        T* dst = A + col * (R + VE) + q * VE;
        if (col < np) {
            const T* g = a.in + (int64_t)a.pairs[p0 + col].x * a.ld + q * VE;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(dst)), "l"(g) : "memory");
        } else {
#pragma unroll
            for (int k = 0; k < VE; ++k) dst[k] = (T)0;
        }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
}

// [pair][row] pieces <-> [row][pair]
template <typename T, int NC, int NCP, bool IN>
__device__ __forceinline__ void transpose_block(int R, const T* S, T* D) {
    constexpr int VE = 16 / (int)sizeof(T);
    struct alignas(16) Piece {
        T v[VE];
    };
    for (int e = threadIdx.x; e < R / VE * NC; e += RA_THREADS) {
        const int q = e / NC, col = e - q * NC;
        if (IN) {
            const Piece x = *reinterpret_cast<const Piece*>(S + col * (R + VE) + q * VE);
#pragma unroll
            for (int k = 0; k < VE; ++k) D[(q * VE + k) * NCP + col] = x.v[k];
        } else {
            Piece x;
#pragma unroll
            for (int k = 0; k < VE; ++k) x.v[k] = S[(q * VE + k) * NCP + col];
            *reinterpret_cast<Piece*>(D + col * (R + VE) + q * VE) = x;
        }
    }
}

template <typename T, int NC>
__global__ void __launch_bounds__(RA_THREADS) k_rcr_m2l(RcrArgs<T> a) {
    constexpr int NCP = NC + 4;  // row stride of the buffers (16-byte aligned, 4 mod 8)
    constexpr int NCG = NC / 4;
    extern __shared__ __align__(16) unsigned char ra_raw[];
    T* ra_smem = reinterpret_cast<T*>(ra_raw);
    const int p = a.p, P = p * p, R = 2 * P;
    const int ysz = y_off(p);
    T* tab = ra_smem;                 // the slot's [Yf | Yb | Zf | Zb]
    const T* Yf = tab;
    const T* Yb = tab + ysz;
    const T* Zf = tab + 2 * ysz;
    const T* Zb = Zf + 4 * p;
    T* CX = tab + a.slot_floats;      // the distance's [A blocks | tau, sigma]
    const T* TS = CX + coax_off(p, p);
    T* A = CX + a.coax_floats;      // gathered multipoles (the next chunk's, while the stages run)
    T* B = A + R * NCP;
    T* C = B + R * NCP;
    int* rg_y = reinterpret_cast<int*>(C + R * NCP);
    int* rg_cx = rg_y + a.nrg_y;
    int* units = rg_cx + a.nrg_cx;      // [p (p + 1) / 2]: n | m << 5 of every order m <= n
    int* yo = units + RCR_PMAX * (RCR_PMAX + 1) / 2;  // [RCR_PMAX + 1] first float of each degree's Y blocks
    int* co = yo + RCR_PMAX + 1;        // [RCR_PMAX + 1] first float of each order's coaxial block
    int* s_dst = co + RCR_PMAX + 1;
    const int tid = threadIdx.x;
    if (tid == 0) {
        // row groups longest first
        constexpr int TR = RcrTile<T>::R;
        int g = 0;
        for (int n = p - 1; n >= 0; --n)
            for (int q = 0; q < 2; ++q)
                for (int odd = 0; odd < 2; ++odd)
                    for (int og = 0; og * TR < (odd ? n : n + 1); ++og)
                        rg_y[g++] = q | (odd << 1) | (n << 2) | (og << 7);
        g = 0;
        for (int m = 0; m < p; ++m)
            for (int q = 0; q < 2; ++q)
                for (int r = 0; r < (m ? 2 : 1); ++r)
                    for (int og = 0; og * TR < p - m; ++og)
                        rg_cx[g++] = q | (r << 1) | (m << 2) | (og << 7);
        for (int k = 0; k <= p; ++k) {
            yo[k] = y_off(k);
            co[k] = coax_off(p, k);
        }
        g = 0;
        for (int n = 0; n < p; ++n)
            for (int m = 0; m <= n; ++m) units[g++] = n | (m << 5);
    }
    const int nch = *a.nchunks;
    const int c0 = (int)((int64_t)blockIdx.x * nch / gridDim.x), c1 = (int)((int64_t)(blockIdx.x + 1) * nch / gridDim.x);
    const auto gather = [&](const int4& ch) {
        if (a.wide) gather_wide<T, NC>(a, ch.y, ch.z, A);
        else gather_async<T, NC, NCP>(a, ch.y, ch.z, A);
    };
    if (c0 < c1) gather(a.chunks[c0]);
    int cur = -1;
    for (int chunk = c0; chunk < c1; ++chunk) {
        const int4 ch = a.chunks[chunk];
        const int slot = ch.x, p0 = ch.y, np = ch.z;
        __syncthreads();  // the previous chunk's epilogue has read B and s_dst
        if (slot != cur) {
            const Quad<T>* sr = reinterpret_cast<const Quad<T>*>(a.rot + (int64_t)slot * a.slot_floats);
            Quad<T>* dr = reinterpret_cast<Quad<T>*>(tab);
            for (int e = tid; e < a.slot_floats / 4; e += RA_THREADS) dr[e] = sr[e];
            const Quad<T>* sc = reinterpret_cast<const Quad<T>*>(a.coax + (int64_t)a.dist_of[slot] * a.coax_floats);
            Quad<T>* dc = reinterpret_cast<Quad<T>*>(CX);
            for (int e = tid; e < a.coax_floats / 4; e += RA_THREADS) dc[e] = sc[e];
            cur = slot;
        }
        if (tid < NC) s_dst[tid] = tid < np ? a.pairs[p0 + tid].y : -1;
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        bulk_wait_read();  // the additions of the previous chunk have read B
        __syncthreads();
        if (a.wide) {
            transpose_block<T, NC, NCP, true>(R, A, C);
            __syncthreads();
        }
        z_stage<T, NCP, NCG>(p, units, Zf, a.wide ? C : A, B);
        __syncthreads();
        if (chunk + 1 < c1) {  // A is free: the next chunk's multipoles arrive during the stages
            gather(a.chunks[chunk + 1]);
        }
        y_stage<T, NCP, NC>(a, rg_y, yo, Yf, B, C);
        __syncthreads();
        coax_stage<T, NCP, NC>(a, rg_cx, co, CX, C, B);
        __syncthreads();
        // B -> C: the conversion of Eq. rcr1, per (n, m) and 4 pairs:
        // Re phi~ = Re phi - tau Im chi, Im phi~ = Im phi + tau Re chi, chi~_n = chi_n - sigma chi_{n+1}
        for (int e = tid; e < p * (p + 1) / 2 * NCG; e += RA_THREADS) {
            const int u = e / NCG, cg = e - u * NCG, info = units[u];
            const int n = info & 31, m = info >> 5, parts = m ? 2 : 1;
            const int re = n * n + (m ? 2 * m - 1 : 0);
            const T tau = TS[(n * p + m) * 2], sigma = TS[(n * p + m) * 2 + 1];
            Quad<T> ph[2], ch[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                if (k < parts) {
                    ph[k] = *reinterpret_cast<const Quad<T>*>(B + (re + k) * NCP + cg * 4);
                    ch[k] = *reinterpret_cast<const Quad<T>*>(B + (P + re + k) * NCP + cg * 4);
                }
            }
            if (m > 0) {
                Quad<T> o0 = ph[0], o1 = ph[1];
                o0.x = fma(-tau, ch[1].x, o0.x);
                o0.y = fma(-tau, ch[1].y, o0.y);
                o0.z = fma(-tau, ch[1].z, o0.z);
                o0.w = fma(-tau, ch[1].w, o0.w);
                o1.x = fma(tau, ch[0].x, o1.x);
                o1.y = fma(tau, ch[0].y, o1.y);
                o1.z = fma(tau, ch[0].z, o1.z);
                o1.w = fma(tau, ch[0].w, o1.w);
                *reinterpret_cast<Quad<T>*>(C + re * NCP + cg * 4) = o0;
                *reinterpret_cast<Quad<T>*>(C + (re + 1) * NCP + cg * 4) = o1;
            } else {
                *reinterpret_cast<Quad<T>*>(C + re * NCP + cg * 4) = ph[0];
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                if (k < parts) {
                    Quad<T> c = ch[k];
                    if (n + 1 < p) {  // chi_{n+1}^m: row + 2n + 1
                        const Quad<T> nx = *reinterpret_cast<const Quad<T>*>(B + (P + re + k + 2 * n + 1) * NCP + cg * 4);
                        c.x = fma(-sigma, nx.x, c.x);
                        c.y = fma(-sigma, nx.y, c.y);
                        c.z = fma(-sigma, nx.z, c.z);
                        c.w = fma(-sigma, nx.w, c.w);
                    }
                    *reinterpret_cast<Quad<T>*>(C + (P + re + k) * NCP + cg * 4) = c;
                }
            }
        }
        __syncthreads();
        y_stage<T, NCP, NC>(a, rg_y, yo, Yb, C, B);
        __syncthreads();
        z_stage<T, NCP, NCG>(p, units, Zb, B, C);
        __syncthreads();
        if (a.wide) {  // one bulk addition a pair
            transpose_block<T, NC, NCP, false>(R, C, B);
            fence_async_smem();
            __syncthreads();
            constexpr int VE = 16 / (int)sizeof(T);
            if (tid < np) bulk_add(a.out + (int64_t)s_dst[tid] * a.ld, B + tid * (R + VE), R * (uint32_t)sizeof(T));
            bulk_commit();
            continue;
        }
        const int R8 = (R + 7) & ~7;
        for (int e = tid; e < R8 * NC; e += RA_THREADS) {
            int row, col;
            block_elem<NC>(e, row, col);
            if (row < R && col < np) atomicAdd(a.out + (int64_t)s_dst[col] * a.ld + row, C[row * NCP + col]);
        }
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    bulk_wait_all();
}

int slot_floats(int p) { return 2 * y_off(p) + 8 * p; }
int coax_floats(int p) { return coax_off(p, p) + pad4(2 * p * p); }

int tile_rows(int size) { return size == 8 ? RcrTile<double>::R : RcrTile<float>::R; }

int rg_y_count(int p, int size) {
    const int tr = tile_rows(size);
    int g = 0;
    for (int n = 0; n < p; ++n) g += (n + tr) / tr + (n + tr - 1) / tr;
    return 2 * g;
}

int rg_cx_count(int p, int size) {
    const int tr = tile_rows(size);
    int g = 0;
    for (int m = 0; m < p; ++m) g += (m ? 2 : 1) * ((p - m + tr - 1) / tr);
    return 2 * g;
}

int apply_smem(int p, int nc, int size) {
    const int P = p * p;
    const int floats = slot_floats(p) + coax_floats(p) + 3 * (2 * P) * (nc + 4);
    const int ints = rg_y_count(p, size) + rg_cx_count(p, size) + RCR_PMAX * (RCR_PMAX + 1) / 2 + 2 * (RCR_PMAX + 1) + nc;
    return floats * size + ints * 4;
}

// Whether a chunk may take the 16-byte route: a row of whole 16-byte pieces, and nc rows each a piece longer,
// [pair][R + VE], no larger than the buffer [R][nc + 4] they share with the stages (FP32: nc <= R, which 32
// pairs at p = 2 are not).
bool rcr_wide(int p, int size, int nc) {
    const int R = 2 * p * p, VE = 16 / size;
    return R % VE == 0 && nc * VE <= 4 * R;
}

template <typename T, int NC>
void launch_apply(Ctx* c, const RcrTables& rt, const RcrArgs<T>& a) {
    cuda_check(cudaFuncSetAttribute(k_rcr_m2l<T, NC>, cudaFuncAttributeMaxDynamicSharedMemorySize, rt.smem), "rcr smem");
    cuda_check(cudaFuncSetAttribute(k_rcr_m2l<T, NC>, cudaFuncAttributePreferredSharedMemoryCarveout, 100),
               "rcr carveout");
    k_rcr_m2l<T, NC><<<rt.nsm * rt.ctas_per_sm, RA_THREADS, rt.smem, stream_of(c)>>>(a);
}

void rot_matrix(double theta, double phi, bool inverse, bool y_part, double* q) {
    // y_part: Ry(+-theta); else Rz(+-phi); row-major, u' = R u
    const double s = inverse ? -1.0 : 1.0;
    for (int i = 0; i < 9; ++i) q[i] = 0.0;
    if (y_part) {
        const double c = std::cos(theta), sn = s * std::sin(theta);
        q[0] = c;
        q[2] = sn;
        q[4] = 1.0;
        q[6] = -sn;
        q[8] = c;
    } else {
        const double c = std::cos(phi), sn = s * std::sin(phi);
        q[0] = c;
        q[1] = -sn;
        q[3] = sn;
        q[4] = c;
        q[8] = 1.0;
    }
}

}  // namespace

void gauss_legendre_nodes(int nq, double* xi, double* w) {
    for (int i = 0; i < (nq + 1) / 2; ++i) {
        double x = std::cos(PI * (i + 0.75) / (nq + 0.5)), dp = 0.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = x;
            for (int k = 2; k <= nq; ++k) {
                const double pk = ((2.0 * k - 1.0) * x * p1 - (k - 1.0) * p0) / k;
                p0 = p1;
                p1 = pk;
            }
            if (nq == 1) p1 = x, p0 = 1.0;
            dp = nq * (x * p1 - p0) / (x * x - 1.0);
            const double dx = p1 / dp;
            x -= dx;
            if (std::fabs(dx) < 1e-16) break;
        }
        const double wi = 2.0 / ((1.0 - x * x) * dp * dp);
        xi[i] = -x;
        w[i] = wi;
        xi[nq - 1 - i] = x;
        w[nq - 1 - i] = wi;
    }
}

// NC a multiple of 8 keeps the row stride NC + 4 at 4 mod 8 (conflict-free columns in FP32); the
// most resident CTAs per SM up to two (the stages are latency-bound; measured on GB300: p = 12
// 24 pairs x 2 CTAs 121 ms against 8 x 3 129 ms; p = 16 8 x 2 249 ms against 24 x 1 317 ms),
// then the largest chunk.  0: the tables do not fit.
int rcr_chunk(int p, int size, int* ctas) {
    int best = 0, pick = 0;
    if (p < 1 || p > RCR_PMAX) return 0;
    for (int nc : {32, 24, 16, 8}) {
        const int sm = apply_smem(p, nc, size);
        if (sm > SMEM_MAX) continue;
        const int k = std::min(2, SMEM_PER_SM / (sm + 1024));
        if (k * 64 + nc > best) {
            best = k * 64 + nc;
            pick = nc;
            if (ctas) *ctas = k;
        }
    }
    return pick;
}

void rcr_free(RcrTables& rt) {
    for (Buf* b : {&rt.rot, &rt.coax, &rt.dist_of}) {
        if (b->ptr) cudaFree(b->ptr);
        b->ptr = nullptr;
        b->cap = 0;
    }
    rt.p = 0;
}

template <typename T>
void rcr_build(Ctx* c, int p, RcrTables& rt) {
    if (p < 1 || p > RCR_PMAX) throw Error{LHV_EUNSUPPORTED, "RCR translations run p <= 20"};
    cudaStream_t s = stream_of(c);
    rcr_free(rt);
    std::vector<int> offs, slot_of;
    m2l_offsets(offs, slot_of);
    // per slot: t = target - source = -(source offset) = |t| (sin th cos ph, sin th sin ph, cos th)
    // the blocks depend on theta or phi alone, which many offsets share: one job per distinct angle
    std::vector<RotJob> jobs;
    std::vector<int> job_of;
    std::map<std::pair<int, long long>, int> known;  // (which of the four, angle in units of 1e-12) -> job
    for (int k = 0; k < NUM_OFFSETS; ++k) {
        const double tx = -offs[3 * k], ty = -offs[3 * k + 1], tz = -offs[3 * k + 2];
        const double tl = std::sqrt(tx * tx + ty * ty + tz * tz);
        const double th = std::acos(std::max(-1.0, std::min(1.0, tz / tl)));
        const double ph = std::atan2(ty, tx);
        // Y(theta), S basis; Y(-theta), R basis; Z(phi), S basis; Z(-phi), R basis
        for (int which = 0; which < 4; ++which) {
            const bool y = which < 2, inverse = (which & 1) != 0;
            const auto at = known.emplace(std::make_pair(which, std::llround((y ? th : ph) * 1e12)), (int)jobs.size());
            if (at.second) {
                jobs.emplace_back();
                rot_matrix(th, ph, inverse, y, jobs.back().q);
                jobs.back().r_basis = inverse ? 1 : 0;
                jobs.back().pad = 0;
            }
            job_of.push_back(at.first->second);
        }
    }
    std::vector<double> xq(p), wq(p);
    gauss_legendre_nodes(p, xq.data(), wq.data());
    // distinct distances of the offsets
    std::vector<int> d2s, dist_of(NUM_OFFSETS);
    for (int k = 0; k < NUM_OFFSETS; ++k) {
        const int d2 = offs[3 * k] * offs[3 * k] + offs[3 * k + 1] * offs[3 * k + 1] + offs[3 * k + 2] * offs[3 * k + 2];
        auto it = std::find(d2s.begin(), d2s.end(), d2);
        if (it == d2s.end()) {
            dist_of[k] = (int)d2s.size();
            d2s.push_back(d2);
        } else {
            dist_of[k] = (int)(it - d2s.begin());
        }
    }
    std::vector<double> t3, dist;
    for (int d2 : d2s) {
        t3.push_back(0.0);
        t3.push_back(0.0);
        t3.push_back(std::sqrt((double)d2));
        dist.push_back(std::sqrt((double)d2));
    }
    const int P = p * p, NE = p * (4 * p * p - 1) / 3;
    const int sf = slot_floats(p), cf = coax_floats(p);
    Buf djobs, djob_of, dq, dense, fused, ddist, dres;
    float resid = 0.f;
    auto cleanup = [&] {
        for (Buf* b : {&djobs, &djob_of, &dq, &dense, &fused, &ddist, &dres}) cudaFree(b->ptr);
    };
    try {
        ensure(c, djobs, (int64_t)jobs.size() * sizeof(RotJob));
        ensure(c, djob_of, (int64_t)job_of.size() * 4);
        cuda_check(cudaMemcpyAsync(djob_of.ptr, job_of.data(), job_of.size() * 4, cudaMemcpyHostToDevice, s),
                   "rcr job index");
        ensure(c, dq, 2 * p * 8);
        ensure(c, dense, (int64_t)jobs.size() * NE * 8);
        ensure(c, dres, 16);
        cuda_check(cudaMemcpyAsync(djobs.ptr, jobs.data(), jobs.size() * sizeof(RotJob), cudaMemcpyHostToDevice, s),
                   "rcr jobs");
        cuda_check(cudaMemcpyAsync(dq.ptr, xq.data(), p * 8, cudaMemcpyHostToDevice, s), "rcr nodes");
        cuda_check(cudaMemcpyAsync(dq.as<double>() + p, wq.data(), p * 8, cudaMemcpyHostToDevice, s), "rcr weights");
        cuda_check(cudaMemsetAsync(dres.ptr, 0, 16, s), "rcr resid");
        const int smem = (NE + P + RB_BATCH * 2 * P + RB_BATCH) * 8;
        cuda_check(cudaFuncSetAttribute(k_rcr_rotations, cudaFuncAttributeMaxDynamicSharedMemorySize, smem),
                   "rcr rotation smem");
        k_rcr_rotations<<<(int)jobs.size(), RB_THREADS, smem, s>>>(djobs.as<RotJob>(), p, dq.as<double>(),
                                                                    dq.as<double>() + p, dense.as<double>());
        count_launch(c);
        check_launch("rcr rotations");
        ensure(c, rt.rot, (int64_t)NUM_OFFSETS * sf * (int64_t)sizeof(T));
        k_rcr_pack<T><<<NUM_OFFSETS, 256, 0, s>>>(dense.as<double>(), djob_of.as<int>(), p, sf, rt.rot.as<T>(), dres.as<float>());
        count_launch(c);
        check_launch("rcr pack");
        build_m2l_at(c, p, t3, fused);
        ensure(c, ddist, (int64_t)dist.size() * 8);
        cuda_check(cudaMemcpyAsync(ddist.ptr, dist.data(), dist.size() * 8, cudaMemcpyHostToDevice, s), "rcr dist");
        ensure(c, rt.coax, (int64_t)d2s.size() * cf * (int64_t)sizeof(T));
        k_rcr_coax<T><<<(int)d2s.size(), 256, 0, s>>>(fused.as<double>(), ddist.as<double>(), p, cf, rt.coax.as<T>(),
                                                   dres.as<float>() + 1);
        count_launch(c);
        check_launch("rcr coaxial");
        ensure(c, rt.dist_of, NUM_OFFSETS * 4);
        cuda_check(cudaMemcpyAsync(rt.dist_of.ptr, dist_of.data(), NUM_OFFSETS * 4, cudaMemcpyHostToDevice, s),
                   "rcr distances");
        float hr[2] = {0.f, 0.f};
        cuda_check(cudaMemcpyAsync(hr, dres.ptr, 8, cudaMemcpyDeviceToHost, s), "rcr resid read");
        cuda_check(cudaStreamSynchronize(s), "rcr tables");
        resid = std::max(hr[0], hr[1]);
    } catch (...) {
        cleanup();
        throw;
    }
    cleanup();
    // the structure the products assume (phases, classes, conversion coefficients) holds to
    // the tables' FP64 rounding
    if (!(resid < 1e-9f)) {
        rcr_free(rt);
        throw Error{LHV_EUNSUPPORTED, "RCR tables failed their structural check"};
    }
    rt.p = p;
    rt.slot_floats = sf;
    rt.coax_floats = cf;
    rt.resid = resid;
    rt.nc = rcr_chunk(p, sizeof(T), &rt.ctas_per_sm);
    if (rt.nc == 0) throw Error{LHV_EUNSUPPORTED, "RCR tables exceed shared memory"};
    rt.smem = apply_smem(p, rt.nc, sizeof(T));
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    rt.nsm = sms > 0 ? sms : 152;
}

template <typename T>
void rcr_apply(Ctx* c, const RcrTables& rt, Grouped& gp, const T* mult, T* loc, int64_t ld) {
    RcrArgs<T> a{};
    a.chunks = gp.chunks.as<int4>();
    a.pairs = gp.pairs.as<int2>();
    a.nchunks = gp.choff.as<int>() + gp.ngroups;
    a.rot = rt.rot.as<T>();
    a.coax = rt.coax.as<T>();
    a.dist_of = rt.dist_of.as<int>();
    a.in = mult;
    a.out = loc;
    a.ld = ld;
    a.p = rt.p;
    a.slot_floats = rt.slot_floats;
    a.coax_floats = rt.coax_floats;
    a.nrg_y = rg_y_count(rt.p, sizeof(T));
    a.nrg_cx = rg_cx_count(rt.p, sizeof(T));
    a.wide = rcr_wide(rt.p, sizeof(T), rt.nc) && ld * sizeof(T) % 16 == 0;
    switch (rt.nc) {
        case 32: launch_apply<T, 32>(c, rt, a); break;
        case 24: launch_apply<T, 24>(c, rt, a); break;
        case 16: launch_apply<T, 16>(c, rt, a); break;
        default: launch_apply<T, 8>(c, rt, a); break;
    }
    count_launch(c);
    check_launch("rcr m2l");
}

template void rcr_build<float>(Ctx*, int, RcrTables&);
template void rcr_build<double>(Ctx*, int, RcrTables&);
template void rcr_apply<float>(Ctx*, const RcrTables&, Grouped&, const float*, float*, int64_t);
template void rcr_apply<double>(Ctx*, const RcrTables&, Grouped&, const double*, double*, int64_t);

}  // namespace lhv
