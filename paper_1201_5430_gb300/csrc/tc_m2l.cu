// Tensor-core (tcgen05, TF32) translations: M2L, and L2L with the same kernel.
//
// The fused operator of a translation t is [[T, C12 T], [0, C22 T]] (Eqs. mr3, drt10, drt11): the
// same translation T for both potentials, then the conversion, which couples each (n, m) to
// at most six reals of the translated chi and whose coefficients are linear in t.  So the
// products are only  phi^ = T phi,  chi^ = T chi  (4 p^4 multiply-adds' flops a pair instead of
// the 6 p^4 of the fused table, and a third of its operator bytes: one P x P block shared by both
// potentials, P = p^2), and the conversion runs on the accumulators:
//   phi~_n^m = phi^_n^m + a (tx + i ty) chi^_n^{m+1} + b (tx - i ty) chi^_n^{m-1} + i z tz chi^_n^m
//   chi~_n^m = chi^_n^m + d (ty + i tx) chi^_{n+1}^{m-1} + e (ty - i tx) chi^_{n+1}^{m+1} + f tz chi^_{n+1}^m
// in the scaled real basis of operators.cu (t in box sides):
//   a = -sqrt((n-m)(n+m+1)) / 2n,  b = sqrt((n+m)(n-m+1)) / 2n,  z = m / n  (0 at n = 0),
//   d = sqrt((n-m+1)(n-m+2)) / 2(n+1),  e = -sqrt((n+m+1)(n+m+2)) / 2(n+1),
//   f = -sqrt((n+1-m)(n+1+m)) / (n+1)   (d = e = f = 0 at n = p - 1: the chi_p term is dropped);
//   at m = 0 the m - 1 terms are the conjugates of the m + 1 terms: a and e doubled, b = d = 0.
// L2L converts in the same (R) basis; its T block carries the change of scale from the parent's
// box to the child's of phi, and chi takes half of it (one length more, Eq. 4).  M2M is not taken here: its
// error would be larger than in FP32 (run_l2l's rule in expansions.cu).
// The scalar reference case is the same kernel with one potential and no conversion.
//
// D (128 pairs x N) = X (128 x P) T^T (P x N) per potential, D in TMEM in FP32 (phi^ and chi^
// side by side, 2 P <= 512 columns up to p = 16; above, the outputs are split into ranges of
// degrees of at most 256 columns, each with the halo degree that chi~ reads).  Precision: every
// operand split a = hi + lo, hi = tf32(a), lo = tf32(a - hi); D accumulates hi.hi + hi.lo + lo.hi.
//
// One persistent CTA per SM, its warps specialised, K walked in chunks of 16 through a ring of
// shared stages (canonical no-swizzle K-major tiles):
//   warps 8-15  gather the FP32 source rows (a chunk ahead in registers, two groups of four warps on
//               alternate chunks), split them and store the hi / lo tiles;
//   warp 16     brings the operator's hi / lo tile of the chunk with one bulk copy;
//   warp 17     issues the MMAs (2 k-steps x 3 products x potentials) and commits the stage;
//   warps 0-7   read the accumulators (thread = pair), convert, and stage bands of columns as
//               [pair][column]; the copy engine adds a pair's band to its row (bulk reductions).
// K runs from the high source degrees down and each stage takes the small cross products before
// hi.hi: the accumulator rounds toward zero at its own magnitude, which then is small until the
// last steps.  Far field against FP64, sphere surface at p = 12: v 3.2e-7, s 3.1e-7 (FP32 CUDA cores
// 3.6e-7, 3.3e-7); in ascending order, and in the fused-table kernel before, 1.2e-6, 1.5e-6.
// Measured (products, ms an evaluation, fused-table kernel before / this one with the additions by
// atomicAdd / by bulk reductions): sphere surface of 2^20 at p = 12, 4.13 M pairs 7.26 / 4.56 / 4.24; scalar
// cube of 2^20 at p = 12, 6.04 M pairs 4.01 / 2.28 / 1.96; offset rings of 2^21 at p = 16, 1.33 M
// pairs 4.33 / 2.54 / 2.32.  Without the epilogue the first takes 1.97: the conversion runs in turn with
// the products where one accumulator set fills TMEM.  No unit is near its rate (sphere surface of 2^19, 3.81 M
// pairs, ncu): tensor pipe 20 %, issue slots 42 %, L1 and shared memory 45 %, ALU 31 %, FMA 18 %; of the stalls the
// long scoreboard (the gathers and the reads of TMEM) leads with 5.8 warps an issue.  Operand traffic a pair at p = 12: 1.15 KB of source (split here instead of two
// arrays) and 1.3 KB of operator, against 3.5 and 3.9 of the fused tables.
//
// Every mbarrier wait gives up after a fixed number of polls, sets the error word for the host
// and an abort word that ends every role; copies and MMAs in flight are waited for (bounded)
// before TMEM is freed.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "lhv_group.cuh"
#include "lhv_internal.cuh"
#include "tc_common.cuh"

namespace lhv {

namespace {

constexpr int M2_EPI_WARPS = 8, M2_PROD_WARPS = 8, M2_GROUPS = 2;
constexpr int M2_WARPS = M2_EPI_WARPS + M2_PROD_WARPS + 2;
constexpr int M2_THREADS = 32 * M2_WARPS;
constexpr int M2_MAX_STAGES = 4;
constexpr int M2_MAX_RANGES = 4;
constexpr int M2_X_TILE = TC_PAIRS * TC_KC * 4;  // bytes of one operand tile of the pairs
constexpr int M2_BAND = 64;                // columns (a potential) staged at once
constexpr int M2_STG_LD = M2_BAND + 4;     // staging [pair][column]: a quad of a pair to a bank group of its own
constexpr int M2_TMEM = 512;               // TMEM columns: one or two accumulator buffers
constexpr int M2_SMEM_MAX = 226 * 1024;    // dynamic shared memory (the static part is below 1 KB)

struct M2lArgs {
    const int4* chunks;
    const int2* pairs;
    const int* choff;
    int g0, g1;
    int swap;                // 1: the pairs are (destination, source)
    const float* in;
    float* out;
    int64_t ld;
    int p, P;
    const float* tiles;      // per slot: ranges x K chunks x [hi | lo] tiles
    int64_t group_stride;    // floats per slot
    int nranges;
    int n0[M2_MAX_RANGES], n1[M2_MAX_RANGES];   // output degrees [n0, n1) of each range
    int c0[M2_MAX_RANGES], nlen[M2_MAX_RANGES]; // its columns [c0, c0 + nlen) (with the halo, 16-padded)
    int64_t roff[M2_MAX_RANGES];
    int nstages, stage_bytes;
    int nbuf;                // accumulator buffers (each M2_TMEM / nbuf columns)
    const float* conv;       // [p (p + 1) / 2 + 8][8]: a, b, z, d | e, f, 0, 0 of (n, m) at n (n + 1) / 2 + m
    const float* tvec;       // [ngroups][4]: t of each operator, in box sides of the conversion's basis
    float chi_scale;         // chi^ = chi_scale T chi (1; L2L 1/2)
    int ngroups;             // operators (a group's is g % ngroups)
    int* err;
    int64_t wait_limit;      // polls after which a wait gives up
};

// floats of the conversion table, padded for the reads of the eight orders of a last unit
__host__ __device__ constexpr int conv_floats(int p) { return (p * (p + 1) / 2 + 8) * 8; }

struct M2lShared {
    uint64_t full_a[M2_MAX_STAGES], full_b[M2_MAX_STAGES], empty[M2_MAX_STAGES];
    uint64_t acc_full[2], acc_empty[2], done;
    uint32_t tmem;
    int abort;       // set by a role whose wait gave up
};

// bounded wait that also ends when another role has given up
__device__ __forceinline__ bool m2_wait(uint64_t* bar, uint32_t parity, M2lShared& sh, const M2lArgs& args) {
    const uint32_t a = smem_u32(bar);
    for (int64_t it = 0; it < args.wait_limit; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
        if ((it & 63) == 63 && *(volatile int*)&sh.abort) return false;
    }
    *(volatile int*)&sh.abort = 1;
    atomicExch(args.err, 1);
    return false;
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_copy(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
// first column of a range's accumulators: ranges above the first start 16 columns in, since the
// epilogue reads the column before a degree
__device__ __forceinline__ uint32_t acc_base(int range) { return range ? 16u : 0u; }

// Barrier of the 256 epilogue threads; whether any of them passed `leave`, the same answer for all.  (A word in
// shared memory that each reads after the barrier is not: a fast warp can set it for its next item before a slow one has
// read it for this one, and the two would part at different barriers.)
__device__ __forceinline__ bool epi_any(bool leave) {
    uint32_t any;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.or.pred q, 1, 256, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}\n"
        : "=r"(any)
        : "r"((uint32_t)leave)
        : "memory");
    return any != 0;
}
// the two epilogue warps of a lane quarter
__device__ __forceinline__ void quarter_sync(int quarter) {
    asm volatile("bar.sync %0, 64;" ::"r"(2 + quarter) : "memory");
}
__device__ __forceinline__ void tmem_ld1(uint32_t addr, uint32_t& a) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(a) : "r"(addr));
}
__device__ __forceinline__ void tmem_ld2(uint32_t addr, uint32_t& a, uint32_t& b) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(a), "=r"(b) : "r"(addr));
}
__device__ __forceinline__ void tmem_ld16_async(uint32_t addr, uint32_t* r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(addr));
}
// the loads before it have arrived; the registers may be read after it (ties them to the wait)
template <int N>
__device__ __forceinline__ void tmem_wait(uint32_t (&r)[N]) {
    static_assert(N == 16 || N == 20, "");
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                   "+r"(r[15])
                 :
                 : "memory");
    if constexpr (N == 20) asm volatile("" : "+r"(r[N - 4]), "+r"(r[N - 3]), "+r"(r[N - 2]), "+r"(r[N - 1]) : : "memory");
}

// chi of the orders mb - 1 .. mb + 8 of degree N: x[k] = column N^2 + 2 mb - 3 + k, so order
// mb + i is (Re, Im) = (x[2 i + 2], x[2 i + 3]).  The last pair is read where order mb + 8
// exists only (the reads stay inside the accumulators); columns past the degree hold other
// coefficients and are masked by the caller.
__device__ __forceinline__ void tmem_orders(uint32_t col, int N, int mb, uint32_t (&x)[20]) {
    tmem_ld16_async(col, x);
    tmem_ld2(col + 16, x[16], x[17]);
    if (mb + 8 <= N) tmem_ld2(col + 18, x[18], x[19]);
    else x[18] = x[19] = 0u;
}
// order 0 is one real at x[3]: (Re, Im) = (x[3], 0), and there is no order -1
template <int N>
__device__ __forceinline__ void order_zero(uint32_t (&x)[N]) {
    x[0] = x[1] = 0u;
    x[2] = x[3];
    x[3] = 0u;
}

// (Re, Im) of the orders M .. M + 3 (M a multiple of 4) of degree n to d[0 .. 8), d = the column of Re of
// order M.  Orders past n are not stored, and order 0 is the one real v[1].  An odd degree's
// orders start on a quad (n^2 - 1 = 0 mod 4), whose first column belongs to the degree below where M = 0;
// an even one's a column before.
__device__ __forceinline__ void store_orders(float* d, const float (&v)[8], int M, int n) {
    if (n & 1) {
        if (M == 0) {
            d[1] = v[1];
            *reinterpret_cast<float2*>(d + 2) = make_float2(v[2], v[3]);
        } else {
            *reinterpret_cast<float4*>(d) = make_float4(v[0], v[1], v[2], v[3]);
        }
        if (M + 2 <= n) *reinterpret_cast<float4*>(d + 4) = make_float4(v[4], v[5], v[6], v[7]);
    } else {
        if (M > 0) d[0] = v[0];
        if (M + 2 <= n) {
            *reinterpret_cast<float4*>(d + 1) = make_float4(v[1], v[2], v[3], v[4]);
            if (M + 4 <= n) {
                *reinterpret_cast<float2*>(d + 5) = make_float2(v[5], v[6]);
                d[7] = v[7];
            } else {
                d[5] = v[5];
            }
        } else {
            d[1] = v[1];
        }
    }
}

// Converts the orders [mb, mb + 8) of degree n of this thread's pair and writes them to the
// staging columns op (phi) and oc (chi), column n^2 at op[0].  x: chi of degree n as
// read by tmem_orders with order_zero applied; on return that of the next degree, so
// that a run of degrees reads each once.
__device__ __forceinline__ void convert_orders(const float* cv, uint32_t tp, uint32_t tc, int c0, int p, int n,
                                               int mb, float tx, float ty, float tz, float cs, uint32_t (&x)[20],
                                               float* op, float* oc) {
    uint32_t y[20], f[16];
    const bool up = n + 1 < p;
    if (up) tmem_orders(tc + (uint32_t)((n + 1) * (n + 1) - c0 + 2 * mb - 3), n + 1, mb, y);
    if (n > 0) tmem_ld16_async(tp + (uint32_t)(n * n - c0 + 2 * mb - 1), f);
    else tmem_ld1(tp - (uint32_t)c0, f[1]);
    tmem_wait(f);
    if (up) tmem_wait(y);
    else
#pragma unroll
        for (int k = 0; k < 20; ++k) y[k] = 0u;
    if (mb == 0) {
        order_zero(y);
        f[0] = f[1];
        f[1] = 0u;
    }
    const float* k0 = cv + (n * (n + 1) / 2 + mb) * 8;
    // four orders at a time without branches (their chains interleave); orders past n are not stored
#pragma unroll
    for (int h = 0; h < 8; h += 4) {
        if (mb + h > n) break;
        float vo[8], vq[8];
#pragma unroll
        for (int i = h; i < h + 4; ++i) {
            const int m = mb + i;
            const float4 g = *reinterpret_cast<const float4*>(k0 + 8 * i);
            const float2 e = *reinterpret_cast<const float2*>(k0 + 8 * i + 4);
            const float ax = g.x * tx, ay = g.x * ty, bx = g.y * tx, by = g.y * ty, z = g.z * tz;
            const float dx = g.w * tx, dy = g.w * ty, ex = e.x * tx, ey = e.x * ty, fz = e.y * tz;
            auto F = [](uint32_t u) { return __uint_as_float(u); };
            const float mr = F(x[2 * i]), mi = F(x[2 * i + 1]), cr = F(x[2 * i + 2]), ci = F(x[2 * i + 3]);
            const float pr = m < n ? F(x[2 * i + 4]) : 0.f, pi = m < n ? F(x[2 * i + 5]) : 0.f;
            const float umr = F(y[2 * i]), umi = F(y[2 * i + 1]), ucr = F(y[2 * i + 2]), uci = F(y[2 * i + 3]),
                        upr = F(y[2 * i + 4]), upi = F(y[2 * i + 5]);  // degree n + 1
            const float o0 = fmaf(ax, pr, fmaf(-ay, pi, fmaf(bx, mr, fmaf(by, mi, fmaf(-z, ci, F(f[2 * i]))))));
            const float q0 = fmaf(ey, upr, fmaf(ex, upi, fmaf(dy, umr, fmaf(-dx, umi, fmaf(fz, ucr, cs * cr)))));
            const float o1 = fmaf(ax, pi, fmaf(ay, pr, fmaf(bx, mi, fmaf(-by, mr, fmaf(z, cr, F(f[2 * i + 1]))))));
            const float q1 = fmaf(ey, upi, fmaf(-ex, upr, fmaf(dy, umi, fmaf(dx, umr, fmaf(fz, uci, cs * ci)))));
            const bool zero = i == 0 && m == 0;
            vo[2 * (i - h)] = o0;
            vo[2 * (i - h) + 1] = zero ? o0 : o1;
            vq[2 * (i - h)] = q0;
            vq[2 * (i - h) + 1] = zero ? q0 : q1;
        }
        store_orders(op + (2 * (mb + h) - 1), vo, mb + h, n);
        store_orders(oc + (2 * (mb + h) - 1), vq, mb + h, n);
    }
#pragma unroll
    for (int k = 0; k < 20; ++k) x[k] = y[k];
}

// NPOT: two potentials, converted in the epilogue, or the one of the scalar case
template <int NPOT>
__global__ void __launch_bounds__(M2_THREADS, 1) k_tc_m2l(const __grid_constant__ M2lArgs a) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ M2lShared sh;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int S = a.nstages, nk = a.P / TC_KC;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh.tmem)),
                     "r"((uint32_t)M2_TMEM)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (t == 0) {
        for (int s = 0; s < M2_MAX_STAGES; ++s) {
            mbar_init(&sh.full_a[s], M2_PROD_WARPS / M2_GROUPS);
            mbar_init(&sh.full_b[s], 1);
            mbar_init(&sh.empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&sh.acc_full[b], 1);
            mbar_init(&sh.acc_empty[b], M2_EPI_WARPS);
        }
        mbar_init(&sh.done, 1);
        sh.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (NPOT == 2) {
        float* cv = reinterpret_cast<float*>(smem + (size_t)S * a.stage_bytes);
        for (int e = t; e < conv_floats(a.p); e += M2_THREADS) cv[e] = a.conv[e];
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh.tmem;
    const int c_beg = a.choff[a.g0];
    const int nwork = (a.choff[a.g1] - c_beg) * a.nranges;  // items: (chunk of <= 128 pairs, range)
    float* conv = reinterpret_cast<float*>(smem + (size_t)S * a.stage_bytes);  // the conversion table (NPOT = 2)
    float* stg = conv + (NPOT == 2 ? conv_floats(a.p) : 0);  // the epilogue warps' staging
    const int mine = nwork > (int)blockIdx.x ? (nwork - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;

    if (warp >= M2_EPI_WARPS && warp < M2_EPI_WARPS + M2_PROD_WARPS) {
        // ---- gather and split.  The two groups of four warps take alternate K chunks, so that the
        // store, the proxy fence and the arrival of one overlap the other's.  This thread: rows
        // 32 (w % 4) + 8 j + lane % 8, 16 bytes at k group lane / 8.
        constexpr int RJ = 4;
        const int pw = warp - M2_EPI_WARPS, grp = pw / (M2_PROD_WARPS / M2_GROUPS);
        const int row0 = (pw % (M2_PROD_WARPS / M2_GROUPS)) * 32 + (lane & 7), kg = lane >> 3;
        const int total = mine * nk;  // K chunks of this CTA's items
        int cur[RJ], nxt[RJ];
        // source boxes of this thread's rows in the CTA's n-th item
        auto ids = [&](int n, int (&s)[RJ]) {
#pragma unroll
            for (int j = 0; j < RJ; ++j) s[j] = -1;
            if (n >= mine) return;
            const int4 ch = a.chunks[c_beg + ((int)blockIdx.x + n * (int)gridDim.x) / a.nranges];
#pragma unroll
            for (int j = 0; j < RJ; ++j)
                if (row0 + 8 * j < ch.z) {
                    const int2 pr = a.pairs[ch.y + row0 + 8 * j];
                    s[j] = a.swap ? pr.y : pr.x;
                }
        };
        float4 v[NPOT][RJ], w[NPOT][RJ];
        auto load = [&](const int (&s)[RJ], int k, float4 (&d)[NPOT][RJ]) {
#pragma unroll
            for (int q = 0; q < NPOT; ++q)
#pragma unroll
                for (int j = 0; j < RJ; ++j)
                    d[q][j] = s[j] >= 0 ? __ldg(reinterpret_cast<const float4*>(a.in + (int64_t)s[j] * a.ld + q * a.P +
                                                                               (nk - 1 - k) * TC_KC + kg * 4))
                                        : make_float4(0.f, 0.f, 0.f, 0.f);
        };
        int have = grp / nk;  // the item whose ids are in cur; nxt holds the following item's
        if (grp < total) {
            ids(have, cur);
            ids(have + 1, nxt);
            load(cur, grp % nk, v);
        }
        for (int g = grp; g < total; g += M2_GROUPS) {
            if (g + M2_GROUPS < total) {
                const int n2 = (g + M2_GROUPS) / nk, k2 = (g + M2_GROUPS) - n2 * nk;
                if (n2 != have) {
                    if (n2 == have + 1) {
#pragma unroll
                        for (int j = 0; j < RJ; ++j) cur[j] = nxt[j];
                    } else {
                        ids(n2, cur);  // items of one K chunk (p = 4)
                    }
                    have = n2;
                    ids(have + 1, nxt);
                }
                load(cur, k2, w);
            }
            const int st = g % S;
            if (!__all_sync(0xffffffffu, m2_wait(&sh.empty[st], ((uint32_t)(g / S) & 1u) ^ 1u, sh, a))) break;
            unsigned char* base = smem + (size_t)st * a.stage_bytes;
#pragma unroll
            for (int q = 0; q < NPOT; ++q)
#pragma unroll
                for (int j = 0; j < RJ; ++j) {
                    const uint32_t o = tile_off(row0 + 8 * j, kg * 4);
                    const float4 x = v[q][j];
                    float4 h, l;
                    h.x = tf32_rna(x.x);
                    h.y = tf32_rna(x.y);
                    h.z = tf32_rna(x.z);
                    h.w = tf32_rna(x.w);
                    l.x = tf32_rna(x.x - h.x);
                    l.y = tf32_rna(x.y - h.y);
                    l.z = tf32_rna(x.z - h.z);
                    l.w = tf32_rna(x.w - h.w);
                    *reinterpret_cast<float4*>(base + (2 * q) * M2_X_TILE + o) = h;
                    *reinterpret_cast<float4*>(base + (2 * q + 1) * M2_X_TILE + o) = l;
                }
            fence_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.full_a[st]);
#pragma unroll
            for (int q = 0; q < NPOT; ++q)
#pragma unroll
                for (int j = 0; j < RJ; ++j) v[q][j] = w[q][j];
        }
    } else if (warp == M2_EPI_WARPS + M2_PROD_WARPS) {
        if (lane == 0) {
            // ---- operator tiles
            int st = 0;
            uint32_t ph = 1;
            int64_t issued = 0;
            bool ok = true;
            for (int item = blockIdx.x; item < nwork && ok; item += gridDim.x) {
                const int r = item % a.nranges;
                const int slot = a.chunks[c_beg + item / a.nranges].x % a.ngroups;
                const uint32_t bytes = (uint32_t)a.nlen[r] * TC_KC * 4 * 2;
                const float* src = a.tiles + (int64_t)slot * a.group_stride + a.roff[r];
                for (int k = 0; k < nk; ++k) {
                    ok = m2_wait(&sh.empty[st], ph, sh, a);
                    if (!ok) break;
                    mbar_expect_tx(&sh.full_b[st], bytes);
                    bulk_copy(smem + (size_t)st * a.stage_bytes + 2 * NPOT * M2_X_TILE, src + (int64_t)(nk - 1 - k) * (bytes / 4),
                              bytes, &sh.full_b[st]);
                    ++issued;
                    if (++st == S) {
                        st = 0;
                        ph ^= 1u;
                    }
                }
            }
            // every copy has landed before the CTA may end: the last one of each stage
            for (int s = 0; s < S; ++s) {
                const int64_t uses = issued / S + (s < issued % S);
                if (uses > 0) mbar_wait(&sh.full_b[s], (uint32_t)((uses - 1) & 1));
            }
        }
    } else if (warp == M2_EPI_WARPS + M2_PROD_WARPS + 1) {
        if (lane == 0) {
            // ---- MMA issue
            int st = 0, n = 0;
            uint32_t ph = 0;
            bool ok = true;
            const uint32_t lbo = 128, sbo = (TC_KC / 4) * 128;
            for (int item = blockIdx.x; item < nwork && ok; item += gridDim.x, ++n) {
                const int nlen = a.nlen[item % a.nranges], b = n % a.nbuf;
                const uint32_t idesc = make_idesc(TC_PAIRS, nlen);
                const uint32_t d0 = tmem + (uint32_t)(b * (M2_TMEM / a.nbuf)) + acc_base(item % a.nranges);
                ok = m2_wait(&sh.acc_empty[b], ((uint32_t)(n / a.nbuf) & 1u) ^ 1u, sh, a);
                if (!ok) break;
                for (int k = 0; k < nk; ++k) {
                    ok = m2_wait(&sh.full_a[st], ph, sh, a) && m2_wait(&sh.full_b[st], ph, sh, a);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t base = smem_u32(smem + (size_t)st * a.stage_bytes);
                    const uint32_t bh = base + 2 * NPOT * M2_X_TILE, bl = bh + (uint32_t)nlen * TC_KC * 4;
                    // the small cross products first, then hi.hi (see the top)
#pragma unroll
                    for (int part = 0; part < 3; ++part)
#pragma unroll
                        for (int ks = TC_KC / 8 - 1; ks >= 0; --ks) {
                            const uint32_t step = ks * 2 * 128;
                            const uint64_t B = make_desc((part == 0 ? bl : bh) + step, lbo, sbo);
#pragma unroll
                            for (int q = 0; q < NPOT; ++q) {
                                const uint64_t X =
                                    make_desc(base + (2 * q + (part == 1)) * M2_X_TILE + step, lbo, sbo);
                                mma_tf32(d0 + (uint32_t)(q * nlen), X, B, idesc,
                                         (k == 0 && part == 0 && ks == TC_KC / 8 - 1) ? 0 : 1);
                            }
                        }
                    mma_commit(&sh.empty[st]);
                    if (++st == S) {
                        st = 0;
                        ph ^= 1u;
                    }
                }
                if (ok) mma_commit(&sh.acc_full[b]);
            }
            mma_commit(&sh.done);
            mbar_wait(&sh.done, 0);  // nothing in flight when TMEM is freed
        }
    } else {
        // ---- epilogue: thread = pair 32 (warp % 4) + lane; the two warps of a lane quarter share the
        // columns.  Bands of columns are staged [pair][column] and added to the pairs' rows by the copy engine
        // while the next band is read.
        const int quarter = warp & 3, half = warp >> 2, row = quarter * 32 + lane;
        float* st_p = stg + row * M2_STG_LD;
        float* st_c = st_p + TC_PAIRS * M2_STG_LD;  // chi
        auto release = [&](int b) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.acc_empty[b]);
        };
        for (int n = 0; n < mine; ++n) {
            const int item = (int)blockIdx.x + n * (int)gridDim.x, r = item % a.nranges, b = n % a.nbuf;
            const int4 ch = a.chunks[c_beg + item / a.nranges];
            const int2 pr = row < ch.z ? a.pairs[ch.y + row] : make_int2(-1, -1);
            const int dst = a.swap ? pr.x : pr.y;
            float* out = a.out + (int64_t)dst * a.ld;  // not used where dst < 0
            // where a wait gave up, all epilogue warps leave together, at this item
            if (epi_any(!m2_wait(&sh.acc_full[b], (uint32_t)(n / a.nbuf) & 1u, sh, a))) break;
            tc_fence_after();
            const int n0 = a.n0[r], n1 = a.n1[r], c0 = a.c0[r], nlen = a.nlen[r];
            const uint32_t tp =
                tmem + (uint32_t)(b * (M2_TMEM / a.nbuf)) + acc_base(r) + ((uint32_t)(quarter * 32) << 16);
            if (NPOT == 1) {
                const int ncols = n1 * n1 - c0;  // a multiple of 4
                // each warp stages and adds its own 32 columns of a band
                for (int cb = 32 * half; cb < nlen; cb += M2_BAND) {
                    bulk_wait_read();
                    __syncwarp();
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        if (cb + 16 * k >= nlen) break;
                        uint32_t x[16];
                        tmem_ld16_async(tp + (uint32_t)(cb + 16 * k), x);
                        tmem_wait(x);
#pragma unroll
                        for (int i = 0; i < 16; i += 4)
                            *reinterpret_cast<uint4*>(st_p + 32 * half + 16 * k + i) =
                                make_uint4(x[i], x[i + 1], x[i + 2], x[i + 3]);
                    }
                    fence_async_smem();
                    __syncwarp();
                    const int nc = min(32, ncols - cb);
                    if (dst >= 0 && nc > 0) bulk_add(out + c0 + cb, st_p + 32 * half, (uint32_t)nc * 4);
                    bulk_commit();
                }
                release(b);
            } else {
                const uint32_t tc = tp + (uint32_t)nlen;
                const float4 tv = __ldg(reinterpret_cast<const float4*>(a.tvec) + ch.x % a.ngroups);
                for (int na = n0; na < n1;) {
                    // degrees [na, nb) fit the band; an even nb where there is one, so that the band
                    // [s0, s1) of whole quads holds no columns of other degrees (those are zero)
                    int nb = na + 1;
                    while (nb < n1 && (nb + 1) * (nb + 1) - na * na <= M2_BAND) ++nb;
                    if ((nb & 1) && nb < n1 && nb > na + 1) --nb;
                    const int s0 = na * na & ~3, s1 = (nb * nb + 3) & ~3;
                    bulk_wait_read();
                    quarter_sync(quarter);
                    if (half == 0) {
                        if (na & 1) st_p[0] = st_c[0] = 0.f;
                        if (nb & 1)
                            for (int c = nb * nb - s0; c < s1 - s0; ++c) st_p[c] = st_c[c] = 0.f;
                    }
                    // runs of degrees in blocks of eight orders: one block is split between the two warps
                    // of a lane quarter by degree, several are taken in turn
                    for (int mb = 0; mb < nb; mb += 8) {
                        int d0 = max(na, mb), d1 = nb;
                        if (nb <= 8) {
                            const int mid = (na + nb + 1) / 2;
                            if (half) d0 = mid;
                            else d1 = mid;
                        } else if (((mb >> 3) & 1) != half) {
                            continue;
                        }
                        if (d0 >= d1) continue;
                        uint32_t x[20];
                        tmem_orders(tc + (uint32_t)(d0 * d0 - c0 + 2 * mb - 3), d0, mb, x);
                        tmem_wait(x);
                        if (mb == 0) order_zero(x);
                        for (int dn = d0; dn < d1; ++dn) {
                            const int at = dn * dn - s0;
                            convert_orders(conv, tp, tc, c0, a.p, dn, mb, tv.x, tv.y, tv.z, a.chi_scale, x,
                                                 st_p + at, st_c + at);
                        }
                    }
                    if (nb == n1) release(b);
                    fence_async_smem();
                    quarter_sync(quarter);
                    // one warp adds phi, the other chi
                    if (dst >= 0)
                        bulk_add(out + half * a.P + s0, half ? st_c : st_p, (uint32_t)(s1 - s0) * 4);
                    bulk_commit();
                    na = nb;
                }
            }
        }
        bulk_wait_all();
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)M2_TMEM) : "memory");
}

// tiles[group][range][k chunk][hi | lo][tile_off order] of the translation block T of the fused
// tables: T[k][c] = ops[group][k ldo + c], k, c < P
__global__ void k_m2l_tiles(const float* __restrict__ ops, int64_t op_floats, int ldo, M2lArgs a,
                            float* __restrict__ tiles) {
    for (int g = blockIdx.x; g < a.ngroups; g += gridDim.x) {
        const float* Ag = ops + (int64_t)g * op_floats;
        float* tg = tiles + (int64_t)g * a.group_stride;
        for (int r = 0; r < a.nranges; ++r) {
            const int nlen = a.nlen[r], tile = nlen * TC_KC;
            for (int e = threadIdx.x; e < a.P / TC_KC * tile; e += blockDim.x) {
                const int i = e / tile, q = e - i * tile, k = q / nlen, c = q - k * nlen;
                const int kk = i * TC_KC + k, cc = a.c0[r] + c;
                const float v = cc < a.P ? Ag[(int64_t)kk * ldo + cc] : 0.f;
                const float h = tf32_rna(v);
                float* base = tg + a.roff[r] + (int64_t)i * 2 * tile;
                const uint32_t o = tile_off(c, k) / 4;
                base[o] = h;
                base[tile + o] = tf32_rna(v - h);
            }
        }
    }
}

int m2l_fixed_smem(int p, int npot) {
    return (npot * TC_PAIRS * M2_STG_LD + (npot == 2 ? conv_floats(p) : 0)) * 4;
}

// One past the last column that the epilogue reads of chi of the degrees [n0, n1) and their
// halo (tmem_orders), counted from the first column of the range.
int chi_read_end(int p, int n0, int n1) {
    int end = 0;
    for (int n = n0; n < n1; ++n)
        for (int mb = 0; mb <= n; mb += 8)
            for (int N = n; N <= std::min(n + 1, p - 1); ++N)
                end = std::max(end, N * N - n0 * n0 + 2 * mb - 3 + 18 + (mb + 8 <= N ? 2 : 0));
    return end;
}

// Ranges, strides and stages of truncation number p.  One range of output degrees holds all
// columns up to p = 16 (2 x 256 of the 512); above, each range carries the halo degree that its
// conversion reads.  The accumulators are double-buffered where two fit (the scalar case, p <= 8).
// Splitting p = 12 and 16 into ranges of 256 columns so that two fit was slower (sphere
// surface of 2^20, p = 12: products 3.6 ms against 1.8 without the epilogue, 9.3 against 4.9 with
// it): the narrow MMAs are bound by their operand reads from shared memory, and the reads of
// TMEM queue behind them.
M2lArgs m2l_layout(int p, int npot, int ngroups) {
    M2lArgs a{};
    a.p = p;
    a.P = p * p;
    a.ngroups = ngroups;
    a.nbuf = npot == 1 || p <= 8 ? 2 : 1;
    int64_t off = 0;
    int nmax = 0;
    for (int n0 = 0; n0 < p;) {
        const int r = a.nranges++, c0 = n0 * n0, room = M2_TMEM / a.nbuf - (r ? 16 : 0);
        if (r >= M2_MAX_RANGES) throw Error{LHV_EUNSUPPORTED, "M2L output ranges"};
        auto width = [&](int n1) {  // columns of the degrees [n0, n1) with their halo, in 16s
            const int hi = n1 < p && npot == 2 ? (n1 + 1) * (n1 + 1) : n1 * n1;
            return (hi - c0 + 15) / 16 * 16;
        };
        auto fits = [&](int n1) {
            const int w = width(n1);
            return w <= 256 && npot * w <= room && (npot == 1 || w + chi_read_end(p, n0, n1) <= room);
        };
        int n1 = n0 + 1;
        while (n1 < p && fits(n1 + 1)) ++n1;
        if (npot == 1 && n1 < p) n1 &= ~1;  // whole quads of columns
        if (n1 <= n0 || !fits(n1)) throw Error{LHV_EUNSUPPORTED, "M2L accumulators"};
        a.n0[r] = n0;
        a.n1[r] = n1;
        a.c0[r] = c0;
        a.nlen[r] = width(n1);
        a.roff[r] = off;
        off += (int64_t)(a.P / TC_KC) * 2 * a.nlen[r] * TC_KC;
        nmax = std::max(nmax, a.nlen[r]);
        n0 = n1;
    }
    a.group_stride = off;
    a.stage_bytes = 2 * npot * M2_X_TILE + 2 * nmax * TC_KC * 4;
    a.nstages = std::min(M2_MAX_STAGES, (M2_SMEM_MAX - m2l_fixed_smem(p, npot)) / a.stage_bytes);
    return a;
}

}  // namespace

bool tc_trans_supported(int p) { return p % 4 == 0 && p >= 4 && p <= 24; }

void tc_trans_tiles(Ctx* c, TransKind kind, const float* fused, int p, bool scalar, Buf& tiles) {
    const int ng = kind == TRANS_M2L ? NUM_OFFSETS : 8;
    M2lArgs a = m2l_layout(p, scalar ? 1 : 2, ng);
    const int64_t nt = a.group_stride * ng;
    // conversion table, then the translation vectors
    std::vector<float> tab((size_t)conv_floats(p), 0.f);
    const double in_chi = kind == TRANS_L2L ? 0.5 : 1.0;  // chi^ = in_chi T chi in these coefficients
    for (int n = 0; n < p; ++n)
        for (int m = 0; m <= n; ++m) {
            float* v = &tab[(size_t)(n * (n + 1) / 2 + m) * 8];
            const double two = m ? 1.0 : 2.0, one = m ? 1.0 : 0.0;
            if (n > 0) {
                v[0] = (float)(-two * in_chi * std::sqrt((double)(n - m) * (n + m + 1)) / (2.0 * n));
                v[1] = (float)(one * in_chi * std::sqrt((double)(n + m) * (n - m + 1)) / (2.0 * n));
                v[2] = (float)(in_chi * m / n);
            }
            if (n + 1 < p) {
                v[3] = (float)(one * in_chi * std::sqrt((double)(n - m + 1) * (n - m + 2)) / (2.0 * (n + 1)));
                v[4] = (float)(-two * in_chi * std::sqrt((double)(n + m + 1) * (n + m + 2)) / (2.0 * (n + 1)));
                v[5] = (float)(-in_chi * std::sqrt((double)(n + 1 - m) * (n + 1 + m)) / (n + 1));
            }
        }
    std::vector<int> offs, slot_of;
    m2l_offsets(offs, slot_of);
    for (int g = 0; g < ng; ++g)
        for (int k = 0; k < 4; ++k) {
            // M2L: t = target - source = -offset; L2L of child octant o: o - 0.5, in child sides
            const float o = (float)((g >> k) & 1);
            tab.push_back(k == 3 ? 0.f : kind == TRANS_M2L ? (float)-offs[3 * g + k] : o - 0.5f);
        }
    ensure(c, tiles, (nt + (int64_t)tab.size()) * (int64_t)sizeof(float));
    k_m2l_tiles<<<ng, 256, 0, stream_of(c)>>>(fused, 4 * (int64_t)a.P * a.P, 2 * a.P, a, tiles.as<float>());
    count_launch(c);
    check_launch("translation tiles");
    cuda_check(cudaMemcpyAsync(tiles.as<float>() + nt, tab.data(), tab.size() * sizeof(float), cudaMemcpyHostToDevice,
                               stream_of(c)),
               "translation tables");
    cuda_check(cudaStreamSynchronize(stream_of(c)), "translation tiles");
}

void run_tc_trans(Ctx* c, TransKind kind, const Grouped& gp, int g0, int g1, int p, bool scalar, const float* tiles,
                  const float* in, float* out, int64_t ld, int* err) {
    M2lArgs a = m2l_layout(p, scalar ? 1 : 2, kind == TRANS_M2L ? NUM_OFFSETS : 8);
    a.chunks = gp.chunks.as<int4>();
    a.pairs = gp.pairs.as<int2>();
    a.choff = gp.choff.as<int>();
    a.g0 = g0;
    a.g1 = g1;
    a.swap = kind == TRANS_L2L;
    a.in = in;
    a.out = out;
    a.ld = ld;
    a.tiles = tiles;
    a.conv = tiles + a.group_stride * a.ngroups;
    a.tvec = a.conv + conv_floats(p);
    a.chi_scale = kind == TRANS_M2L ? 1.0f : 0.5f;
    a.err = err;
    a.wait_limit = ctx_wait_limit(c);
    // above half an SM's shared memory: one CTA (and its 512 TMEM columns) per SM
    const size_t smem =
        std::max<size_t>((size_t)a.nstages * a.stage_bytes + m2l_fixed_smem(p, scalar ? 1 : 2), 120 * 1024);
    auto kernel = scalar ? k_tc_m2l<1> : k_tc_m2l<2>;
    cuda_check(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem), "translation smem");
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    kernel<<<sms, M2_THREADS, smem, stream_of(c)>>>(a);
    count_launch(c);
    check_launch("tc translation");
}

}  // namespace lhv
