// Grouped scatter GEMM: every dense translation of the FMM as "one operator,
// many boxes".
//
// A translation applies one of a few fixed real matrices A_g (M2L: one of 316
// offsets; M2M / L2L: one of 8 child octants; P2M / L2P coefficient maps: one
// matrix) to the coefficient vector of a source box and adds the result to a
// destination box.  Pairs (source, destination) are bucketed by operator g, and
// each CTA multiplies A_g (R x C, k-major in memory) by a chunk of up to NC
// gathered source vectors:  Y (R x NC) = A_g X (C x NC), then scatters Y.
// Every operator is therefore read once per chunk of NC pairs instead of once
// per pair, and all levels of an M2L pass run in one launch (the scaled
// operators are level independent).
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "lhv_internal.cuh"
#include "lhv_group.cuh"

namespace lhv {

namespace {

__global__ void k_zero_int(int n, int* a) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) a[i] = 0;
}

__global__ void k_chunk_counts(int ng, const int* __restrict__ gcount, int nc, int* __restrict__ cc) {
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < ng; g += gridDim.x * blockDim.x)
        cc[g] = (gcount[g] + nc - 1) / nc;
}

__global__ void k_chunk_fill(int ng, const int* __restrict__ gcount, const int* __restrict__ goff,
                             const int* __restrict__ choff, int nc, int4* __restrict__ chunks) {
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < ng; g += gridDim.x * blockDim.x) {
        const int cnt = gcount[g], base = goff[g], c0 = choff[g];
        for (int k = 0; k * nc < cnt; ++k) chunks[c0 + k] = make_int4(g, base + k * nc, min(nc, cnt - k * nc), 0);
    }
}

__global__ void k_copy_int(int n, const int* __restrict__ a, int* __restrict__ b) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) b[i] = a[i];
}

// the totals of the exclusive scans go one past the end: off[ng] = total
__global__ void k_set_total(int ng, const int* __restrict__ cnt, int* __restrict__ off) {
    if (threadIdx.x == 0 && blockIdx.x == 0) off[ng] = (ng > 0 ? off[ng - 1] + cnt[ng - 1] : 0);
}

// The children of the levels 3 .. L by (level, octant).  Block b of nblk takes a contiguous range of the
// real boxes; FILL = false counts them per group to cnt[group][b], and the last block turns the
// counts into positions, choff[group] into the group's first chunk (choff[ngroups]: their number)
// and lists the chunks; FILL = true writes the pairs (child, parent) there.  Two launches where ten (count,
// scan, totals, cursors, fill, and three for the chunks) took 25 to 60 us, twice an evaluation.
constexpr int OCT_GROUPS = 8 * MAX_LEVELS;
struct OctLevels {
    int L;
    int off[MAX_LEVELS + 1];
};
template <bool FILL>
__global__ void __launch_bounds__(256) k_oct_list(OctLevels lv, const int* __restrict__ loff,
                                                  const uint64_t* __restrict__ bkey, const int* __restrict__ bparent,
                                                  int nblk, int* __restrict__ cnt, int nc, int* __restrict__ choff,
                                                  int4* __restrict__ chunks, int2* __restrict__ pairs,
                                                  int* __restrict__ ticket) {
    __shared__ int at[OCT_GROUPS], first[OCT_GROUPS + 1], chunk0[OCT_GROUPS + 1], lo[MAX_LEVELS + 2];
    const int ng = (lv.L - 2) * 8, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    for (int l = t; l <= lv.L + 1; l += blockDim.x) lo[l] = loff[l];
    for (int g = t; g < ng; g += blockDim.x) at[g] = FILL ? cnt[g * nblk + blockIdx.x] : 0;
    __syncthreads();
    const int64_t nb = lo[lv.L + 1] - lo[3];
    const int b0 = lo[3] + (int)(nb * blockIdx.x / nblk), b1 = lo[3] + (int)(nb * (blockIdx.x + 1) / nblk);
    for (int rb = b0 + t; rb < b1; rb += blockDim.x) {
        int l = 3;
        while (l < lv.L && rb >= lo[l + 1]) ++l;
        const int b = lv.off[l] + (rb - lo[l]);
        const int pos = atomicAdd(&at[(l - 3) * 8 + (int)(bkey[b] & 7ull)], 1);
        if (FILL) pairs[pos] = make_int2(b, lv.off[l - 1] + bparent[b]);
    }
    if (FILL) return;
    __syncthreads();
    for (int g = t; g < ng; g += blockDim.x) __stcg(cnt + g * nblk + blockIdx.x, at[g]);
    if (!last_block(ticket, nblk)) return;
    for (int g = warp; g < ng; g += 8) {
        int carry = 0;
        for (int i0 = 0; i0 < nblk; i0 += 32) {
            const int v = i0 + lane < nblk ? __ldcg(cnt + g * nblk + i0 + lane) : 0;
            int x = v;
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (i0 + lane < nblk) __stcg(cnt + g * nblk + i0 + lane, carry + x - v);
            carry += __shfl_sync(0xffffffffu, x, 31);
        }
        if (lane == 0) at[g] = carry;
    }
    __syncthreads();
    if (t == 0) {
        int f = 0, c = 0;
        for (int g = 0; g < ng; ++g) {
            first[g] = f;
            chunk0[g] = c;
            f += at[g];
            c += (at[g] + nc - 1) / nc;
        }
        chunk0[ng] = c;
    }
    __syncthreads();
    for (int i = t; i < ng * nblk; i += blockDim.x) __stcg(cnt + i, __ldcg(cnt + i) + first[i / nblk]);
    for (int g = t; g <= ng; g += blockDim.x) choff[g] = chunk0[g];
    for (int c = t; c < chunk0[ng]; c += blockDim.x) {
        int a = 0, b = ng - 1;  // the last group whose first chunk is <= c
        while (a < b) {
            const int mid = (a + b + 1) >> 1;
            if (chunk0[mid] <= c) a = mid; else b = mid - 1;
        }
        const int k = (c - chunk0[a]) * nc;
        chunks[c] = make_int4(a, first[a] + k, min(nc, at[a] - k), 0);
    }
}

constexpr int GG_THREADS = 256;
constexpr int KC = 16;  // operator rows (input coefficients) staged per step
constexpr int GG_DEPTH = 4;  // steps of operator rows in flight

// RT = 16 * TM output rows per work item; NC columns, TN = NC / 16 per thread.  SPLIT: the translations
// between levels (split K, chunks in parts, pairs swapped, items in turn); M2L's instances stay free of
// all that.  GemmArgs grows with care: two more ints in it, and the compiler gave the NC = 32, TM = 8
// instance 79 registers instead of 106 (M2L of levels of p = 18 to 20 45 ms instead of 35).
template <typename T, int NC, int TM, bool SPLIT>
__global__ void __launch_bounds__(GG_THREADS) k_group_gemm(GemmArgs<T> a) {
    constexpr int TN = NC / 16;
    constexpr int RT = 16 * TM;
    constexpr int XS = NC + 4;  // row stride of X (keeps 16-byte alignment, breaks the worst bank conflicts)
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* X = reinterpret_cast<T*>(smem_raw);       // [C][XS]
    T* A = X + (size_t)a.C * XS;                 // [2][KC][RT] (double buffer)
    __shared__ int s_work;
    __shared__ int s_src[NC], s_dst[NC];
    const int t = threadIdx.x;
    const int cg = t % 16, rg = t / 16;
    const int nrt = (a.R + RT - 1) / RT;
    const int c_beg = a.choff[a.g0], c_end = a.choff[a.g1];
    // split K: segment ks covers inputs [ks kper, (ks + 1) kper) (kper a multiple of KC); the
    // segments' partial products meet in the atomic adds of the epilogue
    const int nks = SPLIT && a.ksplit > 1 ? a.ksplit : 1;
    const int kper = SPLIT ? (a.C + nks * KC - 1) / (nks * KC) * KC : a.C;
    const int sub = SPLIT && (a.between & BETWEEN_WIDE) ? TC_PAIRS / NC : 1;  // parts of a chunk
    const int nwork = SPLIT ? (c_end - c_beg) * sub * nrt * nks : (c_end - c_beg) * nrt;
    int last_key = -1;
    int turn = SPLIT ? (int)blockIdx.x : 0;
    for (;;) {
        __syncthreads();
        int w;
        if (SPLIT && !a.work) {
            w = turn;
            turn += gridDim.x;
        } else {
            if (t == 0) s_work = atomicAdd(a.work, 1);
            __syncthreads();
            w = s_work;
        }
        if (w >= nwork) break;
        const int ks = SPLIT ? w % nks : 0, wc = SPLIT ? w / nks : w;
        const int part = wc / nrt, rt = wc % nrt;  // part: NC pairs of a chunk
        const int kseg0 = ks * kper, kseg1 = SPLIT ? min(a.C, kseg0 + kper) : a.C;
        if (kseg0 >= kseg1) continue;  // block-uniform: an empty last segment
        const int4 ch = a.chunks[c_beg + (SPLIT ? part / sub : part)];
        const int skip = SPLIT ? part % sub * NC : 0;
        const int g = ch.x, p0 = ch.y + skip, np = SPLIT ? min(NC, ch.z - skip) : ch.z;
        if (SPLIT && np <= 0) continue;
        const int r0 = rt * RT;
        const int key = part * nks + ks;
        if (key != last_key) {
            if (t < NC) {
                if (t < np) {
                    const int2 pr = a.pairs[p0 + t];
                    s_src[t] = SPLIT && (a.between & BETWEEN_SWAPPED) ? pr.y : pr.x;
                    s_dst[t] = SPLIT && (a.between & BETWEEN_SWAPPED) ? pr.x : pr.y;
                } else {
                    s_src[t] = -1;
                    s_dst[t] = -1;
                }
            }
            __syncthreads();
            const int klen = kseg1 - kseg0;
            for (int e = t; e < klen * NC; e += GG_THREADS) {
                const int col = e / klen, k = kseg0 + (e - col * klen);
                const int s = s_src[col];
                X[k * XS + col] = (s >= 0) ? a.in[(int64_t)s * a.ldin + k] : (T)0;
            }
            last_key = key;
        }
        // rows of this thread: r0 + rg*TM + j; skip the zero block (rows >= psplit read inputs >= psplit only)
        const int myrow0 = r0 + rg * TM;
        const int pcol = a.psplit_c > 0 ? a.psplit_c : a.psplit;
        const int kstart = (a.psplit > 0 && myrow0 >= a.psplit) ? pcol : 0;
        const int kb = max((a.psplit > 0 && r0 >= a.psplit) ? pcol : 0, kseg0);  // this item's K range [kb, ke)
        const int ke = kseg1;
        T acc[TM][TN];
#pragma unroll
        for (int j = 0; j < TM; ++j)
#pragma unroll
            for (int c = 0; c < TN; ++c) acc[j][c] = 0;
        const T* Ag = a.ops + (int64_t)(g % a.ops_mod) * a.C * a.R;
        // operator rows [kc, kc + KC) of this row tile: each thread owns EPT entries of a step;
        // the entries of the next GG_DEPTH steps are in flight in registers (a ring indexed at
        // compile time) while the current step computes from shared memory
        constexpr int EPT = KC * RT / GG_THREADS;
        T nxt[GG_DEPTH][EPT];
        auto load = [&](int kc, T(&dst)[EPT]) {
#pragma unroll
            for (int q = 0; q < EPT; ++q) {
                const int e = t + q * GG_THREADS;
                const int kk = e / RT, r = e - kk * RT;
                const int k = kc + kk, row = r0 + r;
                dst[q] = (k < ke && row < a.R) ? Ag[(int64_t)k * a.R + row] : (T)0;
            }
        };
#pragma unroll
        for (int d = 0; d < GG_DEPTH; ++d) load(kb + d * KC, nxt[d]);
        int buf = 0;
        for (int kc0 = kb; kc0 < ke; kc0 += GG_DEPTH * KC) {
#pragma unroll
            for (int d = 0; d < GG_DEPTH; ++d) {
                const int kc = kc0 + d * KC;
                if (kc >= ke) break;
                T* Ab = A + buf * KC * RT;
#pragma unroll
                for (int q = 0; q < EPT; ++q) Ab[t + q * GG_THREADS] = nxt[d][q];
                __syncthreads();
                if (kc + GG_DEPTH * KC < ke) load(kc + GG_DEPTH * KC, nxt[d]);
                const int kn = min(KC, ke - kc);
                for (int kk = 0; kk < kn; ++kk) {
                    if (kc + kk < kstart) continue;
                    T av[TM], xv[TN];
#pragma unroll
                    for (int j = 0; j < TM; ++j) av[j] = Ab[kk * RT + rg * TM + j];
#pragma unroll
                    for (int c = 0; c < TN; ++c) xv[c] = X[(kc + kk) * XS + cg * TN + c];
#pragma unroll
                    for (int j = 0; j < TM; ++j)
#pragma unroll
                        for (int c = 0; c < TN; ++c) acc[j][c] += av[j] * xv[c];
                }
                buf ^= 1;
            }
        }
#pragma unroll
        for (int c = 0; c < TN; ++c) {
            const int col = cg * TN + c;
            const int d = s_dst[col];
            if (d < 0) continue;
            T* o = a.out + (int64_t)d * a.ldout;
#pragma unroll
            for (int j = 0; j < TM; ++j) {
                const int row = myrow0 + j;
                if (row >= a.R) continue;
                const T v = acc[j][c] * a.scale;
                if (a.mode == GEMM_STORE) o[row] = v;
                else if (a.mode == GEMM_ADD) o[row] += v;
                else atomicAdd(o + row, v);
            }
        }
    }
}

template <typename T, int NC, int TM, bool SPLIT>
void launch_gemm(Ctx* c, GemmArgs<T> a) {
    const size_t smem = sizeof(T) * ((size_t)a.C * (NC + 4) + 2 * (size_t)KC * 16 * TM);
    cuda_check(cudaFuncSetAttribute(k_group_gemm<T, NC, TM, SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
               "gemm attr");
    int per_sm = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_group_gemm<T, NC, TM, SPLIT>, GG_THREADS, smem);
    if (per_sm < 1) per_sm = 1;
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // a level whose items all start at once takes them in turn; more, of uneven work (the zero
    // block), are handed out by a counter, which costs the clearing (FP64 ring of 32,768, M2M 0.90 ms in
    // turn, 0.75 by the counter)
    const int64_t items = (a.pairs_hint / NC + (a.g1 - a.g0)) * ((a.R + 16 * TM - 1) / (16 * TM)) * std::max(a.ksplit, 1);
    if (SPLIT && a.pairs_hint > 0 && items <= (int64_t)sms * per_sm) a.work = nullptr;
    else cuda_check(cudaMemsetAsync(a.work, 0, 4, stream_of(c)), "gemm work");
    k_group_gemm<T, NC, TM, SPLIT><<<sms * per_sm, GG_THREADS, smem, stream_of(c)>>>(a);
    count_launch(c);
    check_launch("group gemm");
}

}  // namespace

void grouped_finish(Ctx* c, Grouped& gp, int nc) {
    // pairs are in place; build the chunk list (group-major, NC pairs per chunk)
    cudaStream_t s = stream_of(c);
    const int ng = gp.ngroups;
    int* cc = gp.tmp.as<int>();
    k_chunk_counts<<<grid_for(ng, 128), 128, 0, s>>>(ng, gp.gcount.as<int>(), nc, cc);
    count_launch(c);
    exclusive_scan(c, ng, cc, gp.choff.as<int>(), gp.scan_tmp.as<int>(), nullptr);
    k_set_total<<<1, 32, 0, s>>>(ng, cc, gp.choff.as<int>());
    count_launch(c);
    k_chunk_fill<<<grid_for(ng, 128), 128, 0, s>>>(ng, gp.gcount.as<int>(), gp.goff.as<int>(), gp.choff.as<int>(), nc,
                                                   gp.chunks.as<int4>());
    count_launch(c);
    check_launch("chunks");
}

void oct_list(Ctx* c, const TreeBufs& tb, const Levels& lv, Grouped& gp, int nc) {
    const int nb = lv.off[lv.L + 1] - lv.off[3];
    gp.ngroups = (lv.L - 2) * 8;
    gp.nc = nc;
    const int nblk = grid_for(nb, 256, 64);
    ensure(c, gp.gcount, gp.ngroups * nblk * 4);
    ensure(c, gp.choff, (gp.ngroups + 1) * 4);
    ensure(c, gp.pairs, std::max(nb, 1) * (int64_t)8);
    ensure(c, gp.chunks, (int64_t)(nb / nc + gp.ngroups + 1) * 16);
    ensure(c, gp.work, 64);
    OctLevels ol{};
    ol.L = lv.L;
    for (int l = 0; l <= MAX_LEVELS; ++l) ol.off[l] = lv.off[l];
    const auto pass = [&](auto fill) {
        k_oct_list<decltype(fill)::value><<<nblk, 256, 0, stream_of(c)>>>(
            ol, tb.counts.as<int>() + 32, tb.bkey.as<uint64_t>(), tb.bparent.as<int>(), nblk, gp.gcount.as<int>(), nc,
            gp.choff.as<int>(), gp.chunks.as<int4>(), gp.pairs.as<int2>(), &tb.params.as<TreeParams>()->ticket);
        count_launch(c);
    };
    pass(std::false_type{});
    pass(std::true_type{});
    check_launch("level pairs");
}

void grouped_prepare(Ctx* c, Grouped& gp, int ngroups, int64_t max_pairs, int nc) {
    gp.ngroups = ngroups;
    ensure(c, gp.gcount, (ngroups + 1) * 4);
    ensure(c, gp.goff, (ngroups + 1) * 4);
    ensure(c, gp.gcursor, (ngroups + 1) * 4);
    ensure(c, gp.choff, (ngroups + 1) * 4);
    ensure(c, gp.tmp, (ngroups + 1) * 4);
    ensure(c, gp.scan_tmp, (scan_tmp_ints(ngroups + 1) + 64) * 4);
    ensure(c, gp.pairs, std::max<int64_t>(max_pairs, 1) * 8);
    ensure(c, gp.chunks, (max_pairs / nc + ngroups + 1) * 16);
    ensure(c, gp.work, 64);
    k_zero_int<<<grid_for(ngroups + 1, 128), 128, 0, stream_of(c)>>>(ngroups + 1, gp.gcount.as<int>());
    count_launch(c);
}

void grouped_offsets(Ctx* c, Grouped& gp) {
    cudaStream_t s = stream_of(c);
    exclusive_scan(c, gp.ngroups, gp.gcount.as<int>(), gp.goff.as<int>(), gp.scan_tmp.as<int>(), nullptr);
    k_set_total<<<1, 32, 0, s>>>(gp.ngroups, gp.gcount.as<int>(), gp.goff.as<int>());
    count_launch(c);
    k_copy_int<<<grid_for(gp.ngroups + 1, 128), 128, 0, s>>>(gp.ngroups + 1, gp.goff.as<int>(), gp.gcursor.as<int>());
    count_launch(c);
}

template <typename T>
int gemm_nc(int C) {
    // largest NC whose gathered X fits next to the operator stage in ~200 KB
    const int limit = 200 * 1024;
    for (int nc : {64, 32, 16})
        if ((size_t)C * (nc + 4) * sizeof(T) + 2 * (size_t)KC * 128 * sizeof(T) <= (size_t)limit) return nc;
    return 16;
}

template <int NC, bool SPLIT = false, typename T>
static void launch_tm(Ctx* c, const GemmArgs<T>& a, int tm) {
    if (tm == 8) launch_gemm<T, NC, 8, SPLIT>(c, a);
    else if (tm == 4) launch_gemm<T, NC, 4, SPLIT>(c, a);
    else launch_gemm<T, NC, 2, SPLIT>(c, a);
}

template <typename T>
void run_group_gemm(Ctx* c, const Grouped& gp, GemmArgs<T> a) {
    a.chunks = gp.chunks.as<int4>();
    a.pairs = gp.pairs.as<int2>();
    a.choff = gp.choff.as<int>();
    a.work = gp.work.as<int>();
    // a list of the tensor cores' wide chunks: each as several items of 16 pairs
    const int nc = gp.nc == TC_PAIRS ? 16 : gp.nc;
    if (nc != gp.nc) a.between |= BETWEEN_WIDE;
    // rows per tile 16 TM: the tallest tile that still leaves every SM a few work items
    // (a small level's few chunks would otherwise run as a handful of long serial tiles)
    int tm = 8;
    if (a.pairs_hint > 0) {
        const int64_t chunks = a.pairs_hint / nc + (a.g1 - a.g0);
        while (tm > 2 && chunks * ((a.R + 16 * tm - 1) / (16 * tm)) < 4 * 152) tm /= 2;
    }
    // split K when the items would leave most resident blocks idle (a short level's few chunks
    // each run one long serial K loop); only where the outputs are added atomically anyway
    a.ksplit = 1;
    if (a.between && nc == 16 && a.mode == GEMM_ATOMIC && a.pairs_hint > 0) {
        const int64_t items = (a.pairs_hint / nc + (a.g1 - a.g0)) * ((a.R + 16 * tm - 1) / (16 * tm));
        while (a.ksplit < 8 && items * a.ksplit < 2 * 152 * 4 && a.C >= 4 * KC * a.ksplit) a.ksplit *= 2;
    }
    if (a.between && nc == 16) launch_tm<16, true>(c, a, tm);
    else if (nc == 64) launch_tm<64>(c, a, tm);
    else if (nc == 32) launch_tm<32>(c, a, tm);
    else launch_tm<16>(c, a, tm);
}

template int gemm_nc<float>(int);
template int gemm_nc<double>(int);
template void run_group_gemm<float>(Ctx*, const Grouped&, GemmArgs<float>);
template void run_group_gemm<double>(Ctx*, const Grouped&, GemmArgs<double>);

}  // namespace lhv
