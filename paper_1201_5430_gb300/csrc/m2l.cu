// M2L with conversion (Sec. 4.4): for every box of levels 2..L and every box of
// its interaction list (children of the parent's colleagues that are not
// colleagues: at most 189 of the 316 possible offsets),
//   local += [[T, C12 T], [0, C22 T]] multipole,   T = (S|R)(t), t = target - source
// with C12, C22 the R-basis conversion of Eq. drt10 at the same t (Eqs. mr3,
// CVL14).  In the scaled basis the fused operator depends only on the integer
// offset, so pairs of all levels are bucketed by offset and run as one grouped
// GEMM (group_gemm.cu).
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "lhv_group.cuh"
#include "lhv_internal.cuh"

namespace lhv {

namespace {

__device__ inline void key_coords(uint64_t key, int level, int& x, int& y, int& z) {
    x = y = z = 0;
    for (int k = 0; k < level; ++k) {
        x |= (int)((key >> (3 * k)) & 1ull) << k;
        y |= (int)((key >> (3 * k + 1)) & 1ull) << k;
        z |= (int)((key >> (3 * k + 2)) & 1ull) << k;
    }
}

// Offsets of the levels in the global box order, for the one launch over levels 2 .. L.
struct TableLevels {
    int L;
    int off[MAX_LEVELS + 2];
};

// ---- pair list of one truncation number: buckets by offset slot, straight from the colleagues ----
// The interaction list of a target box is the children of its parent's colleagues that are not
// its own colleagues.  Block b of nblk takes a contiguous range of the real target boxes of
// levels 2 .. L, one thread per (target, parent's colleague q); a child's offset follows from q and
// the two octants (the low three key bits), so no key is decoded.  FILL = false writes the
// block's pairs per slot to counts[slot][b]; after their exclusive scan (= the first pair of
// every (slot, block)) FILL = true writes the pairs there, ranked by a shared-memory counter.  Two
// passes over 26 colleagues a box in place of a 316-entry table row a box, written once and read
// twice, and one global atomic per pair on 316 counters: sphere surface of 2^20 at p = 12,
// 4.13 M pairs, the lists took 1.33 ms, now 0.20.
template <bool FILL>
__global__ void __launch_bounds__(256) k_m2l_pairs(TableLevels lv, const int* __restrict__ loff,
                                                   const uint64_t* __restrict__ bkey, const int* __restrict__ bparent,
                                                   const int* __restrict__ bcol, const int* __restrict__ bcbeg,
                                                   const int* __restrict__ bcend, const int* __restrict__ slot_of,
                                                   int nblk, int* __restrict__ counts, int2* __restrict__ pairs,
                                                   unsigned long long* __restrict__ total) {
    __shared__ int cnt[NUM_OFFSETS], slots[343];
    __shared__ int s_pairs;
    for (int i = threadIdx.x; i < NUM_OFFSETS; i += blockDim.x)
        cnt[i] = FILL ? counts[(int64_t)i * nblk + blockIdx.x] : 0;
    for (int i = threadIdx.x; i < 343; i += blockDim.x) slots[i] = slot_of[i];
    if (threadIdx.x == 0) s_pairs = 0;
    __syncthreads();
    const int64_t nt = loff[lv.L + 1] - loff[2];
    const int64_t b0 = nt * blockIdx.x / nblk, b1 = nt * (blockIdx.x + 1) / nblk;
    int mine = 0;
    for (int64_t it = b0 * 27 + threadIdx.x; it < b1 * 27; it += blockDim.x) {
        const int rb = loff[2] + (int)(it / 27), q = (int)(it % 27);
        if (q == 13) continue;  // the parent's own children are all colleagues
        int level = 2;
        while (level < lv.L && rb >= loff[level + 1]) ++level;
        const int o = lv.off[level], po = lv.off[level - 1];
        const int gb = o + (rb - loff[level]);
        // parent indices are relative to level - 1, child ranges relative to level
        const int pc = bcol[((int64_t)po + bparent[gb]) * 27 + q];
        if (pc < 0) continue;
        const int to = (int)(bkey[gb] & 7ull);
        const int bx = 2 * (q / 9 - 1) - (to & 1), by = 2 * (q / 3 % 3 - 1) - (to >> 1 & 1), bz = 2 * (q % 3 - 1) - (to >> 2);
        for (int s = bcbeg[po + pc]; s < bcend[po + pc]; ++s) {
            const int so = (int)(bkey[o + s] & 7ull);
            const int slot = slots[(bx + (so & 1) + 3) * 49 + (by + (so >> 1 & 1) + 3) * 7 + bz + (so >> 2) + 3];
            if (slot < 0) continue;  // a colleague of the target
            const int at = atomicAdd(&cnt[slot], 1);
            if (FILL) pairs[at] = make_int2(o + s, gb);
            ++mine;
        }
    }
    if constexpr (!FILL) {
        for (int o = 16; o > 0; o >>= 1) mine += __shfl_down_sync(0xffffffffu, mine, o);
        if ((threadIdx.x & 31) == 0 && mine) atomicAdd(&s_pairs, mine);
        __syncthreads();
        for (int i = threadIdx.x; i < NUM_OFFSETS; i += blockDim.x) counts[(int64_t)i * nblk + blockIdx.x] = cnt[i];
        if (threadIdx.x == 0 && s_pairs) atomicAdd(total, (unsigned long long)s_pairs);
    }
}

// The chunks of at most nc pairs of every slot (every block scans the slots, then takes a share of
// the chunks: 33,000 of the sphere surface took one block 22 us): first[slot * nblk] is the slot's first
// pair, *npairs the number of pairs; choff[slot] its first chunk, choff[316] their number.
__global__ void __launch_bounds__(256) k_m2l_chunks(int nblk, const int* __restrict__ first,
                                                     const int* __restrict__ npairs, int nc, int* __restrict__ choff,
                                                     int4* __restrict__ chunks) {
    __shared__ int pair0[NUM_OFFSETS + 1], chunk0[NUM_OFFSETS + 1];
    const int t = threadIdx.x;
    for (int g = t; g <= NUM_OFFSETS; g += blockDim.x) pair0[g] = g < NUM_OFFSETS ? first[(int64_t)g * nblk] : *npairs;
    __syncthreads();
    if (t < 32) {  // exclusive scan of the slots' chunk counts
        int carry = 0;
        for (int g0 = 0; g0 < NUM_OFFSETS; g0 += 32) {
            const int g = g0 + t;
            const int n = g < NUM_OFFSETS ? (pair0[g + 1] - pair0[g] + nc - 1) / nc : 0;
            int x = n;
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (t >= o) x += y;
            }
            if (g < NUM_OFFSETS) chunk0[g] = carry + x - n;
            carry += __shfl_sync(0xffffffffu, x, 31);
        }
        if (t == 0) chunk0[NUM_OFFSETS] = carry;
    }
    __syncthreads();
    if (blockIdx.x == 0)
        for (int g = t; g <= NUM_OFFSETS; g += blockDim.x) choff[g] = chunk0[g];
    for (int c = blockIdx.x * blockDim.x + t; c < chunk0[NUM_OFFSETS]; c += gridDim.x * blockDim.x) {
        int lo = 0, hi = NUM_OFFSETS - 1;  // the last slot whose first chunk is <= c
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (chunk0[mid] <= c) lo = mid; else hi = mid - 1;
        }
        const int p0 = pair0[lo] + (c - chunk0[lo]) * nc;
        chunks[c] = make_int4(lo, p0, min(nc, pair0[lo + 1] - p0), 0);
    }
}

// table[t][slot] = GLOBAL index of the source box at offset `slot`, or -1 (the
// table is cleared to -1 before).  One thread per (target box of any level 2 .. L,
// colleague q of its parent): the children of that colleague that are not
// colleagues of the target.
__global__ void k_m2l_table(int t0, TableLevels lv, const int* __restrict__ loff,
                            const uint64_t* __restrict__ bkey, const int* __restrict__ bparent,
                            const int* __restrict__ bcol, const int* __restrict__ bcbeg,
                            const int* __restrict__ bcend, const int* __restrict__ slot_of, int* __restrict__ table,
                            unsigned long long* __restrict__ pairs) {
    unsigned long long cnt = 0;
    const int64_t nt = loff[lv.L + 1] - loff[2];  // real target boxes of levels 2 .. L
    for (int64_t it = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; it < nt * 27;
         it += (int64_t)gridDim.x * blockDim.x) {
        const int rb = loff[2] + (int)(it / 27), q = (int)(it % 27);
        int level = 2;
        while (level < lv.L && rb >= loff[level + 1]) ++level;
        const int o = lv.off[level], po = lv.off[level - 1];
        const int gb = o + (rb - loff[level]);
        // parent indices are relative to level - 1, child ranges relative to level
        const int pc = bcol[((int64_t)po + bparent[gb]) * 27 + q];
        if (pc < 0) continue;
        int tx, ty, tz;
        key_coords(bkey[gb], level, tx, ty, tz);
        int* row = table + (int64_t)(gb - t0) * NUM_OFFSETS;
        for (int s = bcbeg[po + pc]; s < bcend[po + pc]; ++s) {
            int sx, sy, sz;
            key_coords(bkey[o + s], level, sx, sy, sz);
            const int dx = sx - tx, dy = sy - ty, dz = sz - tz;
            if (dx >= -1 && dx <= 1 && dy >= -1 && dy <= 1 && dz >= -1 && dz <= 1) continue;
            row[slot_of[(dx + 3) * 49 + (dy + 3) * 7 + (dz + 3)]] = o + s;
            ++cnt;
        }
    }
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, o);
    if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(pairs, cnt);
}

}  // namespace

void m2l_prepare(Ctx* c, const OpTables& ops, const TreeBufs& tb, const Levels& lv, Buf& table_buf, Grouped& gp,
                 int nc, bool uniform, unsigned long long* pair_counter) {
    cudaStream_t s = stream_of(c);
    const int L = lv.L;
    const int t0 = lv.off[2];
    const int* count = tb.counts.as<int>();
    TableLevels tl{};
    tl.L = L;
    for (int l = 0; l <= L + 1 && l <= MAX_LEVELS + 1; ++l) tl.off[l] = lv.off[l];
    const int64_t nt = lv.off[L + 1] - t0;  // target box slots of levels 2 .. L
    const int* loff = count + 32;  // the level scan's offsets of the real boxes
    if (uniform) {
        gp.ngroups = NUM_OFFSETS;
        gp.nc = nc;
        // blocks of at least 16 target boxes, two rounds of the threads (4096 elements, 832 boxes: 20 us a
        // pass with 64, 10 with 16); two per SM read and rank the pairs of a large tree
        const int nblk = (int)std::max<int64_t>(1, std::min<int64_t>(2 * 152, nt / 16));
        const int64_t ncnt = (int64_t)NUM_OFFSETS * nblk;
        ensure(c, gp.gcount, (ncnt + 1) * 4);
        ensure(c, gp.choff, (NUM_OFFSETS + 1) * 4);
        ensure(c, gp.scan_tmp, (scan_tmp_ints(ncnt) + 64) * 4);
        ensure(c, gp.pairs, nt * 189 * 8);
        ensure(c, gp.chunks, (nt * 189 / nc + NUM_OFFSETS + 1) * 16);
        ensure(c, gp.work, 64);
        int* counts = gp.gcount.as<int>();
        auto pass = [&](auto fill) {
            k_m2l_pairs<decltype(fill)::value><<<nblk, 256, 0, s>>>(
                tl, loff, tb.bkey.as<uint64_t>(), tb.bparent.as<int>(), tb.bcol.as<int>(), tb.bcbeg.as<int>(),
                tb.bcend.as<int>(), ops.slot_of.as<int>(), nblk, counts, gp.pairs.as<int2>(), pair_counter);
            count_launch(c);
        };
        pass(std::false_type{});
        exclusive_scan(c, ncnt, counts, counts, gp.scan_tmp.as<int>(), counts + ncnt);
        pass(std::true_type{});
        k_m2l_chunks<<<grid_for(nt * 64 / nc, 256, 152), 256, 0, s>>>(nblk, counts, counts + ncnt, nc, gp.choff.as<int>(), gp.chunks.as<int4>());
        count_launch(c);
        check_launch("m2l pairs");
        return;
    }
    // a truncation number per level: buckets by (level, slot) through the interaction table, whose
    // rows cover the global boxes [off[2], off[L+1])
    ensure(c, table_buf, nt * NUM_OFFSETS * 4);
    int* table = table_buf.as<int>();
    fill_level_rows<int>(c, lv, count, 2, L, NUM_OFFSETS, t0, table, -1);  // the rows of real boxes
    k_m2l_table<<<grid_for(nt * 27, 128), 128, 0, s>>>(
        t0, tl, loff, tb.bkey.as<uint64_t>(), tb.bparent.as<int>(), tb.bcol.as<int>(), tb.bcbeg.as<int>(),
        tb.bcend.as<int>(), ops.slot_of.as<int>(), table, pair_counter);
    count_launch(c);
    check_launch("m2l table");
    M2LItems it{};
    it.table = table;
    it.loff = loff;
    it.t0 = t0;
    it.L = L;
    for (int l = 0; l <= MAX_LEVELS; ++l) it.off[l] = lv.off[l];
    build_grouped(c, gp, NUM_OFFSETS * (L - 1), nt * NUM_OFFSETS, nt * 189, nc, it);
}

template <typename T>
void m2l_apply(Ctx* c, const Plan<T>& pl, const Levels& lv, const int* count, Grouped& gp, const T* mult, T* loc) {
    const int L = lv.L;
    if (pl.rcr) {  // rotation - coaxial - rotation (rcr.cu)
        rcr_apply<T>(c, *pl.rcr, gp, mult, loc, pl.ld);
        return;
    }
    // the complex form's tensor-core products read the multipoles split into TF32 hi/lo once
    // (one p at every level; the other forms split in the kernel)
    const float* mhi = nullptr;
    const float* mlo = nullptr;
    if constexpr (sizeof(T) == 4) {
        if (pl.psi && ctx_m2l_tc(c) && pl.m2l_tiles[2]) {
            const int64_t first = (int64_t)lv.off[2] * pl.ld, rows = (int64_t)(lv.off[L + 1] - lv.off[2]) * pl.ld;
            Buf& bh = ctx_tmp(c, 12);
            Buf& bl = ctx_tmp(c, 13);
            ensure(c, bh, (first + rows) * 4);
            ensure(c, bl, (first + rows) * 4);
            tc_split(c, lv, count, 2, L, pl.ld, mult, bh.as<float>(), bl.as<float>());
            mhi = bh.as<float>();
            mlo = bl.as<float>();
        }
    }
    // one launch per run of levels with the same p (one launch in all when uniform)
    for (int l0 = 2; l0 <= L;) {
        int l1 = l0 + 1;
        if (pl.uniform) l1 = L + 1;
        else
            while (l1 <= L && pl.p[l1] == pl.p[l0]) ++l1;
        const int P = pl.p[l0] * pl.p[l0];
        GemmArgs<T> a{};
        a.g0 = pl.uniform ? 0 : (l0 - 2) * NUM_OFFSETS;
        a.g1 = pl.uniform ? NUM_OFFSETS : (l1 - 2) * NUM_OFFSETS;
        a.ops = pl.m2l[l0];
        a.ops_mod = NUM_OFFSETS;
        a.R = pl.rows(P);  // scalar case: the translation block alone, no chi
        a.C = pl.rows(P);
        a.psplit = pl.split_out(P);  // the fused zero block (two-potential form only)
        a.in = mult;
        a.ldin = pl.ld;
        a.out = loc;
        a.ldout = pl.ld;
        a.mode = GEMM_ATOMIC;
        a.scale = (T)1;
        bool done = false;
        if constexpr (sizeof(T) == 4) {
            if (ctx_m2l_tc(c) && pl.m2l_tiles[l0]) {
                if (pl.psi) run_tc_gemm(c, gp, a, pl.m2l_tiles[l0], mhi, mlo, ctx_err_flag(c));
                else
                    run_tc_trans(c, TRANS_M2L, gp, a.g0, a.g1, pl.p[l0], pl.scalar, pl.m2l_tiles[l0], mult, loc, pl.ld,
                                 ctx_err_flag(c));
                done = true;
            }
        }
        if (!done) run_group_gemm<T>(c, gp, a);
        l0 = l1;
    }
}

template void m2l_apply<float>(Ctx*, const Plan<float>&, const Levels&, const int*, Grouped&, const float*, float*);
template void m2l_apply<double>(Ctx*, const Plan<double>&, const Levels&, const int*, Grouped&, const double*,
                                double*);

}  // namespace lhv
