// Chain kernel of the population annealing for windows whose rank-load rows are short enough to be
// scored from registers: "one warp per chain, one layer per lane".
//
// A chain of Algorithm 3 is a sequence of dependent rounds; what bounds a level is the latency of a
// round times the rounds of a chain, over the chains an SM keeps in flight.  The kernel shortens and
// removes rounds:
//  * Rejections without rank loads.  For any rank p of a layer, max_p (W + d) >= W[p] + d[p].  With one
//    fixed rank per layer (the busiest of the window as a whole) and f_i = sum_l q[i][l][p_l], the new
//    expert cost of the row-shard that gives sample i and takes i2 is at least F - f_i + f_i2, F the sum of
//    f over its samples (kept as the slack Esum - F).  Score and energy are monotone in it, so the lane that proposes a step can
//    reject it by itself from cell statistics, F and two scalars: 32 steps at a time, no rank load read.
//    Windows whose samples follow one routing mix have the same busiest rank nearly everywhere, and
//    then every rejection is decided this way and what is scored is accepted (large, wide, heavy, medium of
//    the named windows: all but 1e-4 of the rejections); with four routing mixes an eighth to a third
//    is.  A candidate that is not rejected by its bound is scored exactly.  The bound is worked out in single precision with an
//    allowance for its roundings: in 64-bit integers it was a third of a round's instructions (with the decision shared by two
//    lanes: heavy 89.2 -> 81.4 ms, wide 8.22 -> 8.04, medium 0.87 -> 0.84).
//  * Rows in registers.  A lane holds whole layers (layer = lane, lane + 32, ...) of the two slices and the two
//    demand rows: 16-byte loads, one trip, no shuffles, no staging; the new slices are stored from the
//    same registers.
//  * Compressed rows (COMP: rank counts of 8 and more whose full rows do not fit the registers).  A row keeps, per
//    layer, the loads of the three ranks that are busiest in the window and an upper bound of every
//    other rank's load: the sum over the samples of each one's largest count among those ranks.
//    While the bound does not exceed the three, their maximum is the layer's maximum; where it
//    does, the layer's loads are added up from the samples of the row-shard.  Used when the seed's
//    row-shards nearly all satisfy it (checked on the device, see k_member_rows): 16 bytes per layer
//    instead of 4*P: an eighth of the traffic at 32 ranks.
//  * No staging area, so 12 to 16 chains per SM instead of 5 to 10.
// What bounds it now: with 14 to 16 chains per SM (heavy) the instructions of a round, about 4900 cycles with four
// warps per scheduler; with 7 (large) their latency, about 3900 cycles; launched once for all levels (medium)
// about 2700 cycles a round and 20 us a level for the slowest chain, the barrier and the states.  A level's time before (the
// warp-per-chain kernel; medium: warp per candidate) and now: heavy 15.0 -> 3.9 ms, wide 1.2 -> 0.41 ms,
// large 0.21 -> 0.13 ms, medium 50 -> 36 us (plans: 301 -> 78, 24.0 -> 8.1 to 10.8 over windows of the kind, 4.8 -> 2.8,
// 1.12 -> 0.87 ms).
// Step for step this is the sequential chain: proposals are evaluated against the current state,
// feasible ones are decided in step order, and the speculation is redone after an acceptance.
//
// Two forms.  CHIP: the rank loads of a chain live in shared memory, every chain is resident at once
// and one launch runs all levels; a CTA holds several chains and works out the level barrier
// for itself.  Otherwise one launch per level, rank loads as slices of a pool shared copy-on-write (see AnnealArgs).
#include <algorithm>
#include <string.h>

#include "rp_level_end.cuh"
#include "rp_anneal_row.cuh"

struct ChainR {                                      // bookkeeping of the chain within this level
    i64 B[3];
    u64 dig;
    int best_step, best_nlog, nlog, n_imp;
    int has_snap, pad;
};

struct StepX {                   // what a lane keeps about the step it proposes for
    u32 flags, bz;
    u64 thr;
    float thrf;                  // thr / 2^32, rounded up; infinite where every rise is accepted
    int i[4];                    // samples; for a relocation i[2], i[3] are target cells
    int c[4];                    // cell of sample i[x] (i[2], i[3] themselves for a relocation)
    int t[4], f[4];              // length of sample i[x] and its demand on the fixed ranks (0 for relocation targets)
};

__device__ __forceinline__ int4 sub4(const int4 &a, const int4 &b) { return make_int4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w); }
__device__ __forceinline__ int4 add4(const int4 &a, const int4 &b) { return make_int4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }

// Busiest loads of the layers in `who` (bit x: layer x + first) of row-shard rg once sample mi has left it
// (sgn = -1) or joined it (+1) and mi2 (>= 0: a swap) the other way round, added up from the samples that sit
// there; lane x receives layer x + first, the other lanes keep `mine`.  The samples are first collected in `list`
// (its last entry is the counter), then sixteen of their counts are in flight at a time, a rank per lane: nearly always a
// single layer is asked for, of a row-shard of a hundred short samples.  Kept small: a form with the collection
// unrolled took 110000 cycles a call on wide and slowed the other chains of the SM threefold (instruction fetches).
#define ROW_LIST 256
__device__ __noinline__ int rp_row_exact_max(int N, int P, int LP, const int *__restrict__ q, const unsigned short *cells,
                                             const unsigned short *rg_of, int *list, int rg, unsigned who, int first, int mi, int mi2,
                                             int sgn, int mine)
{
    const int lane = threadIdx.x & 31;
    int *count = list + ROW_LIST;
#pragma unroll 1
    for (; who; who &= who - 1) {
        const int at = __ffs(who) - 1;
        const int *layer = q + (size_t)(at + first) * P;
        int best = 0;
#pragma unroll 1
        for (int p0 = 0; p0 < P; p0 += 32) {
            const bool on = p0 + lane < P;
            const int *col = layer + (on ? p0 + lane : 0);
            int acc = sgn * __ldg(col + (size_t)mi * LP), seg = (N + 3) & ~3;
            if (mi2 >= 0) acc -= sgn * __ldg(col + (size_t)mi2 * LP);
#pragma unroll 1
            for (int b = 0; b < N; b += seg) {
                __syncwarp();
                if (lane == 0) *count = 0;
                __syncwarp();
                const int e = min(b + seg, N);
#pragma unroll 8
                for (int i = b + 4 * lane; i < e; i += 128) {
                    const uint2 v = __ldcg((const uint2 *)(cells + i));            // (the blob is padded to 16 bytes)
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        const unsigned c = ((h & 2 ? v.y : v.x) >> (16 * (h & 1))) & 0xffffu;
                        if (i + h < e && (int)rg_of[c] == rg) { const int x = atomicAdd(count, 1); if (x < ROW_LIST) list[x] = i + h; }
                    }
                }
                __syncwarp();
                const int n = *count;
                if (n > ROW_LIST) { seg = ROW_LIST; b = -seg; continue; }          // too many at once: again, a piece at a time
#pragma unroll 1
                for (int x0 = 0; x0 < n; x0 += 16) {
                    int v[16];
#pragma unroll
                    for (int x = 0; x < 16; ++x) v[x] = x0 + x < n ? __ldg(col + (size_t)list[x0 + x] * LP) : 0;
#pragma unroll
                    for (int x = 0; x < 16; ++x) acc += v[x];
                }
            }
            best = max(best, (int)__reduce_max_sync(0xffffffffu, on ? acc : 0));
        }
        if (lane == at) mine = best;
    }
    return mine;
}

// Shared memory of the chains of a CTA.
struct RowChain {
    u64 *Q;
    i64 *Esum, *Afx, *Jfx, *U, *Sc, *slack;
    int *T, *cnt;
    ChainR *book;
    int *wtab, *spare;           // !CHIP: slice of each row-shard, and its spare
    unsigned short *cell, *snap; // CHIP: assignment, trajectory-best layout, rank loads
    int4 *W;
    i64 *att, *top1, *top2;      // shards of several slots: attention key of a cell; largest and second largest stage cost
    unsigned short *topc;        // of each (row-shard, stage), and the cell of the largest
    char *base;
};

__device__ __forceinline__ RowChain row_chain(const AnnealArgs &A, const RowArgs &X, char *sm_chain, int w)
{
    RowChain c;
    char *sm = sm_chain + (size_t)w * X.chain_bytes;
    c.base = sm;
    c.Q = (u64 *)(sm + A.bl.off_Q);
    c.Esum = (i64 *)(sm + A.bl.off_Esum);
    c.Afx = (i64 *)(sm + A.bl.off_Afx);
    c.Jfx = (i64 *)(sm + A.bl.off_Jfx);
    c.U = (i64 *)(sm + A.bl.off_U);
    c.Sc = (i64 *)(sm + A.bl.off_S);                                     // S0, S1, S2, energy
    c.T = (int *)(sm + A.bl.off_T);
    c.cnt = (int *)(sm + A.bl.off_cnt);
    c.slack = (i64 *)(sm + X.off_F);
    c.book = (ChainR *)(sm + X.off_book);
    c.wtab = (int *)(sm + X.off_wtab);
    c.spare = (int *)(sm + X.off_spare);
    c.cell = (unsigned short *)(sm + X.off_cell);
    c.snap = (unsigned short *)(sm + X.off_snap);
    c.W = (int4 *)(sm + X.off_W);
    c.att = (i64 *)(sm + X.off_top);
    c.top1 = c.att + A.dm.K;
    c.top2 = c.top1 + (size_t)A.dm.RG * A.dm.S;
    c.topc = (unsigned short *)(c.top2 + (size_t)A.dm.RG * A.dm.S);
    return c;
}

// Largest and second largest cost of stage s over the slots of row-shard (row of cell `rb`, shard g).
__device__ __forceinline__ void row_top_stage(const RpDims &dm, const RowChain &ch, const int *dpl, const int *dpo, int rb, int g, int rg, int s)
{
    const i64 ca = dm.ahat[s] * dm.C, cb = dm.bhat[s];
    i64 v1 = -1, v2 = 0;
    int c1 = 0;
    for (int x = dpo[g]; x < dpo[g + 1]; ++x) {
        const int c = rb + dpl[x];
        const i64 v = ca * ch.T[c] + cb * (i64)ch.Q[c];
        if (v > v1) { v2 = v1 < 0 ? 0 : v1; v1 = v; c1 = c; }
        else if (v > v2) v2 = v;
    }
    ch.top1[rg * dm.S + s] = v1; ch.top2[rg * dm.S + s] = v2; ch.topc[rg * dm.S + s] = (unsigned short)c1;
}

__device__ __forceinline__ i64 row_energy(i64 s0, i64 s1, i64 s2)       // rp_energy of non-negative scores
{
    return s0 + (i64)((u64)s1 / 1000000ull) + (i64)((u64)s2 / 1000000000ull);
}

// Resident chains the register budget is set for.  Heavy (one chunk per lane) at 12 / 14 / 16 / 19 / 24 chains: 96 / 87.5 /
// 90 / 100 / 112 ms a plan (spills from 19 on); wide (two) at 12 / 14 / 16 / 19: 10.8 / 11.9 / 11.9 / 16.0 ms; four chunks need the
// registers of 12.
#define ROW_CHAINS_PER_SM(LPL, CPL) ((LPL) * (CPL) == 1 ? 14 : 12)

// The level barrier of up to 32 members by one warp, a member a lane: incumbent (inc, *win = its slot or -1), then, unless this
// was the last level, ancestors of members m0 .. m1-1.  No CTA-wide barrier between its parts (tiny 333 -> 308 us a plan); with
// eight members a lane one warp takes longer than eight do with their barriers (medium 913 -> 978 us).
__device__ __forceinline__ void row_barrier_warp(const AnnealArgs &A, int P, const u64 *eL, const i64 *bestL, bool last, u64 cq, u32 resample_x,
                                                 int m0, int m1, i64 *inc, int *win, int *anc, int lane)
{
    const u64 r = lane < P ? __ldcg(eL + lane) : 0x7fffffffffffffffull;
    const i64 e[1] = { (i64)(r & ~(1ull << 63)) };
    i64 b0 = inc[0], b1 = inc[1], b2 = inc[2];
    int bj = 0x7fffffff;
    if (r >> 63) {                               // its trajectory best beats the incumbent
        b0 = __ldcg(bestL + 3 * lane); b1 = __ldcg(bestL + 3 * lane + 1); b2 = __ldcg(bestL + 3 * lane + 2);
        bj = lane;
    }
    const u32 hi = (u32)((u64)e[0] >> 32), mh = __reduce_min_sync(0xffffffffu, hi);
    const i64 emin = (i64)(((u64)mh << 32) | __reduce_min_sync(0xffffffffu, hi == mh ? (u32)e[0] : 0xffffffffu));
    int slot = -1;
    if (__any_sync(0xffffffffu, bj != 0x7fffffff)) {
        slot = le_lexmin_lane(b0, b1, b2, bj);
        if (lane == slot) { inc[0] = b0; inc[1] = b1; inc[2] = b2; }
    }
    if (lane == 0) *win = slot;                  // that chain stored its trajectory-best layout in its row of cand_layout
    if (last) return;
    const u64 M = (u64)(emin > A.dm.SC ? emin : A.dm.SC);
    u64 w[1];
    le_weights<1>(e, emin, M, cq, w);
    u64 F = lane < P ? w[0] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const u64 x = __shfl_up_sync(0xffffffffu, F, o); if (lane >= o) F += x; }
    const u64 Ftot = __shfl_sync(0xffffffffu, F, 31), u0 = (u64)(((unsigned __int128)resample_x * Ftot) >> 32);
    for (int m = m0; m < m1; ++m) {
        // slots with P * F <= at (those past the last member hold the total: never)
        const unsigned __int128 at = (unsigned __int128)u0 + (unsigned __int128)m * Ftot;
        const int n = __popc(__ballot_sync(0xffffffffu, (unsigned __int128)P * F <= at));
        if (lane == 0) anc[m] = n;
    }
}

// LPL layers per lane, CPL 16-byte chunks per layer (X.cpl <= CPL of them in use).
template <int LPL, int CPL, bool CHIP, bool COMP>
__global__ void __launch_bounds__(CHIP ? ROW_THREADS : 32, CHIP ? 1 : ROW_CHAINS_PER_SM(LPL, CPL))
k_anneal_row(const AnnealArgs A, const RowArgs X)
{
    constexpr int NCH = LPL * CPL;
    const RpDims &dm = A.dm;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int NT = CHIP ? ROW_THREADS : 32;
    const int cw = CHIP ? X.cw : 1;                                      // chains of this CTA: warps 0 .. cw-1; the others
    const int j = CHIP ? blockIdx.x * cw + warp : blockIdx.x;            // (CHIP) help to move states and at the level barrier
    const int P = A.Ppop;
    const bool live = !CHIP || (warp < cw && j < P);
    char *sm_cta = (char *)smraw;                                        // tables shared by the CTA's chains
    char *sm_chain = (char *)smraw + X.off_chain;
    const RowChain ch = row_chain(A, X, sm_chain, CHIP ? min(warp, cw - 1) : 0);
    const int *dpl = (const int *)(sm_cta + A.sl.off_dpl);
    const int *dpo = (const int *)(sm_cta + A.sl.off_dpo);
    const char *sm_tab = sm_cta + X.off_tab - A.sl.off_rg;
    const unsigned short *rg_of = (const unsigned short *)(sm_tab + A.sl.off_rg);
    const unsigned short *g_of = (const unsigned short *)(sm_tab + A.sl.off_g);
    const unsigned short *rowbase = (const unsigned short *)(sm_tab + A.sl.off_row);
    RpSmemState st = { nullptr, ch.T, ch.Q, ch.cnt, ch.Esum, ch.Afx, ch.U };

    if (!CHIP && __ldcg(&A.status[RP_SW_TIMEOUT])) return;               // the call has failed already: nothing to do
    const int L = dm.L, cpl = CPL == 1 ? 1 : X.cpl, rc = L * cpl;        // 16-byte chunks per layer and per row
    const int rot = (CPL > 1 && (cpl & (cpl - 1)) == 0) ? cpl - 1 : 0;   // lanes start at different chunks: fewer bank conflicts
    const bool ident = dm.own_shard;
    const bool sum32 = dm.sum32;
    const i64 aC = dm.asum * dm.C, bS = dm.bsum;
    const float aCf = (float)aC, bSf = (float)bS, ECf = (float)dm.EC;
    const int4 *qr = (const int4 *)X.qr;
    unsigned short *cells = CHIP ? ch.cell : (unsigned short *)(A.blob_dst + (size_t)j * A.bl.bytes + A.bl.off_cell);
    const int nh16 = (A.bl.off_cell + 15) >> 4, nhw = A.bl.off_cell >> 2;     // the blob's arrays before the assignment
    const int n4 = dm.N >> 2;
    const StepRec *recs = (const StepRec *)(ch.base + X.off_recs);

    // ---- prologue: the static tables and the ancestor's terminal state ---------------------------
    {
        const int nd = A.sl.off_t >> 2, nc = (A.sl.bytes - A.sl.off_rg) >> 2;
        for (int x = tid; x < nd; x += NT) ((int *)sm_cta)[x] = __ldg((const int *)A.static_blk + x);
        for (int x = tid; x < nc; x += NT) ((int *)(sm_cta + X.off_tab))[x] = __ldg((const int *)(A.static_blk + A.sl.off_rg) + x);
    }
    int half_w = 0, inc_slot = -1;
    __shared__ i64 inc_s[3];
    __shared__ int failed_s;
    for (int w = 0; w < cw; ++w) {
        const int jj = CHIP ? blockIdx.x * cw + w : j;
        if (CHIP && jj >= P) break;
        const RowChain c = CHIP ? row_chain(A, X, sm_chain, w) : ch;
        const int src = min(max(A.anc[jj], 0), P - 1);
        const char *bsrc = A.blob_src + (size_t)src * A.bl.bytes;
        const int4 *hs = (const int4 *)bsrc;
#pragma unroll 8
        for (int x = tid; x < nh16; x += NT) ((int4 *)c.base)[x] = __ldg(hs + x);
        const i64 *fs = X.F_src + (size_t)src * dm.RG;
#pragma unroll 4
        for (int rg = tid; rg < dm.RG; rg += NT) c.slack[rg] = __ldg(fs + rg);
        const unsigned short *cs = (const unsigned short *)(bsrc + A.bl.off_cell);        // 8-byte aligned
        unsigned short *cd = CHIP ? c.cell : cells;
#pragma unroll 8
        for (int x = tid; x < n4; x += NT) ((uint2 *)cd)[x] = __ldg((const uint2 *)cs + x);
        for (int i = (n4 << 2) + tid; i < dm.N; i += NT) cd[i] = __ldg(cs + i);
        if (!CHIP) {
            const int *ts = (const int *)(bsrc + A.bl.off_wtab);
            // A slice that only this member holds when the level starts is rewritten in place; a shared
            // one is left at its first rewrite for this chain's spare slice of that row-shard (entry
            // j*RG + rg of the free list, which holds at least RG slices per member).
            const int n_free = A.wfree_head[1];
#pragma unroll 4
            for (int rg = lane; rg < dm.RG; rg += 32) {
                const int s = __ldg(ts + rg);
                const size_t at = (size_t)j * dm.RG + rg;
                const int sp = at < (size_t)n_free ? __ldg(&A.wfree[at]) : -2;
                c.wtab[rg] = s;
                c.spare[rg] = __ldg(&A.wref[s]) == 1 ? -1 : sp;
            }
        } else {
            // rank loads of the ancestor: its slices, or its cell of the pool
            half_w = A.wloc_dst[jj] >= P ? 1 : 0;
            const int cell = A.slices ? 0 : rp_src_cell(A, src, jj);
            const int *ts = (const int *)(bsrc + (A.slices ? A.bl.off_wtab : 0));
            for (int rg = warp; rg < dm.RG; rg += NT / 32) {
                const size_t s = A.slices ? (size_t)__ldg(ts + rg) : (size_t)cell * dm.RG + rg;
                const int4 *ws = (const int4 *)(X.Wr + s * X.rlp);
#pragma unroll 4
                for (int x = lane; x < rc; x += 32) c.W[(size_t)rg * rc + x] = __ldg(ws + x);
            }
            if (tid == 0) atomicAdd((u64 *)&A.counters[src == jj ? 6 : 5], (u64)2 * dm.RG * dm.LP * 4);
        }
    }
    if (CHIP) {
        if (tid < 3) inc_s[tid] = A.lo.inc_score[tid];
        __syncthreads();
        // every chain of the launch has read its start state (the pool is about to be written) from here on
        if (tid == 0) { __threadfence(); atomicAdd(A.lo.done, 1); }
        if (A.stall_test && blockIdx.x == 0) {       // inspection hook: chain 0 waits for an arrival that never comes
            if (tid == 0 && !rp_wait_count(A.lo.done, 0x7fffffff, A)) atomicExch(&A.status[RP_SW_TIMEOUT], 1);
            return;
        }
    } else if (A.stall_test && j == 0) {
        // inspection hook: a bounded wait on a barrier phase that nothing completes
        u64 *mbar = (u64 *)(ch.base + X.off_book + ((sizeof(ChainR) + 7) & ~(size_t)7));
        if (lane == 0) rp_mbar_init(mbar, 1);
        __syncwarp();
        if (!rp_mbar_wait(mbar, 0, A.wait_polls)) {
            if (lane == 0) atomicExch(&A.status[RP_SW_TIMEOUT], 1);
            return;
        }
    }
    __syncwarp();

    const int n_levels = CHIP ? A.n_levels : 1;
    // CHIP: the step records of a level depend on nothing but the schedule: the warps without a chain work out those of
    // the next level (its first X.recs steps) while the chains run.
    auto make_recs = [&](int ln, int w0, int nw) {
        for (int x = (warp - w0) * 32 + lane; x < cw * X.recs; x += nw * 32) {
            const int w = x / X.recs, k = x - w * X.recs;
            ((StepRec *)(sm_chain + (size_t)w * X.chain_bytes + X.off_recs))[(ln & 1) * X.recs + k] =
                rp_make_step_rec(A, ln, A.levels[ln].tau, (u32)k, (u32)(blockIdx.x * cw + w));
        }
    };
    if (CHIP) { make_recs(0, 0, NT / 32); __syncthreads(); }
    int moved = 0;                                                   // states this thread's chain took over
    i64 sum_feas = 0, sum_acc = 0, sum_imp = 0, sum_rows = 0;       // CHIP: of all levels so far
    for (int ln = 0; ln < n_levels; ++ln) {
    const int level = CHIP ? ln : A.level;
    const u64 tau = CHIP ? A.levels[ln].tau : A.tau;
    const bool last = CHIP ? (ln == n_levels - 1) : (A.last != 0);
    int n_feas = 0, n_acc = 0;                  // feasible moves this lane proposed; accepted ones (the same in every lane)
    i64 n_rows = 0;                             // rows and slices they name, likewise per lane
    if (live) {
        if (!ident) {
            for (int c = lane; c < dm.K; c += 32) ch.att[c] = aC * ch.T[c] + bS * (i64)ch.Q[c];
            for (int x = lane; x < dm.RG * dm.S; x += 32) {
                const int rg = x / dm.S;
                row_top_stage(dm, ch, dpl, dpo, rg / dm.G * dm.D, rg % dm.G, rg, x % dm.S);
            }
        }
        if (lane == 0) {
            ch.book->B[0] = ch.Sc[0]; ch.book->B[1] = ch.Sc[1]; ch.book->B[2] = ch.Sc[2];
            ch.book->dig = 0; ch.book->best_step = 0; ch.book->best_nlog = 0; ch.book->nlog = 0; ch.book->n_imp = 0;
            ch.book->has_snap = 0;
        }
        __syncwarp();
        for (int kb = 0; kb < A.steps; kb += SPEC) {
            const int nb = min(SPEC, A.steps - kb);
            // ---- the next 32 steps, one per lane: random words, candidate cells, lengths, fixed-rank demands ----
            StepX sr;
            sr.flags = 0; sr.bz = 0; sr.thr = 0; sr.thrf = 0.f;
#pragma unroll
            for (int x = 0; x < 4; ++x) { sr.i[x] = -1; sr.c[x] = 0; sr.t[x] = 0; sr.f[x] = 0; }
            if (lane < nb) {
                const StepRec r = (CHIP && kb + lane < X.recs) ? recs[(ln & 1) * X.recs + kb + lane] : rp_make_step_rec(A, level, tau, (u32)(kb + lane), (u32)j);
                const bool rl = r.flags & 1u;
                sr.flags = r.flags; sr.bz = r.bz; sr.thr = r.thr;
                sr.thrf = r.flags & 4u ? __int_as_float(0x7f800000) : (float)r.thr * (0x1p-32f * (1.f + 0x1p-20f));
                sr.i[0] = r.i0; sr.i[1] = r.i1; sr.i[2] = r.i2; sr.i[3] = r.i3;
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    if (x >= 2 && rl) { sr.c[x] = sr.i[x]; continue; }
                    sr.c[x] = CHIP ? (int)cells[sr.i[x]] : (int)__ldcg(cells + sr.i[x]);
                    const int2 v = __ldg(X.tf + sr.i[x]);
                    sr.t[x] = v.x; sr.f[x] = v.y;
                }
            }
            int pos = 0;
            while (pos < nb) {
                // ---- proposals of steps kb+pos .. kb+nb-1 against the current state, one per lane: GuidedProposal and
                // feasibility (the rule of rp_propose), then the rejection by the fixed ranks ----------------------------
                bool ok = false, pass = false;
                int mi = 0, mi2 = -1, c1 = 0, c2 = 0, rg1 = 0, rg2 = 0, ti = 0, t2 = 0, df = 0;
                i64 dA1 = 0, dA2 = 0;                // (shards of several slots)
                if (lane >= pos && lane < nb) {
                    const bool reloc = sr.flags & 1u;
                    const int ca = sr.c[0], cb = sr.c[1], xa = sr.c[2], xb = sr.c[3];
                    bool src_b, dst_b;
                    {
                        const int ra = ident ? ca : rg_of[ca], rb = ident ? cb : rg_of[cb], rx = ident ? xa : rg_of[xa], ry = ident ? xb : rg_of[xb];
                        const u64 Ja = (u64)ch.Jfx[ra], Aa = (u64)ch.Afx[ra];
                        // bz * Ja < Aa * 2^32  <=>  floor(bz * Ja / 2^32) < Aa
                        const u64 pr = (Ja >> 32) * sr.bz + (((Ja & 0xffffffffull) * sr.bz) >> 32);
                        const bool by_a = pr < Aa, by_cell = ident || by_a;
                        const i64 *key = by_a ? (ident ? ch.Afx : ch.att) : ch.Jfx;
                        src_b = key[by_cell ? cb : rb] > key[by_cell ? ca : ra];
                        dst_b = key[by_cell ? xb : ry] < key[by_cell ? xa : rx];
                    }
                    mi = src_b ? sr.i[1] : sr.i[0];
                    c1 = src_b ? cb : ca;
                    c2 = dst_b ? xb : xa;
                    mi2 = reloc ? -1 : (dst_b ? sr.i[3] : sr.i[2]);
                    ti = src_b ? sr.t[1] : sr.t[0];
                    t2 = dst_b ? sr.t[3] : sr.t[2];
                    df = (src_b ? sr.f[1] : sr.f[0]) - (dst_b ? sr.f[3] : sr.f[2]);
                    // (everything the score needs is loaded before feasibility is known)
                    rg1 = ident ? c1 : rg_of[c1]; rg2 = ident ? c2 : rg_of[c2];
                    const int g1 = g_of[c1], g2 = g_of[c2];
                    const int T1 = ch.T[c1], T2 = ch.T[c2], n1 = ch.cnt[c1];
                    const i64 S0 = ch.Sc[0], Ecur = ch.Sc[3], k1 = ch.slack[rg1], k2 = ch.slack[rg2], U1o = ch.U[g1], U2o = ch.U[g2];
                    ok = c1 != c2 && T2 - t2 + ti <= dm.C && (reloc ? n1 > 1 : T1 - ti + t2 <= dm.C);
                    const bool tw = ident || rg1 != rg2;
                    if (!ident && ok) {
                        const int Ta = T1 - ti + t2, Tb = T2 + ti - t2;
                        const i64 dq = (i64)t2 * t2 - (i64)ti * ti, Qa = (i64)ch.Q[c1] + dq, Qb = (i64)ch.Q[c2] - dq;
                        i64 A1 = 0, A2 = 0;
                        if (tw) {
                            for (int s = 0; s < dm.S; ++s) {
                                const i64 ca_ = dm.ahat[s] * dm.C, cb_ = dm.bhat[s];
                                const i64 va = ca_ * Ta + cb_ * Qa, vb = ca_ * Tb + cb_ * Qb;
                                const int x1 = rg1 * dm.S + s, x2 = rg2 * dm.S + s;
                                const i64 o1 = ch.topc[x1] == c1 ? ch.top2[x1] : ch.top1[x1], o2 = ch.topc[x2] == c2 ? ch.top2[x2] : ch.top1[x2];
                                A1 += va > o1 ? va : o1; A2 += vb > o2 ? vb : o2;
                            }
                            dA2 = A2 - ch.Afx[rg2];
                        } else A1 = rp_attention(dm, st, dpl, dpo, rowbase[c1] / dm.D, g1, c1, Ta, Qa, c2, Tb, Qb);
                        dA1 = A1 - ch.Afx[rg1];
                    }
                    // Rejected for certain?  The busiest loads fall by at most what the samples put on the fixed ranks plus the
                    // slack (both cells in one row-shard: nothing changes), so x below is the least by which the largest shard
                    // cost can rise and x + 1e-6 * (J1 + J2) - 1e-9 * S2 (S2 <= S0 <= E) the least by which the energy can.  In single
                    // precision, of differences only: a dozen roundings of 2^-24 of the magnitudes in `mag`, allowed for by
                    // 2^-20 of them; what is not rejected here is decided by the exact score.
                    const float k1f = sum32 ? (float)(int)k1 : (float)k1, k2f = sum32 ? (float)(int)k2 : (float)k2, dff = (float)df;
                    const float a1 = ident ? (aCf + bSf * (float)(t2 + ti)) * (float)(t2 - ti) : (float)dA1, a2 = ident ? -a1 : (float)dA2;
                    const float v1 = (float)(U1o - S0), v2 = (float)(U2o - S0), Mf = (float)(Ecur > dm.SC ? Ecur : dm.SC);
                    const float J1 = a1 + (tw ? ECf * (-dff - k1f) : 0.f), J2 = tw ? a2 + ECf * (dff - k2f) : 0.f;
                    const float u1 = v1 + J1 + (g1 == g2 ? J2 : 0.f), u2 = g1 == g2 ? u1 : v2 + J2, x = fmaxf(u1, u2);
                    const float mag = fabsf(v1) + fabsf(v2) + fabsf(a1) + fabsf(a2) + ECf * (2.f * fabsf(dff) + k1f + k2f);
                    const float err = 8.f + 0x1p-20f * mag;
                    const float most = sr.thrf * Mf + 2.f;                   // accepted below (rounded up, see thrf)
                    pass = ok && !(x > err && x + 1e-6f * (J1 + J2) - 1.001e-9f * Mf - err >= most);
                }
                unsigned pmask = __ballot_sync(0xffffffffu, pass);
                int win = -1;                                   // step accepted
                while (pmask) {
                    // ---- exact score of the next candidate -------------------------------------------------------
                    const int ls = __ffs(pmask) - 1;
                    pmask &= pmask - 1;
                    const int wi = __shfl_sync(0xffffffffu, mi, ls), wi2 = __shfl_sync(0xffffffffu, mi2, ls);
                    const unsigned rr = __shfl_sync(0xffffffffu, (unsigned)rg1 | ((unsigned)rg2 << 16), ls);
                    const int r1 = (int)(rr & 0xffffu), r2 = (int)(rr >> 16);
                    const bool touchW = r1 != r2, swap = wi2 >= 0;
                    // What the decision needs: even lanes look at the cell that gives (1), odd lanes at the one that takes (2).  Ahead
                    // of the rows its latency hides behind theirs; with one compressed chunk per lane, the form with the most chains
                    // per SM, the registers count (heavy: 80.3 ms behind the rows, 88.2 ahead; one lane for both sides 84.2 to 86.5).
                    const bool second = lane & 1;
                    int d1, d2, wti, wt2, mc, mr, mg;
                    i64 S0, S1, S2, Ecur, Jo, Uo, eo, wb, dA;
                    auto look = [&]() {
                        const unsigned dd = __shfl_sync(0xffffffffu, (unsigned)c1 | ((unsigned)c2 << 16), ls);
                        d1 = (int)(dd & 0xffffu); d2 = (int)(dd >> 16);
                        wti = __shfl_sync(0xffffffffu, ti, ls); wt2 = __shfl_sync(0xffffffffu, t2, ls);
                        mc = second ? d2 : d1; mr = second ? r2 : r1; mg = g_of[mc];
                        S0 = ch.Sc[0]; S1 = ch.Sc[1]; S2 = ch.Sc[2]; Ecur = ch.Sc[3];
                        Jo = ch.Jfx[mr]; Uo = ch.U[mg]; eo = ch.Esum[mr];
                        // accepted when the energy rises by less than wb (at least 1: never uphill by 0)
                        const u64 thr = __shfl_sync(0xffffffffu, sr.thr, ls), M = (u64)(Ecur > dm.SC ? Ecur : dm.SC);
                        const u64 bh = __umul64hi(thr, M), bl = thr * M;
                        wb = (i64)((bh << 32) | (bl >> 32));
                        wb = wb > 1 ? wb : 1;
                        if ((__shfl_sync(0xffffffffu, sr.flags, ls) & 4u) || (bh >> 31)) wb = 0x7fffffffffffffffll;
                        if (ident) { dA = (aC + bS * (wt2 + wti)) * (wt2 - wti); if (second) dA = -dA; }
                        else { const i64 da1 = __shfl_sync(0xffffffffu, dA1, ls), da2 = __shfl_sync(0xffffffffu, dA2, ls); dA = second && touchW ? da2 : da1; }
                    };
                    if (!(COMP && LPL == 1)) look();
                    int4 d[NCH], w1[NCH], w2[NCH];
                    i64 E1 = 0, E2 = 0;
                    if (touchW) {
                        int4 q2[NCH];
                        const int4 *qi = qr + (size_t)wi * rc, *qj = qr + (size_t)(swap ? wi2 : wi) * rc;
                        const int4 *W1 = CHIP ? ch.W + (size_t)r1 * rc : (const int4 *)(X.Wr + (size_t)ch.wtab[r1] * X.rlp);
                        const int4 *W2 = CHIP ? ch.W + (size_t)r2 * rc : (const int4 *)(X.Wr + (size_t)ch.wtab[r2] * X.rlp);
#pragma unroll
                        for (int y = 0; y < LPL; ++y)
#pragma unroll
                            for (int k = 0; k < CPL; ++k) {
                                const int u = y * CPL + k, ly = lane + 32 * y;
                                d[u] = q2[u] = w1[u] = w2[u] = make_int4(0, 0, 0, 0);
                                if (ly < L && (CPL == 1 || k < cpl)) {
                                    const int c = ly * cpl + (rot ? ((k + lane) & rot) : k);
                                    d[u] = __ldg(qi + c);
                                    if (swap) q2[u] = __ldg(qj + c);
                                    w1[u] = W1[c]; w2[u] = W2[c];
                                }
                            }
                        unsigned over = 0;                      // COMP: layers of this lane whose other ranks may be the busiest
                        int mx[LPL][2];
#pragma unroll
                        for (int y = 0; y < LPL; ++y) {
                            int m1 = 0, m2 = 0;
#pragma unroll
                            for (int k = 0; k < CPL; ++k) {
                                const int u = y * CPL + k;
                                d[u] = sub4(d[u], q2[u]);
                                const int4 a = w1[u] = sub4(w1[u], d[u]), b = w2[u] = add4(w2[u], d[u]);
                                if (COMP) {
                                    m1 = max(max(a.x, a.y), a.z); m2 = max(max(b.x, b.y), b.z);
                                    over |= (a.w > m1 ? 1u : 0u) << (2 * y);
                                    over |= (b.w > m2 ? 2u : 0u) << (2 * y);
                                } else { m1 = max(m1, max4(a)); m2 = max(m2, max4(b)); }
                            }
                            mx[y][0] = m1; mx[y][1] = m2;
                        }
                        if (COMP && __any_sync(0xffffffffu, over != 0)) {
#pragma unroll
                            for (int y = 0; y < LPL; ++y)
#pragma unroll
                                for (int s = 0; s < 2; ++s) {
                                    const unsigned who = __ballot_sync(0xffffffffu, (over >> (2 * y + s)) & 1u);
                                    if (who) mx[y][s] = rp_row_exact_max(dm.N, dm.P, dm.LP, A.q, cells, rg_of, (int *)(ch.base + X.off_list), s ? r2 : r1, who, 32 * y, wi, wi2, s ? 1 : -1, mx[y][s]);
                                }
                        }
                        if (sum32) {
                            int p1 = 0, p2 = 0;
#pragma unroll
                            for (int y = 0; y < LPL; ++y) { p1 += mx[y][0]; p2 += mx[y][1]; }
                            E1 = (i64)__reduce_add_sync(0xffffffffu, (unsigned)p1);
                            E2 = (i64)__reduce_add_sync(0xffffffffu, (unsigned)p2);
                        } else {
#pragma unroll
                            for (int y = 0; y < LPL; ++y) { E1 += mx[y][0]; E2 += mx[y][1]; }
                            E1 = warp_sum_i64(E1);
                            E2 = warp_sum_i64(E2);
                        }
                    }
                    // ---- exact new score and the Metropolis decision: all lanes come to the same result (both cells in one
                    // row-shard: both kinds of lanes see all of the change) --------------------------------------------
                    if (COMP && LPL == 1) look();
                    const i64 Em = second ? E2 : E1;
                    const i64 dJ = dA + (touchW ? dm.EC * (Em - eo) : 0), dJo = touchW ? __shfl_xor_sync(0xffffffffu, dJ, 1) : 0;
                    const int og = __shfl_xor_sync(0xffffffffu, mg, 1);
                    const i64 Jn = Jo + dJ, Un = Uo + dJ + (mg == og ? dJo : 0), Jx = __shfl_xor_sync(0xffffffffu, Jn, 1), Ux = __shfl_xor_sync(0xffffffffu, Un, 1);
                    const i64 n1 = S1 + dJ + dJo;
                    i64 n0 = Un > Ux ? Un : Ux, n2 = Jn > Jx ? Jn : Jx;
                    // where the previous maximum sat on a changed entry and fell, the maximum is searched anew, if the candidate is
                    // not rejected with the smaller one already
                    const bool fb0 = __any_sync(0xffffffffu, Uo >= S0) && n0 < S0, fb2 = __any_sync(0xffffffffu, Jo >= S2) && n2 < S2;
                    if (!fb0 && n0 < S0) n0 = S0;
                    if (!fb2 && n2 < S2) n2 = S2;
                    i64 en = row_energy(n0, n1, n2);
                    bool acc = rp_lex_less(n0, n1, n2, S0, S1, S2) || en - Ecur < wb;
                    if (acc && (fb0 || fb2)) {
                        i64 v0 = 0, v2 = 0;
                        if (fb0) {
                            const int ga = __shfl_sync(0xffffffffu, mg, 0), gb = __shfl_sync(0xffffffffu, mg, 1);
                            for (int g = lane; g < dm.G; g += 32) if (g != ga && g != gb) { const i64 v = ch.U[g]; if (v > v0) v0 = v; }
                            v0 = warp_max_nonneg_i64(v0);
                        }
                        if (fb2) {
                            for (int rg = lane; rg < dm.RG; rg += 32) if (rg != r1 && rg != r2) { const i64 v = ch.Jfx[rg]; if (v > v2) v2 = v; }
                            v2 = warp_max_nonneg_i64(v2);
                        }
                        if (v0 > n0) n0 = v0;
                        if (v2 > n2) n2 = v2;
                        en = row_energy(n0, n1, n2);
                        acc = rp_lex_less(n0, n1, n2, S0, S1, S2) || en - Ecur < wb;
                    }
                    if (!acc) continue;
                    // ---- commit -----------------------------------------------------------------------------------
                    win = ls;
                    n_acc += 1;
                    if (touchW) {
                        int o1 = 0, o2 = 0;
                        if (!CHIP) {
                            // Where the two rewritten slices go: in place when the slice is this chain's
                            // own, else to the spare slice of that row-shard, which then is its own.
                            const int p1 = ch.spare[r1], p2 = ch.spare[r2];
                            o1 = p1 >= 0 ? p1 : ch.wtab[r1]; o2 = p2 >= 0 ? p2 : ch.wtab[r2];
                            __syncwarp();
                            if (lane == 0) {
                                ch.wtab[r1] = o1; ch.spare[r1] = -1; ch.wtab[r2] = o2; ch.spare[r2] = -1;
                                if (p1 == -2 || p2 == -2) atomicExch(&A.status[RP_SW_POOL], 1);     // cannot happen: the list has a spare per row-shard
                            }
                        }
                        int4 *W1 = CHIP ? ch.W + (size_t)r1 * rc : (int4 *)(X.Wr + (size_t)o1 * X.rlp);
                        int4 *W2 = CHIP ? ch.W + (size_t)r2 * rc : (int4 *)(X.Wr + (size_t)o2 * X.rlp);
#pragma unroll
                        for (int y = 0; y < LPL; ++y)
#pragma unroll
                            for (int k = 0; k < CPL; ++k) {
                                const int u = y * CPL + k, ly = lane + 32 * y;
                                if (ly < L && (CPL == 1 || k < cpl)) {
                                    const int c = ly * cpl + (rot ? ((k + lane) & rot) : k);
                                    W1[c] = w1[u]; W2[c] = w2[u];
                                }
                            }
                    }
                    int better = 0;
                    const int wdf = __shfl_sync(0xffffffffu, df, ls);
                    if (lane < 2) {
                        // (all loads before the first store: the compiler cannot tell the arrays apart)
                        const int k = kb + ls, up = second ? 1 : -1, dt = second ? wti - wt2 : wt2 - wti;
                        const i64 dq = (i64)wt2 * wt2 - (i64)wti * wti;
                        ChainR *bk = ch.book;
                        const int T = ch.T[mc], m = ch.cnt[mc], nlog = bk->nlog, n_imp = bk->n_imp;
                        const u64 Q = ch.Q[mc], dig = bk->dig;
                        const i64 af = ch.Afx[mr], sk = ch.slack[mr], at = ident ? 0 : ch.att[mc];
                        const i64 B0 = bk->B[0], B1 = bk->B[1], B2 = bk->B[2];
                        const u32 other = swap ? (u32)wi2 : (u32)d2;
                        const u64 code = ((u64)(swap ? 0 : 1) << 63) ^ ((u64)(u32)k << 40) ^ ((u64)(u32)wi << 20) ^ (u64)other;
                        if (!second || swap) cells[second ? wi2 : wi] = (unsigned short)(second ? d1 : d2);
                        if (!swap) ch.cnt[mc] = m + up;
                        ch.T[mc] = T + dt;
                        ch.Q[mc] = second ? Q - (u64)dq : Q + (u64)dq;
                        if (!ident) { const i64 da = (aC + bS * (wt2 + wti)) * (wt2 - wti); ch.att[mc] = second ? at - da : at + da; }
                        ch.Afx[mr] = af + dA; ch.Jfx[mr] = Jn;
                        if (touchW) { ch.slack[mr] = sk + Em - eo + (second ? -wdf : wdf); ch.Esum[mr] = Em; }
                        ch.U[mg] = Un;
                        if (lane == 0) {
                            ch.Sc[0] = n0; ch.Sc[1] = n1; ch.Sc[2] = n2; ch.Sc[3] = en;
                            if (!CHIP && nlog < A.log_cap) A.log[(size_t)j * A.log_cap + nlog] = make_uint2((u32)wi, other | (swap ? 0u : 0x80000000u));
                            bk->nlog = nlog + 1;
                            bk->dig = (dig ^ code) * 0x100000001B3ull;
                            if (rp_lex_less(n0, n1, n2, B0, B1, B2)) {
                                bk->B[0] = n0; bk->B[1] = n1; bk->B[2] = n2;
                                bk->best_step = k + 1; bk->best_nlog = nlog + 1;
                                bk->n_imp = n_imp + 1;
                                if (CHIP) better = rp_lex_less(n0, n1, n2, inc_s[0], inc_s[1], inc_s[2]) ? 1 : 0;
                            }
                            if (touchW) n_rows += 2;
                        }
                    }
                    // the cached cells of the steps still to come follow the move
                    {
                        const int n = sr.flags & 1u ? 2 : 4;
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            if (x < n && sr.i[x] == wi) sr.c[x] = d2;
                            if (x < n && sr.i[x] == wi2) sr.c[x] = d1;      // (no sample is -1; wi2 != wi, their cells differ)
                        }
                    }
                    __syncwarp();                               // the updates are visible
                    if (!ident && lane < 2 * dm.S) {
                        const bool b = lane >= dm.S;
                        const int c = b ? d2 : d1;
                        row_top_stage(dm, ch, dpl, dpo, rowbase[c], g_of[c], b ? r2 : r1, lane - (b ? dm.S : 0));
                    }
                    if (CHIP && __any_sync(0xffffffffu, better)) {
                        // a trajectory best that beats the incumbent of the level's start: keep its layout
                        for (int x = lane; x < (dm.N + 3) >> 2; x += 32) ((uint2 *)ch.snap)[x] = ((const uint2 *)ch.cell)[x];
                        if (lane == 0) ch.book->has_snap = 1;
                    }
                    if (!ident || CHIP) __syncwarp();
                    break;
                }
                if (ok && (win < 0 || lane <= win)) { n_feas += 1; if (rg1 != rg2) n_rows += mi2 >= 0 ? 4 : 3; }
                pos = win < 0 ? nb : win + 1;
            }
            __syncwarp();                       // the stores to the assignment come before the next batch's reads
        }
        __syncwarp();
    } else if (CHIP && warp >= cw && !last) make_recs(ln + 1, cw, NT / 32 - cw);

    // ---- epilogue of the level: the chain's report and terminal state ------------------------------
    const size_t rep = CHIP ? (size_t)(ln & 1) * P : 0;     // CHIP: two sets of reports taken in turn (a chain that
                                                            // runs ahead must not overwrite what a slower one still reads)
    if (live) {
        n_feas = __reduce_add_sync(0xffffffffu, n_feas);
        n_rows = warp_sum_i64(n_rows);
    }
    if (live && lane == 0) {
        const ChainR *bk = ch.book;
        const i64 B0 = bk->B[0], B1 = bk->B[1], B2 = bk->B[2];
        if (CHIP) {
            // what the level barrier reads first: the energy, and in its top bit whether the trajectory best beats the incumbent
            const bool beats = rp_lex_less(B0, B1, B2, inc_s[0], inc_s[1], inc_s[2]);
            A.lo.F[rep + j] = (u64)ch.Sc[3] | (beats ? 1ull << 63 : 0ull);
        }
        if (!CHIP || A.lo.tr_term) for (int x = 0; x < 3; ++x) A.term[3 * (rep + j) + x] = ch.Sc[x];
        A.best[3 * (rep + j)] = B0; A.best[3 * (rep + j) + 1] = B1; A.best[3 * (rep + j) + 2] = B2;
        if (!CHIP || A.lo.tr_term) { A.best_step[rep + j] = bk->best_step; A.digest[rep + j] = bk->dig; }
        if (!CHIP) A.best_nlog[j] = bk->best_nlog;
        if (!CHIP && !A.last) { A.lo.F[j] = (u64)ch.Sc[3]; atomicMin(A.lo.F + 2 * (size_t)P, (u64)ch.Sc[3]); }
        sum_feas += n_feas; sum_acc += n_acc; sum_imp += bk->n_imp; sum_rows += n_rows;
        if (!CHIP || last) {
            atomicAdd((u64 *)&A.counters[0], (u64)A.steps * n_levels);
            atomicAdd((u64 *)&A.counters[1], (u64)sum_feas);
            atomicAdd((u64 *)&A.counters[2], (u64)sum_acc);
            atomicAdd((u64 *)&A.counters[3], (u64)sum_imp);
            atomicAdd((u64 *)&A.counters[4], (u64)(sum_rows * dm.LP * 4));
        }
    }
    if (CHIP && live && ch.book->has_snap) {
        unsigned short *row = A.lo.cand_layout + (size_t)j * dm.N;
        for (int x = lane; x < dm.N; x += 32) row[x] = ch.snap[x];
    }
    if (!CHIP) {
        char *bdst = A.blob_dst + (size_t)j * A.bl.bytes;
        const int n16 = A.bl.off_cell >> 4;
        for (int x = lane; x < n16; x += 32) ((int4 *)bdst)[x] = ((const int4 *)ch.base)[x];
        for (int x = (n16 << 2) + lane; x < nhw; x += 32) ((int *)bdst)[x] = ((const int *)ch.base)[x];
        int *td = (int *)(bdst + A.bl.off_wtab);
        for (int rg = lane; rg < dm.RG; rg += 32) { td[rg] = ch.wtab[rg]; X.F_dst[(size_t)j * dm.RG + rg] = ch.slack[rg]; }
        return;
    } else {
        // Meet the other chains: the reports are all they wait for, so arrive as soon as they are out.
        __threadfence();
        __syncthreads();
        if (tid == 0) {
            atomicAdd(A.sync, 1);
            // (the pool may be written once every chain has read its start state)
            failed_s = (ln == 0 && !rp_wait_count(A.lo.done, (int)gridDim.x, A)) ? 1 : 0;
        }
        __syncthreads();
        if (failed_s) { if (tid == 0) atomicExch(&A.status[RP_SW_TIMEOUT], 1); return; }
        const RpLevelDev lv = A.levels[ln];              // fetched before the wait
        char *buf_out = ((A.cur0 + ln + 1) & 1) ? A.blob_b1 : A.blob_b0;
        i64 *F_out = X.F_buf + (((A.cur0 + ln + 1) & 1) ? (size_t)P * dm.RG : 0);
        const int nw = dm.RG * rc;
        // Terminal states with plain stores, the warps split over the chains (cw is a power of two), then the members' flags.
        const int hw = warp & (cw - 1), jj = blockIdx.x * cw + hw, ht = (warp / cw) * 32 + lane, hn = NT / cw;
        if (jj < P) {
            const RowChain c = row_chain(A, X, sm_chain, hw);
            char *bdst = buf_out + (size_t)jj * A.bl.bytes;
            int4 *wd = (int4 *)(X.Wr + (size_t)(half_w * P + jj) * dm.RG * X.rlp);
#pragma unroll 4
            for (int x = ht; x < nw; x += hn) wd[x] = c.W[x];
            const int n16 = A.bl.off_cell >> 4;
            for (int x = ht; x < n16; x += hn) ((int4 *)bdst)[x] = ((const int4 *)c.base)[x];
            for (int x = (n16 << 2) + ht; x < nhw; x += hn) ((int *)bdst)[x] = ((const int *)c.base)[x];
            unsigned short *cd = (unsigned short *)(bdst + A.bl.off_cell);
            for (int x = ht; x < n4; x += hn) ((uint2 *)cd)[x] = ((const uint2 *)c.cell)[x];
            for (int i = (n4 << 2) + ht; i < dm.N; i += hn) cd[i] = c.cell[i];
            for (int rg = ht; rg < dm.RG; rg += hn) F_out[(size_t)jj * dm.RG + rg] = c.slack[rg];
            if (A.slices) {
                int *td = (int *)(bdst + A.bl.off_wtab);
                for (int rg = ht; rg < dm.RG; rg += hn) td[rg] = (half_w * P + jj) * dm.RG + rg;
            }
        }
        __threadfence();
        __syncthreads();
        if (tid < cw && blockIdx.x * cw + tid < P)
            asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(A.sync + 1 + blockIdx.x * cw + tid), "r"(ln + 1) : "memory");
        if (tid == 0) failed_s = rp_wait_count(A.sync, (ln + 1) * (int)gridDim.x, A) ? 0 : 1;
        __syncthreads();
        if (failed_s) { if (tid == 0) atomicExch(&A.status[RP_SW_TIMEOUT], 1); return; }

        // ---- the level barrier, worked out by every CTA for itself (all integer, so all agree) -------
        u64 *le_F = (u64 *)(sm_cta + X.off_leF);
        int *le_anc = (int *)(le_F + P);
        const i64 *termL = A.term + 3 * rep, *bestL = A.best + 3 * rep;
        const u64 *eL = A.lo.F + rep;
        __shared__ i64 r0[NT / 32], r1s[NT / 32], r2s[NT / 32], rmin[NT / 32];
        __shared__ int rj[NT / 32];
        __shared__ u64 rsum[LE_MAX_WARPS];
        __shared__ u64 carry_s;
        __shared__ int win_s;
        const bool all_anc = blockIdx.x == 0 && A.lo.tr_anc;        // the first CTA writes the traces
        const int m0 = all_anc ? 0 : blockIdx.x * cw, m1 = all_anc ? P : min(P, m0 + cw);
        if (P <= 32) {
            if (warp == 0) row_barrier_warp(A, P, eL, bestL, last, lv.cq, lv.resample_x, m0, m1, inc_s, &win_s, le_anc, lane);
            __syncthreads();
            if (win_s >= 0) inc_slot = win_s;
        } else {
        // incumbent: the lowest slot among the lexicographically best trajectory-best scores, if it beats it
        i64 b0 = inc_s[0], b1 = inc_s[1], b2 = inc_s[2], emin = 0x7fffffffffffffffll, e_mine = emin;
        int bj = 0x7fffffff;
        for (int m = tid; m < P; m += NT) {
            const u64 r = __ldcg(eL + m);
            const i64 e = (i64)(r & ~(1ull << 63));
            if (r >> 63) {
                const i64 s0 = __ldcg(bestL + 3 * m), s1 = __ldcg(bestL + 3 * m + 1), s2 = __ldcg(bestL + 3 * m + 2);
                if (rp_lex_less(s0, s1, s2, b0, b1, b2)) { b0 = s0; b1 = s1; b2 = s2; bj = m; }
            }
            emin = e < emin ? e : emin;
            e_mine = e;
        }
        {
            const u32 hi = (u32)((u64)emin >> 32), mh = __reduce_min_sync(0xffffffffu, hi);
            const u32 ml = __reduce_min_sync(0xffffffffu, hi == mh ? (u32)emin : 0xffffffffu);
            emin = (i64)(((u64)mh << 32) | ml);
            const int s = le_lexmin_lane(b0, b1, b2, bj), sl = s < 0 ? 0 : s;
            b0 = __shfl_sync(0xffffffffu, b0, sl); b1 = __shfl_sync(0xffffffffu, b1, sl); b2 = __shfl_sync(0xffffffffu, b2, sl);
            bj = __shfl_sync(0xffffffffu, bj, sl);
            if (s < 0) bj = 0x7fffffff;
        }
        if (lane == 0) { r0[warp] = b0; r1s[warp] = b1; r2s[warp] = b2; rj[warp] = bj; rmin[warp] = emin; }
        if (tid == 0) { carry_s = 0; win_s = -1; }
        __syncthreads();
#pragma unroll
        for (int w = 0; w < NT / 32; ++w) emin = rmin[w] < emin ? rmin[w] : emin;
        if (warp == 0) {
            const bool has = lane < NT / 32;
            b0 = has ? r0[lane] : 0; b1 = has ? r1s[lane] : 0; b2 = has ? r2s[lane] : 0;
            bj = has ? rj[lane] : 0x7fffffff;
            const int s = le_lexmin_lane(b0, b1, b2, bj), sl = s < 0 ? 0 : s;
            b0 = __shfl_sync(0xffffffffu, b0, sl); b1 = __shfl_sync(0xffffffffu, b1, sl); b2 = __shfl_sync(0xffffffffu, b2, sl);
            bj = __shfl_sync(0xffffffffu, bj, sl);
            if (lane == 0 && s >= 0 && rp_lex_less(b0, b1, b2, inc_s[0], inc_s[1], inc_s[2])) {
                inc_s[0] = b0; inc_s[1] = b1; inc_s[2] = b2;
                win_s = bj;                     // that chain stored its trajectory-best layout in its row of cand_layout
            }
        }
        __syncthreads();
        if (win_s >= 0) inc_slot = win_s;
        // Boltzmann weights, cumulative weights, ancestors (not after the last level)
        if (!last) {
            const u64 M = (u64)(emin > dm.SC ? emin : dm.SC);
            auto en_of = [&](int m) { return (i64)(__ldcg(eL + m) & ~(1ull << 63)); };
            if (P <= NT) le_prefix_weights_of<1>(P, [&](int) { return e_mine; }, lv.cq, tid, NT, emin, M, le_F, rsum, &carry_s);
            else if (P <= 2 * NT) le_prefix_weights_of<2>(P, en_of, lv.cq, tid, NT, emin, M, le_F, rsum, &carry_s);
            else le_prefix_weights_of<4>(P, en_of, lv.cq, tid, NT, emin, M, le_F, rsum, &carry_s);
            const u64 Ftot = le_F[P - 1];
            const u64 u0 = (u64)(((unsigned __int128)lv.resample_x * Ftot) >> 32);
            for (int m = m0 + tid; m < m1; m += NT) {
                const unsigned __int128 at = (unsigned __int128)u0 + (unsigned __int128)m * Ftot;
                int lo = 0, hi = P - 1;
                while (lo < hi) {                       // smallest slot with P * F > at
                    const int mid = (lo + hi) >> 1;
                    if ((unsigned __int128)P * le_F[mid] > at) hi = mid; else lo = mid + 1;
                }
                le_anc[m] = lo;
            }
            __syncthreads();
        }
        }
        // per-level traces (inspection hook), by the first CTA
        if (blockIdx.x == 0 && A.lo.tr_term) {
            const size_t o = (size_t)level * P;
            for (int x = tid; x < 3 * P; x += NT) { A.lo.tr_term[o * 3 + x] = __ldcg(termL + x); A.lo.tr_best[o * 3 + x] = __ldcg(bestL + x); }
            for (int x = tid; x < P; x += NT) {
                A.lo.tr_best_step[o + x] = __ldcg(A.best_step + rep + x);
                A.lo.tr_digest[o + x] = __ldcg(A.digest + rep + x);
                if (!last) A.lo.tr_anc[o + x] = le_anc[x];
            }
            if (tid < 3) A.lo.tr_inc[(size_t)level * 3 + tid] = inc_s[tid];
        }
        if (last) {
            const i64 wb = (i64)dm.RG * dm.LP * 4;
            if (ht == 0 && jj < P) { if (moved) atomicAdd((u64 *)&A.counters[5], (u64)(2 * wb * moved)); atomicAdd((u64 *)&A.counters[6], (u64)(wb * n_levels)); }
            // The terminal states are the population as they stand: every member descends from itself,
            // its rank loads sit where this level wrote them; the first CTA hands the incumbent over.
            if (tid < cw && blockIdx.x * cw + tid < P) {
                const int me = blockIdx.x * cw + tid;
                A.lo.anc_out[me] = me; A.lo.anc_cur[me] = me;
                A.lo.wloc_out[me] = half_w * P + me; A.wloc_dst[me] = half_w * P + me;
            }
            if (blockIdx.x == 0) {
                if (tid < 3) A.lo.inc_score[tid] = inc_s[tid];
                if (inc_slot >= 0) {
                    const unsigned short *row = A.lo.cand_layout + (size_t)inc_slot * dm.N;
                    for (int i = tid; i < dm.N; i += NT) A.lo.inc_layout[i] = __ldcg(row + i);
                }
            }
            return;
        }
        // next level: a slot continues from its ancestor's terminal state; its own is still on chip
        if (tid == 0) failed_s = 0;
        __syncthreads();
        if (tid < cw && blockIdx.x * cw + tid < P) {
            const int a = le_anc[blockIdx.x * cw + tid];
            if (a != blockIdx.x * cw + tid && !rp_wait_count(A.sync + 1 + a, ln + 1, A)) failed_s = 1;       // its state is complete
        }
        __syncthreads();
        if (failed_s) { if (tid == 0) atomicExch(&A.status[RP_SW_TIMEOUT], 1); return; }
        const int a = jj < P ? le_anc[jj] : jj;
        if (a != jj) {
            const RowChain c = row_chain(A, X, sm_chain, hw);
            const char *bs = buf_out + (size_t)a * A.bl.bytes;
            const int4 *ws = (const int4 *)(X.Wr + (size_t)(half_w * P + a) * dm.RG * X.rlp);
            const unsigned short *cs = (const unsigned short *)(bs + A.bl.off_cell);
#pragma unroll 8
            for (int x = ht; x < nw; x += hn) c.W[x] = __ldcg(ws + x);
#pragma unroll 4
            for (int x = ht; x < nh16; x += hn) ((int4 *)c.base)[x] = __ldcg((const int4 *)bs + x);
#pragma unroll 4
            for (int x = ht; x < n4; x += hn) ((uint2 *)c.cell)[x] = __ldcg((const uint2 *)cs + x);
            for (int i = (n4 << 2) + ht; i < dm.N; i += hn) c.cell[i] = __ldcg(cs + i);
            for (int rg = ht; rg < dm.RG; rg += hn) c.slack[rg] = __ldcg(F_out + (size_t)a * dm.RG + rg);
            if (ht == 0) moved += 1;
        }
        half_w ^= 1;
        __syncthreads();
    }
    }
}

// ---------------------------------------------------------------------------------------------
// Demand rows in the kernel's form, the fixed ranks, and the sums of a member's row-shards.
// ---------------------------------------------------------------------------------------------
// Ranks of a layer by decreasing aggregate load (ties: lower rank): the first is the fixed rank, the first three
// are the columns of a compressed row.  One warp per sample: f_i, and (qr != null) its row: padded to whole
// 16-byte chunks with zeros, or compressed.
__global__ void __launch_bounds__(256)
k_make_rows(RpDims dm, const int *__restrict__ t, const int *__restrict__ q, const int *__restrict__ top, int cols, int comp, int use_f,
            int2 *__restrict__ tf, int *__restrict__ qr)
{
    const int lane = threadIdx.x & 31, nw = gridDim.x * (blockDim.x >> 5);
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < dm.N; i += nw) {
        int f = 0;
        for (int l = lane; l < dm.L; l += 32) {
            const int *row = q + ((size_t)i * dm.L + l) * dm.P;
            const int b0 = __ldg(top + 3 * l), b1 = __ldg(top + 3 * l + 1), b2 = __ldg(top + 3 * l + 2);
            const int x0 = __ldg(row + b0);
            f += x0;
            if (qr && comp) {
                int rest = 0;
                for (int p = 0; p < dm.P; ++p) { const int v = __ldg(row + p); if (p != b0 && p != b1 && p != b2) rest = max(rest, v); }
                ((int4 *)qr)[(size_t)i * dm.L + l] = make_int4(x0, __ldg(row + b1), __ldg(row + b2), rest);
            } else if (qr) {
                int *o = qr + ((size_t)i * dm.L + l) * cols;
                for (int p = 0; p < cols; ++p) o[p] = p < dm.P ? __ldg(row + p) : 0;
            }
        }
        f = __reduce_add_sync(0xffffffffu, f);
        if (lane == 0) tf[i] = make_int2(__ldg(t + i), use_f ? f : 0);
    }
}

// Member m = blockIdx.x, row-shard rg = blockIdx.y: the slack (sum of the busiest loads less the samples' f), and (Wr != null) the row-shard's
// slice in row form, in the place its table names (windows without a table: cell m of the pool).
// Compressed rows also count the row-shards with a layer whose three columns do not decide the maximum; `loose`: counts those
// whose busiest loads exceed their samples' f by more than a sixteenth.
__global__ void __launch_bounds__(256)
k_member_rows(RpDims dm, RpBlob bl, const char *__restrict__ blobs, const char *__restrict__ static_blk, RpStatic sl, const int2 *__restrict__ tf,
              const int *__restrict__ qr, int rlp, int comp, i64 *__restrict__ Fo, int *__restrict__ Wr, const int *__restrict__ wloc, int *__restrict__ undecided, int loose)
{
    extern __shared__ int list[];                       // [N] samples of the row-shard
    __shared__ int n_s, bad_s;
    __shared__ u64 f_s;
    const int m = blockIdx.x, rg = blockIdx.y, tid = threadIdx.x;
    const char *blob = blobs + (size_t)m * bl.bytes;
    const unsigned short *cells = (const unsigned short *)(blob + bl.off_cell);
    const unsigned short *rg_of = (const unsigned short *)(static_blk + sl.off_rg);
    if (tid == 0) { n_s = 0; f_s = 0; bad_s = 0; }
    __syncthreads();
    i64 f = 0;
    for (int i = tid; i < dm.N; i += 256)
        if (__ldg(rg_of + cells[i]) == rg) { f += __ldg(&tf[i].y); if (Wr) list[atomicAdd(&n_s, 1)] = i; }
    if (f) atomicAdd(&f_s, (u64)f);
    __syncthreads();
    if (tid == 0) {
        const i64 es = ((const i64 *)(blob + bl.off_Esum))[rg], slack = es - (i64)f_s;
        Fo[(size_t)m * dm.RG + rg] = slack;
        if (loose && slack * 16 > es) atomicAdd(undecided, 1);
    }
    if (!Wr) return;
    const int n = n_s;
    const size_t slice = bl.off_wtab >= 0 ? (size_t)((const int *)(blob + bl.off_wtab))[rg] : (size_t)wloc[m] * dm.RG + rg;
    int4 *out = (int4 *)(Wr + slice * rlp);
    for (int x = tid; x < rlp >> 2; x += 256) {
        int4 acc = make_int4(0, 0, 0, 0);
#pragma unroll 8
        for (int e = 0; e < n; ++e) acc = add4(acc, __ldg((const int4 *)(qr + (size_t)list[e] * rlp) + x));
        out[x] = acc;
        if (comp && acc.w > max(max(acc.x, acc.y), acc.z)) bad_s = 1;
    }
    __syncthreads();
    if (comp && tid == 0 && bad_s) atomicAdd(undecided, 1);
}

// ---------------------------------------------------------------------------------------------
// Which windows, which form.
// ---------------------------------------------------------------------------------------------
static int lanes_of(int L) { return L <= 32 ? 1 : (L <= 64 ? 2 : (L <= 128 ? 4 : 0)); }      // layers per lane (template values)
static int chunks_of(int cpl) { return cpl <= 1 ? 1 : (cpl <= 2 ? 2 : (cpl <= 4 ? 4 : (cpl <= 8 ? 8 : 0))); }

// Chunks a lane holds per row, as the kernel is instantiated; 0 = not at all.
static int row_chunks(const RpDims &dm, int cpl)
{
    const int l = lanes_of(dm.L), c = chunks_of(cpl);
    return l * c;
}

static int row_chains_per_cta(int pop, int sms) { return pop <= sms ? 1 : (pop <= 2 * sms ? 2 : (pop <= 4 * sms ? 4 : 8)); }

static void chain_layout(const RpDims &dm, const RpBlob &bl, const RpStatic &sl, RowArgs &X, bool chip, int cw, int pop, int steps)
{
    size_t o = 0;
    o = ((size_t)sl.off_t + 15) & ~(size_t)15;
    X.off_tab = (int)o;   o += (size_t)(sl.bytes - sl.off_rg);
    o = (o + 15) & ~(size_t)15;
    X.off_leF = (int)o;   o += chip ? (size_t)12 * pop : 0;
    o = (o + 15) & ~(size_t)15;
    X.off_chain = (int)o;
    size_t c = ((size_t)bl.off_cell + 15) & ~(size_t)15;
    X.off_F = (int)c;     c += (size_t)8 * dm.RG;
    X.off_book = (int)c;  c += ((sizeof(ChainR) + 7) & ~(size_t)7) + 8;
    X.off_wtab = (int)c;  c += chip ? 0 : (size_t)4 * dm.RG;
    X.off_spare = (int)c; c += chip ? 0 : (size_t)4 * dm.RG;
    c = (c + 7) & ~(size_t)7;
    X.off_top = (int)c;   c += dm.own_shard ? 0 : (size_t)8 * dm.K + (size_t)18 * dm.RG * dm.S;
    c = (c + 15) & ~(size_t)15;
    const size_t lay = (2 * (size_t)dm.N + 15) & ~(size_t)15;
    X.off_cell = (int)c;  c += chip ? lay : 0;
    X.off_snap = (int)c;  c += chip ? lay : 0;
    // (records of 256 steps at most, twice)
    X.recs = chip && cw < ROW_THREADS / 32 ? std::min(steps, 256) : 0;
    X.off_recs = (int)c;  c += (size_t)2 * X.recs * sizeof(StepRec);
    c = (c + 15) & ~(size_t)15;
    X.off_list = (int)c;  c += X.comp ? (size_t)4 * (ROW_LIST + 1) : 0;
    X.off_W = (int)c;     c += chip ? (size_t)4 * dm.RG * X.rlp : 0;
    X.chain_bytes = (int)((c + 15) & ~(size_t)15);
    X.smem_bytes = X.off_chain + X.chain_bytes * cw;
    X.cw = cw;
}

// Full rows (padded to whole chunks).
static void full_rows(const RpDims &dm, RowArgs &X)
{
    X.cpl = (dm.P + 3) / 4; X.rlp = dm.L * X.cpl * 4; X.comp = 0;
}

// One launch for all levels, the chains' rank loads on chip: at most eight chunks per lane, every chain resident at once.
#define ROW_SMEM_MAX (220 * 1024)
bool rp_row_fits_chip(rp_ctx *c, const RpBlob &bl, const RpStatic &sl)
{
    RowArgs X;
    memset(&X, 0, sizeof X);
    full_rows(c->dm, X);
    const int nch = row_chunks(c->dm, X.cpl), sms = rp_sms(c);          // (a CTA to an SM)
    if (nch < 1 || nch > 8 || c->Ppop > sms * ROW_MAX_WARPS || c->dm.N > 16384) return false;
    c->row_cw = row_chains_per_cta(c->Ppop, sms);
    chain_layout(c->dm, bl, sl, X, true, c->row_cw, c->Ppop, 0);
    return X.smem_bytes <= ROW_SMEM_MAX;
}

// Rows this window would use in the form that launches once per level: 0 none, 1 full, 2 compressed.
int rp_row_kind(const RpDims &dm)
{
    const int cpl = (dm.P + 3) / 4, nch = row_chunks(dm, cpl);
    if (nch >= 1 && nch <= 4) return 1;
    if (dm.P >= 8 && dm.P <= 128 && lanes_of(dm.L)) return 2;      // (128: ranks the placement kernel orders)
    return 0;
}

// Whether the form that launches once per level is taken by the shared memory of a chain (a warp to itself).  Where DP slot d is
// shard d, as far as it fits: it is the fastest kernel even with one chain per SM (L = 24, P = 16, 1024 members, three levels of
// 200 steps: 63 KB 1.39 ms and 1.71 for the next best kernel, 117 KB 3.8 and 4.8, 140 KB 4.1 and 4.9; L = P = 32, 2048 members,
// three of 100: 94 KB 2.2 and 3.0, 136 KB 6.0 and 8.1).  Else the attention of a shard's slots is looked up
// (8*K + 18*R*G*S bytes more, S stages a move) and four-warp CTAs overtake it: with up to two stages where an SM holds fewer than
// two chains (107 KB 2.3 ms and 2.9, 133 KB 3.7 and 3.2, 166 KB 4.9 and 4.3), with more where it holds fewer than three (four
// stages 72 KB 1.82 and 1.83, 107 KB 2.61 and 2.52; eight stages 54 KB 1.94 and 1.85, 81 KB 2.6 and 2.2, 161 KB 5.4 and 3.1).
bool rp_row_fits_level(const rp_ctx *c, const RpBlob &bl, const RpStatic &sl)
{
    RowArgs X;
    memset(&X, 0, sizeof X);
    X.comp = rp_row_kind(c->dm) == 2;
    chain_layout(c->dm, bl, sl, X, false, 1, c->Ppop, 0);
    const int limit = c->dm.own_shard ? ROW_SMEM_MAX : 227 * 1024 / (c->dm.S <= 2 ? 2 : 3) - 1024;
    return X.smem_bytes <= limit;
}

// Whether rows are kept apart from the rank loads that scoring writes: padded or compressed.
bool rp_row_separate(const rp_ctx *c)
{
    const RpDims &dm = c->dm;
    if (c->row_mode == 1) return (dm.P & 3) != 0;
    const int kind = rp_row_kind(dm);
    return kind == 2 || (kind == 1 && (dm.P & 3));
}
// (the larger form, so that a later choice between the two needs no new memory)
size_t rp_row_ints(const rp_ctx *c)
{
    if (c->row_mode != 1 && rp_row_kind(c->dm) == 2) return (size_t)c->dm.L * 4;
    return (size_t)c->dm.L * ((c->dm.P + 3) / 4) * 4;
}

static void row_args(rp_ctx *c, RowArgs &X)
{
    memset(&X, 0, sizeof X);
    full_rows(c->dm, X);
    if (c->row_mode != 1 && rp_row_kind(c->dm) == 2) { X.cpl = 1; X.rlp = c->dm.L * 4; X.comp = 1; }
    const bool sep = rp_row_separate(c);
    X.qr = sep ? c->d_qr : c->d_q;
    X.Wr = sep ? c->d_Wr : c->d_W;
    X.tf = (const int2 *)c->d_tf;
    X.F_buf = c->d_rowF;
    X.F_src = c->d_rowF + (size_t)c->cur * c->Ppop * c->dm.RG;
    X.F_dst = c->d_rowF + (size_t)(1 - c->cur) * c->Ppop * c->dm.RG;
}

// Rows of the samples, once per context's placement and packing.
int rp_launch_make_rows(rp_ctx *c)
{
    const RpDims &dm = c->dm;
    RowArgs X;
    row_args(c, X);
    const int use_f = (double)dm.L * dm.k * dm.C < 2147483648.0;          // f_i <= L*k*C must fit 32 bits (0 rejects nothing)
    const int want = (dm.N + 7) / 8;
    k_make_rows<<<want < 148 * 4 ? want : 148 * 4, 256, 0, c->stream>>>(
        dm, c->d_t, c->d_q, c->d_top, X.cpl * 4, X.comp, use_f, (int2 *)c->d_tf, rp_row_separate(c) ? c->d_qr : nullptr);
    ++g_rp_launches;
    RP_CUDA(cudaGetLastError());
    return RP_OK;
}

// Row-shard sums (and rows) of members 0 .. n-1 of the current buffer.
int rp_launch_member_rows(rp_ctx *c, int n)
{
    const RpDims &dm = c->dm;
    RowArgs X;
    row_args(c, X);
    const bool sep = rp_row_separate(c);
    const size_t smem = sep ? sizeof(int) * (size_t)dm.N : 0;
    if (smem > 200 * 1024) return RP_ERR_RANGE;
    if (smem > 32 * 1024) RP_CUDA(cudaFuncSetAttribute(k_member_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(200 * 1024)));
    RP_CUDA(cudaMemsetAsync(c->d_undecided, 0, sizeof(int), c->stream));
    k_member_rows<<<dim3(n, dm.RG), 256, smem, c->stream>>>(dm, c->bl, c->buf[c->cur].blob, c->d_static, c->sl, (const int2 *)c->d_tf, X.qr,
                                                            X.rlp, X.comp, c->d_rowF + (size_t)c->cur * c->Ppop * dm.RG,
                                                            sep ? c->d_Wr : nullptr, c->d_wloc, c->d_undecided, c->row_check);
    ++g_rp_launches;
    RP_CUDA(cudaGetLastError());
    c->row_counted = n;
    return RP_OK;
}

template <int LPL, int CPL, bool CHIP, bool COMP>
static int launch_row_t(rp_ctx *c, const AnnealArgs &A, const RowArgs &X, int grid, int threads, int *done)
{
    auto kern = k_anneal_row<LPL, CPL, CHIP, COMP>;
    // (always the same value, above anything a launch asks for: contexts that plan different
    // windows at once on different host threads then never lower each other's limit)
    RP_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, ROW_SMEM_MAX));
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    *done = 0;
    if (CHIP && grid > rp_sms(c)) return RP_OK;
    cfg.gridDim = dim3(grid); cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = X.smem_bytes; cfg.stream = c->stream;
    cudaLaunchAttribute at[1];
    if (CHIP) {
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
        cfg.attrs = at; cfg.numAttrs = 1;
    }
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, A, X);
    if (CHIP && e == cudaErrorCooperativeLaunchTooLarge) { cudaGetLastError(); return RP_OK; }
    RP_CUDA(e);
    ++g_rp_launches; ++c->n_queued;
    *done = 1;
    return RP_OK;
}

// One launch for all levels; *done = 0 when the chains cannot all be resident: fewer SMs are free than the device reported when
// the population was built (a part of a GPU).  The caller then takes another kernel.
int rp_launch_anneal_row_all(rp_ctx *c, const AnnealArgs &A0, int *done)
{
    AnnealArgs A = A0;
    RowArgs X;
    row_args(c, X);
    const int cw = c->row_cw;
    // step records ahead of time as far as shared memory goes
    for (int steps = std::min(A.steps, 256);; steps /= 2) {
        chain_layout(c->dm, c->bl, c->sl, X, true, cw, c->Ppop, steps);
        if (X.smem_bytes <= ROW_SMEM_MAX || steps == 0) break;
    }
    A.w_on_chip = 1;
    A.slices = c->dm.slices;
    A.smem_bytes = (unsigned)X.smem_bytes;
    A.lo.cand_layout = c->d_cand_layout;
    const int grid = (c->Ppop + cw - 1) / cw, nt = ROW_THREADS;
    const int l = lanes_of(c->dm.L), k = chunks_of(X.cpl);
#define ROW_CASE(L_, K_) if (l == L_ && k == K_) return launch_row_t<L_, K_, true, false>(c, A, X, grid, nt, done)
    ROW_CASE(1, 1); ROW_CASE(1, 2); ROW_CASE(1, 4); ROW_CASE(1, 8);
    ROW_CASE(2, 1); ROW_CASE(2, 2); ROW_CASE(2, 4);
    ROW_CASE(4, 1); ROW_CASE(4, 2);
#undef ROW_CASE
    return RP_ERR_STATE;
}

int rp_launch_level_end(rp_ctx *c, const AnnealArgs &A);
int rp_launch_level_turn(rp_ctx *c, const AnnealArgs &A);

int rp_launch_anneal_row(rp_ctx *c, AnnealArgs &A)
{
    RowArgs X;
    row_args(c, X);
    chain_layout(c->dm, c->bl, c->sl, X, false, 1, c->Ppop, 0);
    if (X.smem_bytes > ROW_SMEM_MAX) return RP_ERR_RANGE;
    A.smem_bytes = (unsigned)X.smem_bytes;
    A.slices = 1;
    A.lo.cand_layout = nullptr;
    const int l = lanes_of(c->dm.L), k = chunks_of(X.cpl);
    int done = 0, st = RP_ERR_STATE;
#define ROW_CASE(L_, K_) else if (l == L_ && k == K_) st = launch_row_t<L_, K_, false, false>(c, A, X, c->Ppop, 32, &done)
    if (X.comp) {
        if (l == 1) st = launch_row_t<1, 1, false, true>(c, A, X, c->Ppop, 32, &done);
        else if (l == 2) st = launch_row_t<2, 1, false, true>(c, A, X, c->Ppop, 32, &done);
        else st = launch_row_t<4, 1, false, true>(c, A, X, c->Ppop, 32, &done);
    }
    ROW_CASE(1, 1); ROW_CASE(1, 2); ROW_CASE(1, 4); ROW_CASE(2, 1); ROW_CASE(2, 2); ROW_CASE(4, 1);
#undef ROW_CASE
    RP_TRY(st);
    if (!A.last && rp_row_turns(c)) return rp_launch_level_turn(c, A);
    return rp_launch_level_end(c, A);
}
