// The one-layer-per-lane chain kernel (see rp_anneal_row.cu for what it does and which windows take it).
//
// A round (propose, score, decide, commit) is a chain of dependent instructions of one warp, so what counts is how many there are
// and what they wait for.  The state of a chain is kept as records (cost and attention part of a row-shard in 16 bytes, tokens and
// samples of a cell in 8), its score, energy and trajectory best in registers; both sides of a move look at their entries once, for
// the decision and the commit; a slice table entry carries where the next rewrite goes; what leaves a best layout behind copies it,
// not what finds it; windows whose slot d is shard d have instances of their own.  In cycles, alone on an SM (medium): proposals 874 ->
// 503, scoring 934 -> 740, decision 467 -> 378, commit 902 -> 566; plans 1.12 times as fast.  With the barrier, the dealt-out rows and
// the shared warps below: medium 972 -> 807 us, large 3169 -> 2499, two shards 916 -> 816, ragged 1781 -> 1570, wide 10.9 -> 9.8 ms, heavy
// 83.4 -> 59.3 (windows of perf/cases.py, seed 5, one GPU; times below without a window's sizes are of these).
#pragma once
#include <algorithm>
#include <string.h>

#include "rp_level_end.cuh"
#include "rp_anneal_row.cuh"

struct StepX {                   // what a lane keeps about the step it proposes for
    u32 bz;
    u64 thr;                     // top bit: every rise is accepted
    float thrf;                  // thr / 2^32, rounded up; infinite where every rise is accepted
    int i[4];                    // samples; for a relocation i[2], i[3] are negative
    u32 c[4];                    // cell of sample i[x], or the target cell; its shard (IDENT) or row-shard in the upper half
    int t[4], f[4];              // length of sample i[x] and its demand on the fixed ranks (0 for relocation targets)
};

// The GL lanes that run a chain (all 32 of a warp, or 16): shuffles, votes and sums among them.
template <int GL>
struct Lanes {
    static constexpr unsigned FULL = 0xffffffffu;
    __device__ static __forceinline__ unsigned mask(int lane) { return GL == 32 ? FULL : 0xffffu << (lane & 16); }
    __device__ static __forceinline__ unsigned ballot(bool p, int lane)
    {
        const unsigned b = __ballot_sync(FULL, p);
        return GL == 32 ? b : (b >> (lane & 16)) & 0xffffu;
    }
    __device__ static __forceinline__ bool any(bool p, int lane) { return GL == 32 ? __any_sync(FULL, p) != 0 : ballot(p, lane) != 0; }
    template <class T> __device__ static __forceinline__ T get(T v, int src) { return __shfl_sync(FULL, v, src, GL); }
    template <class T> __device__ static __forceinline__ T swap(T v) { return __shfl_xor_sync(FULL, v, 1); }
    __device__ static __forceinline__ i64 max_nonneg(i64 v)
    {
        if (GL == 32) return warp_max_nonneg_i64(v);
#pragma unroll
        for (int o = GL / 2; o; o >>= 1) { const i64 x = __shfl_xor_sync(FULL, v, o); v = x > v ? x : v; }
        return v;
    }
    // Sum of a in the even lanes, of b in the odd ones.
    template <class T> __device__ static __forceinline__ T pair_sum(T a, T b, bool odd)
    {
        T v = (odd ? b : a) + swap(odd ? a : b);
#pragma unroll
        for (int o = 2; o < GL; o <<= 1) v += __shfl_xor_sync(FULL, v, o);
        return v;
    }
    __device__ static __forceinline__ int sum(int v)
    {
        if (GL == 32) return __reduce_add_sync(FULL, v);
#pragma unroll
        for (int o = GL / 2; o; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
        return v;
    }
    __device__ static __forceinline__ i64 sum(i64 v)
    {
#pragma unroll
        for (int o = GL / 2; o; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
        return v;
    }
};

// For every lane named in `who`: busiest load of its layer `layer_own` of row-shard rg_own once sample mi_own has left it
// (sgn = -1) or joined it (+1) and mi2_own (>= 0: a swap) the other way round, added up from the samples that sit
// there; the other lanes keep `mine`.  The samples are first collected in `list`
// (its last entry is the counter), then sixteen of their counts are in flight at a time, a rank per lane: nearly always a
// single layer is asked for, of a row-shard of a hundred short samples.  Kept small: a form with the collection
// unrolled took 110000 cycles a call on wide and slowed the other chains of the SM threefold (instruction fetches).
static __device__ __noinline__ int rp_row_exact_max(int N, int P, int LP, const int *__restrict__ q, const unsigned short *cells_own,
                                                    const unsigned short *rg_of, int *list, int rg_own, unsigned who, int layer_own, int mi_own,
                                                    int mi2_own, int sgn, int mine)
{
    const int lane = threadIdx.x & 31;
    int *count = list + ROW_LIST;
#pragma unroll 1
    for (; who; who &= who - 1) {
        const int at = __ffs(who) - 1;
        const unsigned short *cells = (const unsigned short *)__shfl_sync(0xffffffffu, (unsigned long long)cells_own, at);
        const int rg = __shfl_sync(0xffffffffu, rg_own, at), mi = __shfl_sync(0xffffffffu, mi_own, at), mi2 = __shfl_sync(0xffffffffu, mi2_own, at);
        const int *layer = q + (size_t)__shfl_sync(0xffffffffu, layer_own, at) * P;
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

// Shared memory of a chain.  Its first cs_bytes, JA to Sc, are what members hand on from level to level.
struct RowChain {
    char *base;
    longlong2 *JA;               // cost and attention part of a row-shard
    i64 *E;                      // its busiest loads
    u64 *Q;                      // squared lengths of a cell
    int2 *TC;                    // its tokens and samples
    i64 *U, *Sc, *slack;         // work of a shard; S0, S1, S2, energy; see RowArgs
    int2 *ws;                    // !CHIP: slice of each row-shard, and the one its next rewrite goes to
    unsigned short *cell, *snap; // CHIP: assignment, trajectory-best layout, rank loads
    int4 *W;
    longlong2 *top;              // shards of several slots: largest and second largest cost of each (row-shard, stage),
    unsigned short *topc;        // the cell of the largest,
    i64 *att;                    // and the attention key of a cell
};

__device__ __forceinline__ RowChain row_chain(const RpDims &dm, const RowArgs &X, char *sm_chain, int w)
{
    RowChain c;
    char *sm = sm_chain + (size_t)w * X.chain_bytes;
    c.base = sm;
    c.JA = (longlong2 *)sm;
    c.E = (i64 *)(sm + X.off_E);
    c.Q = (u64 *)(sm + X.off_Q);
    c.TC = (int2 *)(sm + X.off_TC);
    c.U = (i64 *)(sm + X.off_U);
    c.Sc = (i64 *)(sm + X.off_S);
    c.slack = (i64 *)(sm + X.off_F);
    c.ws = (int2 *)(sm + X.off_ws);
    c.cell = (unsigned short *)(sm + X.off_cell);
    c.snap = (unsigned short *)(sm + X.off_snap);
    c.W = (int4 *)(sm + X.off_W);
    c.top = (longlong2 *)(sm + X.off_top);
    c.att = (i64 *)(sm + X.off_top + (size_t)16 * dm.RG * dm.S);
    c.topc = (unsigned short *)(sm + X.off_top + (size_t)16 * dm.RG * dm.S + (size_t)8 * dm.K);
    return c;
}

// A member's state between the population's blobs (an array for each quantity) and the chain's records, by threads t of n.
__device__ __forceinline__ void row_state_in(const RpDims &dm, const RpBlob &bl, const RowChain &c, const char *b, int t, int n)
{
    const i64 *E = (const i64 *)(b + bl.off_Esum), *Af = (const i64 *)(b + bl.off_Afx), *J = (const i64 *)(b + bl.off_Jfx);
#pragma unroll 2
    for (int x = t; x < dm.RG; x += n) { c.JA[x] = make_longlong2(__ldg(J + x), __ldg(Af + x)); c.E[x] = __ldg(E + x); }
    const u64 *Q = (const u64 *)(b + bl.off_Q);
    const int *T = (const int *)(b + bl.off_T), *m = (const int *)(b + bl.off_cnt);
#pragma unroll 2
    for (int x = t; x < dm.K; x += n) { c.Q[x] = __ldg(Q + x); c.TC[x] = make_int2(__ldg(T + x), __ldg(m + x)); }
    for (int x = t; x < dm.G; x += n) c.U[x] = __ldg((const i64 *)(b + bl.off_U) + x);
    for (int x = t; x < 4; x += n) c.Sc[x] = __ldg((const i64 *)(b + bl.off_S) + x);
}
__device__ __forceinline__ void row_state_out(const RpDims &dm, const RpBlob &bl, const RowChain &c, char *b, int t, int n)
{
    for (int x = t; x < dm.RG; x += n) {
        const longlong2 v = c.JA[x];
        ((i64 *)(b + bl.off_Jfx))[x] = v.x; ((i64 *)(b + bl.off_Afx))[x] = v.y; ((i64 *)(b + bl.off_Esum))[x] = c.E[x];
    }
    for (int x = t; x < dm.K; x += n) {
        const int2 v = c.TC[x];
        ((u64 *)(b + bl.off_Q))[x] = c.Q[x]; ((int *)(b + bl.off_T))[x] = v.x; ((int *)(b + bl.off_cnt))[x] = v.y;
    }
    for (int x = t; x < dm.G; x += n) ((i64 *)(b + bl.off_U))[x] = c.U[x];
    for (int x = t; x < 4; x += n) ((i64 *)(b + bl.off_S))[x] = c.Sc[x];
}
// The records as they are (their size is a multiple of 8 bytes; a blob has room for as many).
__device__ __forceinline__ void row_records_out(const RowArgs &X, const RowChain &c, char *b, int t, int n)
{
    const int n16 = X.cs_bytes >> 4;
    for (int x = t; x < n16; x += n) ((int4 *)b)[x] = ((const int4 *)c.base)[x];
    if ((X.cs_bytes & 8) && t == 0) ((i64 *)b)[2 * n16] = ((const i64 *)c.base)[2 * n16];
}

// Largest and second largest cost of stage s over the slots of row-shard rg (row of cell `rb`, shard g).
__device__ __forceinline__ void row_top_stage(const RpDims &dm, const RowChain &ch, const int *dpl, const int *dpo, int rb, int g, int rg, int s)
{
    const i64 ca = dm.ahat[s] * dm.C, cb = dm.bhat[s];
    i64 v1 = -1, v2 = 0;
    int c1 = 0;
#pragma unroll 4
    for (int x = dpo[g]; x < dpo[g + 1]; ++x) {
        const int c = rb + dpl[x];
        const i64 v = ca * ch.TC[c].x + cb * (i64)ch.Q[c];
        if (v > v1) { v2 = v1 < 0 ? 0 : v1; v1 = v; c1 = c; }
        else if (v > v2) v2 = v;
    }
    ch.top[rg * dm.S + s] = make_longlong2(v1, v2); ch.topc[rg * dm.S + s] = (unsigned short)c1;
}

// Attention cost of a row-shard (first cell of its row `rb`, shard g) with the statistics of two of its cells replaced.
__device__ __forceinline__ i64 row_attention(const RpDims &dm, const RowChain &ch, const int *dpl, const int *dpo, int rb, int g,
                                             int c_a, i64 Ta, i64 Qa, int c_b, i64 Tb, i64 Qb)
{
    i64 sum = 0;
    for (int s = 0; s < dm.S; ++s) {
        i64 worst = 0;
        const i64 ca = dm.ahat[s] * dm.C, cb = dm.bhat[s];
        for (int x = dpo[g]; x < dpo[g + 1]; ++x) {
            const int c = rb + dpl[x];
            i64 T = ch.TC[c].x, Q = (i64)ch.Q[c];
            if (c == c_a) { T = Ta; Q = Qa; }
            if (c == c_b) { T = Tb; Q = Qb; }
            const i64 v = ca * T + cb * Q;
            worst = v > worst ? v : worst;
        }
        sum += worst;
    }
    return sum;
}

__device__ __forceinline__ void row_copy16(int4 *to, const int4 *from)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(to)), "l"(from) : "memory");
}

__device__ __forceinline__ i64 row_energy(i64 s0, i64 s1, i64 s2)       // rp_energy of non-negative scores
{
    return s0 + (i64)((u64)s1 / 1000000ull) + (i64)((u64)s2 / 1000000000ull);
}

// The level barrier of up to 32 members by one warp, a member a lane: incumbent (inc, *win = its slot or -1), then, unless this
// was the last level, ancestors of members m0 .. m1-1.  No CTA-wide barrier between its parts (8 % of a tiny plan); with
// eight members a lane one warp takes longer than eight do with their barriers (7 % of medium's).
__device__ __forceinline__ void row_barrier_warp(const AnnealArgs &A, int P, const u64 *eL, const i64 *bestL, bool last, u64 cq, u32 resample_x,
                                                 int m0, int m1, i64 *inc, int *win, int *anc, int lane)
{
    const u64 r = lane < P ? __ldcg(eL + lane) : 0x7fffffffffffffffull;
    const i64 e[1] = { (i64)(r & ~(1ull << 63)) };
    // (fetched beside the energy, whether its trajectory best beats the incumbent or not)
    const i64 b0 = lane < P ? __ldcg(bestL + 3 * lane) : 0, b1 = lane < P ? __ldcg(bestL + 3 * lane + 1) : 0, b2 = lane < P ? __ldcg(bestL + 3 * lane + 2) : 0;
    const int bj = r >> 63 ? lane : 0x7fffffff;
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

// Warps per SM the register budget is set for.  Registers come in quarters of an SM: 12 leaves 168 a thread and keeps 12 warps
// resident, 13 to 16 leave 128 and keep 16.  Which is better depends on how many warps there are; at 12 / 14 / 16, plans in ms: heavy
// (8192 members, two to a warp) 61.6 / 59.4 / 59.5, 4096 members of 16 layers of 32 ranks (two to a warp) 4.15 / 3.41 / 3.44; where 12 a
// SM hold them all (ROOMY), 1776 members with a warp each, heavy's window at 20 levels of 200 steps 5.95 / 6.55 / 6.82, 1184 5.28 / 5.99,
// 3000 members of 16 layers, two to a warp, 2.83 / 3.00.  (Asked for 16 the compiler orders the code another way and spills less, 24
// bytes for 40, to no gain.)  More chunks, or shards of several slots, need the registers of 12.
#define ROW_WARPS_PER_SM(GL, LPL, CPL, IDENT) ((GL) == 16 || ((LPL) * (CPL) == 1 && (IDENT)) ? 14 : 12)

// GL lanes run a chain, LPL layers per lane, CPL 16-byte chunks per layer (X.cpl <= CPL of them in use).  IDENT: slot d is shard d.
// SPLIT (X.cpl = 2 or 4): the row's chunks are dealt out to the lanes in turn instead, CPL of them to a lane, and a layer's maximum
// meets in shuffles: a load touches consecutive bytes, and no lane is idle for want of layers.  Whole layers of four chunks put the
// lanes of a load 64 bytes apart, twelve lines for 24 layers, eight stores 440 cycles (large 2662 us, dealt out 2499; with candidates
// 3023 and 2999).  With the rank loads on chip only the demand rows would gain, and the shuffles cost more (3 % of two shards).
template <int GL, int LPL, int CPL, bool SPLIT, bool CHIP, bool COMP, bool IDENT, bool ROOMY>
__global__ void __launch_bounds__(CHIP ? ROW_THREADS : 32, CHIP ? 1 : ROOMY ? 12 : ROW_WARPS_PER_SM(GL, LPL, CPL, IDENT))
k_anneal_row(const AnnealArgs A, const RowArgs X)
{
    constexpr int NCH = SPLIT ? CPL : LPL * CPL;
    constexpr bool ONE = GL == 32;                                       // a warp runs one chain: its branches are the warp's
    using G = Lanes<GL>;
    const RpDims &dm = A.dm;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, lg = lane & (GL - 1);
    const unsigned gmask = G::mask(lane);
    constexpr int NT = CHIP ? ROW_THREADS : 32;
    const int cw = CHIP ? X.cw : 32 / GL;                                // chains of this CTA: (CHIP) warps 0 .. cw-1; the others
    const int cx = CHIP ? warp : lane / GL;                              // help to move states and at the level barrier
    const int j = blockIdx.x * cw + cx;
    const int P = A.Ppop;
    const bool live = CHIP ? (warp < cw && j < P) : (ONE || j < P);
    char *sm_cta = (char *)smraw;                                        // tables shared by the CTA's chains
    char *sm_chain = (char *)smraw + X.off_chain;
    const RowChain ch = row_chain(dm, X, sm_chain, CHIP ? min(warp, cw - 1) : cx);
    const int *dpl = (const int *)(sm_cta + A.sl.off_dpl);
    const int *dpo = (const int *)(sm_cta + A.sl.off_dpo);
    const char *sm_tab = sm_cta + X.off_tab - A.sl.off_rg;
    const unsigned short *rg_of = (const unsigned short *)(sm_tab + A.sl.off_rg);
    const unsigned short *g_of = (const unsigned short *)(sm_tab + A.sl.off_g);
    const unsigned short *rowbase = (const unsigned short *)(sm_tab + A.sl.off_row);

    // The first steps before the launch before has ended.  With shards of several slots (whose loop is 2 to 4 % slower with a batch of steps
    // that come from elsewhere: 2183 members of one shard, 27 layers of 8 ranks, 406 steps a level, 19.1 ms without, 19.9 with) only where it starts early:
    // their ROOMY instances do without.
    constexpr bool AHEAD = ONE && !CHIP && (IDENT || !ROOMY);
    if (!CHIP && !AHEAD) {
        rp_wait_for_launch_before();
        if (__ldcg(&A.status[RP_SW_TIMEOUT])) return;                    // the call has failed already: nothing to do
    }
    const int L = dm.L, cpl = CPL == 1 && !SPLIT ? 1 : X.cpl, rc = L * cpl;        // 16-byte chunks per layer and per row
    const int rot = CHIP && CPL > 1 && (cpl & (cpl - 1)) == 0 ? cpl - 1 : 0;     // lanes start at different chunks: fewer bank conflicts
    // 16-byte chunk u of this lane
    auto chunk = [&](int u, bool &on) {
        if (SPLIT) { const int c = lane + 32 * u; on = c < rc; return c; }
        const int ly = lg + GL * (u / CPL), k = u % CPL;
        on = ly < L && (CPL == 1 || k < cpl);
        return ly * cpl + (rot ? ((k + lane) & rot) : k);
    };
    const bool sum32 = dm.sum32;
    const i64 aC = dm.asum * dm.C, bS = dm.bsum;
    const float aCf = (float)aC, bSf = (float)bS, ECf = (float)dm.EC;
    const int4 *qr = (const int4 *)X.qr;
    unsigned short *cells = CHIP ? ch.cell : (unsigned short *)(A.blob_dst + (size_t)(live ? j : 0) * A.bl.bytes + A.bl.off_cell);
    const int n4 = dm.N >> 2;
    const StepRec *recs = (const StepRec *)(ch.base + X.off_recs);

    // ---- prologue: the static tables, the first steps (a launch per level: they depend on nothing the launch before leaves behind) and the
    // ancestor's terminal state -----------------------------------------------------------------
    StepX ahead;
    {
        const int nd = A.sl.off_t >> 2, nc = (A.sl.bytes - A.sl.off_rg) >> 2;
        for (int x = tid; x < nd; x += NT) ((int *)sm_cta)[x] = __ldg((const int *)A.static_blk + x);
        for (int x = tid; x < nc; x += NT) ((int *)(sm_cta + X.off_tab))[x] = __ldg((const int *)(A.static_blk + A.sl.off_rg) + x);
    }
    if (CHIP && X.off_tf) for (int x = tid; x < dm.N; x += NT) ((int2 *)(sm_cta + X.off_tf))[x] = __ldg(X.tf + x);
    if (AHEAD) {
        const StepRec r = rp_make_step_rec(A, A.level, A.tau, (u32)lane, (u32)j);
        const bool rl = r.flags & 1u;
        ahead.i[0] = r.i0; ahead.i[1] = r.i1; ahead.i[2] = rl ? (int)(r.i2 | 0x80000000u) : r.i2; ahead.i[3] = rl ? (int)(r.i3 | 0x80000000u) : r.i3;
        ahead.bz = r.bz; ahead.thr = r.flags & 4u ? 1ull << 63 : r.thr;
        ahead.thrf = r.flags & 4u ? __int_as_float(0x7f800000) : (float)r.thr * (0x1p-32f * (1.f + 0x1p-20f));
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const int2 v = x < 2 || !rl ? __ldg(X.tf + ahead.i[x]) : make_int2(0, 0);
            ahead.t[x] = v.x; ahead.f[x] = v.y;
        }
        rp_wait_for_launch_before();
        if (__ldcg(&A.status[RP_SW_TIMEOUT])) return;                    // the call has failed already: nothing to do
    }
    int half_w = 0, inc_slot = -1;
    __shared__ i64 inc_s[3];
    __shared__ int failed_s;
    if (!CHIP && live) {
        const int src = min(max(A.anc[j], 0), P - 1);
        const char *bsrc = A.blob_src + (size_t)src * A.bl.bytes;
        if (A.level == 0) row_state_in(dm, A.bl, ch, bsrc, lg, GL);
        else {
#pragma unroll 8
            for (int x = lg; x < (X.cs_bytes + 15) >> 4; x += GL) ((int4 *)ch.base)[x] = __ldg((const int4 *)bsrc + x);
        }
        const i64 *fs = X.F_src + (size_t)src * dm.RG;
        const int *ts = (const int *)(bsrc + A.bl.off_wtab);
        // A slice that only this member holds when the level starts is rewritten in place; a shared
        // one is left at its first rewrite for this chain's spare slice of that row-shard (entry
        // j*RG + rg of the free list, which holds at least RG slices per member).  (List and holders, like the ancestors, may be written while
        // this launch is there already: no __ldg, but plain loads, which stay behind the wait; __ldcg took 2 % of large.  The states are of the
        // launch before that one.)
        const int n_free = A.wfree_head[1];
#pragma unroll 4
        for (int rg = lg; rg < dm.RG; rg += GL) {
            ch.slack[rg] = __ldg(fs + rg);
            const int s = __ldg(ts + rg);
            const size_t at = (size_t)j * dm.RG + rg;
            const int sp = at < (size_t)n_free ? A.wfree[at] : -2;
            ch.ws[rg] = make_int2(s, A.wref[s] == 1 ? s : sp);
        }
        const unsigned short *cs = (const unsigned short *)(bsrc + A.bl.off_cell);        // 8-byte aligned
#pragma unroll 8
        for (int x = lg; x < n4; x += GL) ((uint2 *)cells)[x] = __ldg((const uint2 *)cs + x);
        for (int i = (n4 << 2) + lg; i < dm.N; i += GL) cells[i] = __ldg(cs + i);
    }
    if (CHIP) {
        for (int w = 0; w < cw; ++w) {
            const int jj = blockIdx.x * cw + w;
            if (jj >= P) break;
            const RowChain c = row_chain(dm, X, sm_chain, w);
            const int src = min(max(A.anc[jj], 0), P - 1);
            const char *bsrc = A.blob_src + (size_t)src * A.bl.bytes;
            row_state_in(dm, A.bl, c, bsrc, tid, NT);
            const i64 *fs = X.F_src + (size_t)src * dm.RG;
            for (int rg = tid; rg < dm.RG; rg += NT) c.slack[rg] = __ldg(fs + rg);
            const unsigned short *cs = (const unsigned short *)(bsrc + A.bl.off_cell);
            for (int x = tid; x < n4; x += NT) ((uint2 *)c.cell)[x] = __ldg((const uint2 *)cs + x);
            for (int i = (n4 << 2) + tid; i < dm.N; i += NT) c.cell[i] = __ldg(cs + i);
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
        if (tid < 3) inc_s[tid] = A.lo.inc_score[tid];
        __syncthreads();
        // every chain of the launch has read its start state (the pool is about to be written) from here on
        if (tid == 0) { __threadfence(); atomicAdd(A.lo.done, 1); }
        if (A.stall_test && blockIdx.x == 0) {       // inspection hook: chain 0 waits for an arrival that never comes
            if (tid == 0 && !rp_wait_count(A.lo.done, 0x7fffffff, A)) atomicExch(&A.status[RP_SW_TIMEOUT], 1);
            return;
        }
    } else if (A.stall_test && blockIdx.x == 0) {
        // inspection hook: a bounded wait on a barrier phase that nothing completes
        u64 *mbar = (u64 *)(sm_chain + X.off_mbar);
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
    int n_feas = 0, n_acc = 0, n_imp = 0;       // feasible moves this lane proposed; accepted and improving ones (the same in every lane)
    int n_rows = 0;                             // rows and slices they name, per lane (six a step at most)
    i64 S0 = 0, S1 = 0, S2 = 0, Ecur = 0, B0 = 0, B1 = 0, B2 = 0;        // score and energy; trajectory best
    u64 dig = 0;
    int best_step = 0, best_nlog = 0;
    bool has_snap = false, pend = false;        // CHIP: ch.snap holds the best layout; the state at hand is the best, not kept yet
    if (CHIP ? live : true) {
        if (!IDENT && live) {
            for (int c = lg; c < dm.K; c += GL) ch.att[c] = aC * ch.TC[c].x + bS * (i64)ch.Q[c];
            for (int x = lg; x < dm.RG * dm.S; x += GL) {
                const int rg = x / dm.S;
                row_top_stage(dm, ch, dpl, dpo, rg / dm.G * dm.D, rg % dm.G, rg, x % dm.S);
            }
        }
        if (live) { B0 = S0 = ch.Sc[0]; B1 = S1 = ch.Sc[1]; B2 = S2 = ch.Sc[2]; Ecur = ch.Sc[3]; }
        __syncwarp();
        int kb = -GL, nb = 0, pos = 0;          // steps kb .. kb+nb-1 are in the lanes, those before pos decided
        bool done = !live, need = false;
        unsigned pmask = 0;
        StepX sr;
        if (AHEAD) {
            sr = ahead;
#pragma unroll
            for (int x = 0; x < 4; ++x) sr.c[x] = 0;
        } else {
            sr.bz = 0; sr.thr = 0; sr.thrf = 0.f;
#pragma unroll
            for (int x = 0; x < 4; ++x) { sr.i[x] = 0; sr.c[x] = 0; sr.t[x] = 0; sr.f[x] = 0; }
        }
        bool ok = false;
        int mi = 0, mi2 = -1, ti = 0, t2 = 0, df = 0;
        u32 p1 = 0, p2 = 0;
        i64 dA1 = 0, dA2 = 0;                   // (shards of several slots)
        for (;;) {
            bool fresh = false;
            if (pos >= nb && !done) {
                kb += GL;
                done = kb >= A.steps;
                fresh = !done;
                if (!ONE && done) { nb = 0; ok = false; }
            }
            if (ONE ? done : __all_sync(G::FULL, done)) break;
            // ---- the next GL steps, one per lane: random words, candidate cells, lengths, fixed-rank demands ----
            if (ONE ? fresh : __any_sync(G::FULL, fresh)) {
                if (!ONE) {
                    // 32 steps of a chain at a time by all lanes, kept until their turn comes
                    unsigned who = __ballot_sync(G::FULL, fresh && (kb & 31) == 0 && lg == 0);
                    __syncwarp();
                    for (; who; who &= who - 1) {
                        const int at = __ffs(who) - 1, k = __shfl_sync(G::FULL, kb, at) + lane, jj = __shfl_sync(G::FULL, j, at);
                        ((StepRec *)(sm_chain + (size_t)(at / GL) * X.chain_bytes + X.off_recs))[lane] = rp_make_step_rec(A, level, tau, (u32)k, (u32)jj);
                    }
                    __syncwarp();
                }
                if (fresh) {
                    nb = min(GL, A.steps - kb); pos = 0;
                    if (lg < nb) {
                        if (AHEAD && kb == 0) {                         // (all but the cells is known)
#pragma unroll
                            for (int x = 0; x < 4; ++x) sr.c[x] = x < 2 || sr.i[x] >= 0 ? (u32)__ldcg(cells + sr.i[x]) : (u32)sr.i[x] & 0x7fffffffu;
                        } else {
                        StepRec r;
                        const bool kept = !ONE || (CHIP && kb + lane < X.recs);
                        if (kept) r = recs[ONE ? (ln & 1) * X.recs + kb + lane : (kb & 16) + lg];
                        else r = rp_step_picks(A, level, (u32)(kb + lane), (u32)j);
                        const bool rl = r.flags & 1u;
                        sr.i[0] = r.i0; sr.i[1] = r.i1; sr.i[2] = r.i2; sr.i[3] = r.i3;
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            u32 c = (u32)sr.i[x];
                            int2 v = make_int2(0, 0);
                            if (x < 2 || !rl) {
                                c = CHIP ? (u32)cells[sr.i[x]] : (u32)__ldcg(cells + sr.i[x]);
                                v = CHIP && X.off_tf ? ((const int2 *)(sm_cta + X.off_tf))[sr.i[x]] : __ldg(X.tf + sr.i[x]);
                            }
                            sr.c[x] = c; sr.t[x] = v.x; sr.f[x] = v.y;
                        }
                        if (!kept) rp_step_threshold(A, level, tau, (u32)(kb + lane), (u32)j, r);
                        sr.bz = r.bz; sr.thr = r.flags & 4u ? 1ull << 63 : r.thr;
                        sr.thrf = r.flags & 4u ? __int_as_float(0x7f800000) : (float)r.thr * (0x1p-32f * (1.f + 0x1p-20f));
                        if (rl) { sr.i[2] = (int)0x80000000; sr.i[3] = (int)0x80000000; }
                        }
#pragma unroll
                        for (int x = 0; x < 4; ++x) sr.c[x] |= (u32)(IDENT ? g_of[sr.c[x]] : rg_of[sr.c[x]]) << 16;
                    }
                    need = true;
                }
            }
            // ---- proposals of steps kb+pos .. kb+nb-1 against the current state, one per lane: GuidedProposal and
            // feasibility (the rule of rp_propose), then the rejection by the fixed ranks ----------------------------
            if (ONE ? need : true) {
                bool pass = false;
                ok = false;
                if (lg >= pos && lg < nb) {
                    const u32 ca = sr.c[0], cb = sr.c[1], xa = sr.c[2], xb = sr.c[3];
                    const int ra = IDENT ? ca & 0xffffu : ca >> 16, rb = IDENT ? cb & 0xffffu : cb >> 16;
                    const int rx = IDENT ? xa & 0xffffu : xa >> 16, ry = IDENT ? xb & 0xffffu : xb >> 16;
                    const longlong2 Ka = ch.JA[ra];
                    const u64 Ja = (u64)Ka.x, Aa = (u64)Ka.y;
                    // bz * Ja < Aa * 2^32  <=>  floor(bz * Ja / 2^32) < Aa
                    const u64 pr = (Ja >> 32) * sr.bz + (((Ja & 0xffffffffull) * sr.bz) >> 32);
                    const bool by_a = pr < Aa;
                    bool src_b, dst_b;
                    if (IDENT) {
                        const longlong2 Kb = ch.JA[rb], Kx = ch.JA[rx], Ky = ch.JA[ry];
                        src_b = by_a ? Kb.y > Ka.y : Kb.x > Ka.x;
                        dst_b = by_a ? Ky.y < Kx.y : Ky.x < Kx.x;
                    } else {
                        const i64 jb = ch.JA[rb].x, jx = ch.JA[rx].x, jy = ch.JA[ry].x;
                        const i64 aa = ch.att[ca & 0xffffu], ab = ch.att[cb & 0xffffu], ax = ch.att[xa & 0xffffu], ay = ch.att[xb & 0xffffu];
                        src_b = by_a ? ab > aa : jb > Ka.x;
                        dst_b = by_a ? ay < ax : jy < jx;
                    }
                    mi = src_b ? sr.i[1] : sr.i[0];
                    p1 = src_b ? cb : ca;
                    ti = src_b ? sr.t[1] : sr.t[0];
                    p2 = dst_b ? xb : xa;
                    mi2 = dst_b ? sr.i[3] : sr.i[2];
                    t2 = dst_b ? sr.t[3] : sr.t[2];
                    df = (src_b ? sr.f[1] : sr.f[0]) - (dst_b ? sr.f[3] : sr.f[2]);
                    // (everything the score needs is loaded before feasibility is known)
                    const int c1 = p1 & 0xffffu, c2 = p2 & 0xffffu;
                    const int rg1 = IDENT ? c1 : p1 >> 16, rg2 = IDENT ? c2 : p2 >> 16;
                    const int g1 = IDENT ? p1 >> 16 : g_of[c1], g2 = IDENT ? p2 >> 16 : g_of[c2];
                    const int2 h1 = ch.TC[c1], h2 = ch.TC[c2];
                    const i64 k1 = ch.slack[rg1], k2 = ch.slack[rg2], U1o = ch.U[g1], U2o = ch.U[g2];
                    ok = c1 != c2 && h2.x - t2 + ti <= dm.C && h1.x - ti + t2 <= dm.C && (mi2 >= 0 || h1.y > 1);
                    const bool tw = IDENT || rg1 != rg2;
                    if (!IDENT && ok) {
                        const int Ta = h1.x - ti + t2, Tb = h2.x + ti - t2;
                        const i64 dq = (i64)t2 * t2 - (i64)ti * ti, Qa = (i64)ch.Q[c1] + dq, Qb = (i64)ch.Q[c2] - dq;
                        i64 A1 = 0, A2 = 0;
                        if (tw) {
                            for (int s = 0; s < dm.S; ++s) {
                                const i64 ca_ = dm.ahat[s] * dm.C, cb_ = dm.bhat[s];
                                const i64 va = ca_ * Ta + cb_ * Qa, vb = ca_ * Tb + cb_ * Qb;
                                const int x1 = rg1 * dm.S + s, x2 = rg2 * dm.S + s;
                                const longlong2 w1 = ch.top[x1], w2 = ch.top[x2];
                                const i64 o1 = ch.topc[x1] == c1 ? w1.y : w1.x, o2 = ch.topc[x2] == c2 ? w2.y : w2.x;
                                A1 += va > o1 ? va : o1; A2 += vb > o2 ? vb : o2;
                            }
                            dA2 = A2 - ch.JA[rg2].y;
                        } else A1 = row_attention(dm, ch, dpl, dpo, rowbase[c1], g1, c1, Ta, Qa, c2, Tb, Qb);
                        dA1 = A1 - ch.JA[rg1].y;
                    }
                    // Rejected for certain?  The busiest loads fall by at most what the samples put on the fixed ranks plus the
                    // slack (both cells in one row-shard: nothing changes), so x below is the least by which the largest shard
                    // cost can rise and x + 1e-6 * (J1 + J2) - 1e-9 * S2 (S2 <= S0 <= E) the least by which the energy can.  In single
                    // precision, of differences only: a dozen roundings of 2^-24 of the magnitudes in `mag`, allowed for by
                    // 2^-20 of them; what is not rejected here is decided by the exact score.
                    float k1f, k2f;
                    if (sum32) { k1f = (float)(int)k1; k2f = (float)(int)k2; } else { k1f = (float)k1; k2f = (float)k2; }
                    const float dff = (float)df;
                    const float a1 = IDENT ? (aCf + bSf * (float)(t2 + ti)) * (float)(t2 - ti) : (float)dA1, a2 = IDENT ? -a1 : (float)dA2;
                    const float v1 = (float)(U1o - S0), v2 = (float)(U2o - S0), Mf = (float)(Ecur > dm.SC ? Ecur : dm.SC);
                    const float J1 = a1 + (tw ? ECf * (-dff - k1f) : 0.f), J2 = tw ? a2 + ECf * (dff - k2f) : 0.f;
                    const float u1 = v1 + J1 + (g1 == g2 ? J2 : 0.f), u2 = g1 == g2 ? u1 : v2 + J2, x = fmaxf(u1, u2);
                    const float mag = fabsf(v1) + fabsf(v2) + fabsf(a1) + fabsf(a2) + ECf * (2.f * fabsf(dff) + k1f + k2f);
                    const float err = 8.f + 0x1p-20f * mag;
                    const float most = sr.thrf * Mf + 2.f;                   // accepted below (rounded up, see thrf)
                    pass = ok && !(x > err && x + 1e-6f * (J1 + J2) - 1.001e-9f * Mf - err >= most);
                }
                pmask = G::ballot(pass, lane);
                need = false;
            }
            const bool has = pmask != 0;
            const int ls = has ? __ffs(pmask) - 1 : 0;
            bool acc = false;
            if (ONE ? has : __any_sync(G::FULL, has)) {
                // ---- exact score of the next candidate -------------------------------------------------------
                const int wi = G::get(mi, ls), wi2 = G::get(mi2, ls);
                const u32 w1p = G::get(p1, ls), w2p = G::get(p2, ls);
                const int d1 = w1p & 0xffffu, d2 = w2p & 0xffffu;
                const int r1 = IDENT ? d1 : w1p >> 16, r2 = IDENT ? d2 : w2p >> 16;
                const bool touchW = IDENT || r1 != r2, swap = wi2 >= 0;
                // What the decision needs: even lanes look at the cell that gives (1), odd lanes at the one that takes (2).
                const bool second = lg & 1;
                const int mc = second ? d2 : d1, mr = second ? r2 : r1;
                int wti, wt2, mg;
                longlong2 old;
                i64 Uo, eo, sk, wb, dA;
                int2 tc;
                u64 Qo;
                auto look = [&]() {
                    wti = G::get(ti, ls); wt2 = G::get(t2, ls);
                    mg = IDENT ? (second ? w2p : w1p) >> 16 : g_of[mc];
                    old = ch.JA[mr]; Uo = ch.U[mg]; eo = ch.E[mr]; sk = ch.slack[mr]; tc = ch.TC[mc]; Qo = ch.Q[mc];
                    // accepted when the energy rises by less than wb (at least 1: never uphill by 0)
                    const u64 thr = G::get(sr.thr, ls), M = (u64)(Ecur > dm.SC ? Ecur : dm.SC);
                    const u64 bh = __umul64hi(thr, M), bl = thr * M;
                    wb = (i64)((bh << 32) | (bl >> 32));
                    wb = wb > 1 ? wb : 1;
                    if ((i64)thr < 0 || (bh >> 31)) wb = 0x7fffffffffffffffll;
                    if (IDENT) { dA = (aC + bS * (wt2 + wti)) * (wt2 - wti); if (second) dA = -dA; }
                    else { const i64 da1 = G::get(dA1, ls), da2 = G::get(dA2, ls); dA = second && touchW ? da2 : da1; }
                };
                int4 d[NCH], w1[NCH], w2[NCH];
                i64 Em = 0;                                  // busiest loads of the row-shard this lane looks at
                int2 s1 = make_int2(0, 0), s2 = s1;          // !CHIP: slices of the two row-shards
                if (ONE ? touchW : true) {
                    int4 q2[NCH];
                    if (!CHIP) { s1 = ch.ws[r1]; s2 = ch.ws[r2]; }
                    const int4 *qi = qr + (size_t)wi * rc, *qj = qr + (size_t)(swap ? wi2 : wi) * rc;
                    const int4 *W1 = CHIP ? ch.W + (size_t)r1 * rc : (const int4 *)(X.Wr + (size_t)s1.x * X.rlp);
                    const int4 *W2 = CHIP ? ch.W + (size_t)r2 * rc : (const int4 *)(X.Wr + (size_t)s2.x * X.rlp);
#pragma unroll
                    for (int u = 0; u < NCH; ++u) {
                        bool on;
                        const int c = chunk(u, on);
                        d[u] = q2[u] = w1[u] = w2[u] = make_int4(0, 0, 0, 0);
                        if (on && (ONE || (has && touchW))) {
                            d[u] = __ldg(qi + c);
                            if (swap) q2[u] = __ldg(qj + c);
                            w1[u] = W1[c]; w2[u] = W2[c];
                        }
                    }
                    // Under the rows' loads where all levels run in one launch (medium 818 us ahead of them, 807 here; two shards 828 and
                    // 816); behind the sums with one launch per level, whose chains share the SM's load path (wide and heavy a quarter slower
                    // ahead of the loads or here).
                    if (CHIP) look();
                    unsigned over = 0;                      // COMP: layers of this lane whose other ranks may be the busiest
                    constexpr int NM = SPLIT ? CPL : LPL, PER = NCH / NM;
                    int mx[NM][2];
#pragma unroll
                    for (int y = 0; y < NM; ++y) {
                        int m1 = 0, m2 = 0;
#pragma unroll
                        for (int k = 0; k < PER; ++k) {
                            const int u = y * PER + k;
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
                    if (SPLIT) {
#pragma unroll
                        for (int o = 1; o < 8; o <<= 1) {
                            if (o >= cpl) break;
#pragma unroll
                            for (int y = 0; y < NM; ++y) {
                                mx[y][0] = max(mx[y][0], __shfl_xor_sync(G::FULL, mx[y][0], o));
                                mx[y][1] = max(mx[y][1], __shfl_xor_sync(G::FULL, mx[y][1], o));
                            }
                        }
                        if (lane & (cpl - 1))                              // one lane of a layer has its share of the sum
#pragma unroll
                            for (int y = 0; y < NM; ++y) mx[y][0] = mx[y][1] = 0;
                    }
                    if (COMP && __any_sync(G::FULL, over != 0)) {
#pragma unroll
                        for (int y = 0; y < LPL; ++y)
#pragma unroll
                            for (int s = 0; s < 2; ++s) {
                                const unsigned who = __ballot_sync(G::FULL, (over >> (2 * y + s)) & 1u);
                                if (who) mx[y][s] = rp_row_exact_max(dm.N, dm.P, dm.LP, A.q, cells, rg_of, (int *)(sm_chain + X.off_list), s ? r2 : r1, who, lg + GL * y, wi, wi2, s ? 1 : -1, mx[y][s]);
                            }
                    }
                    if (sum32) {
                        int e1 = 0, e2 = 0;
#pragma unroll
                        for (int y = 0; y < NM; ++y) { e1 += mx[y][0]; e2 += mx[y][1]; }
                        if (ONE) {
                            const unsigned f1 = __reduce_add_sync(G::FULL, (unsigned)e1), f2 = __reduce_add_sync(G::FULL, (unsigned)e2);
                            Em = (i64)(second ? f2 : f1);
                        } else Em = (i64)G::pair_sum(e1, e2, second);
                    } else {
                        i64 e1 = 0, e2 = 0;
#pragma unroll
                        for (int y = 0; y < NM; ++y) { e1 += mx[y][0]; e2 += mx[y][1]; }
                        Em = G::pair_sum(e1, e2, second);
                    }
                }
                // ---- exact new score and the Metropolis decision: all lanes come to the same result (both cells in one
                // row-shard: both kinds of lanes see all of the change) --------------------------------------------
                if (!CHIP || !touchW) look();
                const i64 dJ = dA + (touchW ? dm.EC * (Em - eo) : 0), Jn = old.x + dJ;
                i64 Un = Uo + dJ;
                const i64 dJx = G::swap(dJ), dJo = touchW ? dJx : 0, Jx = G::swap(Jn);
                i64 Ux = G::swap(Un);
                if (IDENT ? (w1p >> 16) == (w2p >> 16) : mg == G::swap(mg)) { Un += dJo; Ux = Un; }
                const i64 n1 = S1 + dJ + dJo;
                i64 n0 = Un > Ux ? Un : Ux, n2 = Jn > Jx ? Jn : Jx;
                // where the previous maximum sat on a changed entry and fell, the maximum is searched anew, if the candidate is
                // not rejected with the smaller one already
                const bool fb0 = G::any(Uo >= S0, lane) && n0 < S0, fb2 = G::any(old.x >= S2, lane) && n2 < S2;
                if (!fb0 && n0 < S0) n0 = S0;
                if (!fb2 && n2 < S2) n2 = S2;
                i64 en = row_energy(n0, n1, n2);
                acc = has && (rp_lex_less(n0, n1, n2, S0, S1, S2) || en - Ecur < wb);
                const bool again = acc && (fb0 || fb2);
                if (ONE ? again : __any_sync(G::FULL, again)) {
                    i64 v0 = 0, v2 = 0;
                    if (ONE ? fb0 : __any_sync(G::FULL, again && fb0)) {
                        const int ga = G::get(mg, 0), gb = G::get(mg, 1);
                        for (int g = lg; g < dm.G; g += GL) if (g != ga && g != gb) { const i64 v = ch.U[g]; if (v > v0) v0 = v; }
                        v0 = G::max_nonneg(v0);
                    }
                    if (ONE ? fb2 : __any_sync(G::FULL, again && fb2)) {
                        for (int rg = lg; rg < dm.RG; rg += GL) if (rg != r1 && rg != r2) { const i64 v = ch.JA[rg].x; if (v > v2) v2 = v; }
                        v2 = G::max_nonneg(v2);
                    }
                    if (again) {
                        if (fb0 && v0 > n0) n0 = v0;
                        if (fb2 && v2 > n2) n2 = v2;
                        en = row_energy(n0, n1, n2);
                        acc = rp_lex_less(n0, n1, n2, S0, S1, S2) || en - Ecur < wb;
                    }
                }
                // ---- commit -----------------------------------------------------------------------------------
                const int wdf = G::get(df, ls);
                if (acc) {
                    if (touchW) {
                        // Where the two rewritten slices go: in place when the slice is this chain's own, else to the spare
                        // slice of that row-shard, which then is its own.
                        if (!CHIP) {
                            if (s1.y < 0 || s2.y < 0) {              // cannot happen: the list has a spare per row-shard
                                if (lg == 0) atomicExch(&A.status[RP_SW_POOL], 1);
                                if (s1.y < 0) s1.y = s1.x;
                                if (s2.y < 0) s2.y = s2.x;
                            }
                            if (lg < 2) ch.ws[mr] = second ? make_int2(s2.y, s2.y) : make_int2(s1.y, s1.y);
                        }
                        int4 *W1 = CHIP ? ch.W + (size_t)r1 * rc : (int4 *)(X.Wr + (size_t)s1.y * X.rlp);
                        int4 *W2 = CHIP ? ch.W + (size_t)r2 * rc : (int4 *)(X.Wr + (size_t)s2.y * X.rlp);
#pragma unroll
                        for (int u = 0; u < NCH; ++u) {
                            bool on;
                            const int c = chunk(u, on);
                            if (on) { W1[c] = w1[u]; W2[c] = w2[u]; }
                        }
                        if (lg == 0) n_rows += 2;
                    }
                    const bool imp = rp_lex_less(n0, n1, n2, B0, B1, B2);
                    if (CHIP && pend && !imp) {
                        // the trajectory best, about to be left, beats the incumbent of the level's start: keep its layout
                        for (int x = lane; x < (dm.N + 3) >> 2; x += 32) ((uint2 *)ch.snap)[x] = ((const uint2 *)ch.cell)[x];
                        has_snap = true; pend = false;
                        __syncwarp();
                    }
                    const u32 other = swap ? (u32)wi2 : (u32)d2;
                    if (lg < 2) {
                        const int up = second ? 1 : -1, dt = second ? wti - wt2 : wt2 - wti;
                        const i64 dq = (i64)wt2 * wt2 - (i64)wti * wti;
                        if (!second || swap) cells[second ? wi2 : wi] = (unsigned short)(second ? d1 : d2);
                        ch.TC[mc] = make_int2(tc.x + dt, swap ? tc.y : tc.y + up);
                        ch.Q[mc] = second ? Qo - (u64)dq : Qo + (u64)dq;
                        ch.JA[mr] = make_longlong2(Jn, old.y + dA);
                        ch.U[mg] = Un;
                        if (touchW) { ch.slack[mr] = sk + Em - eo + (second ? -wdf : wdf); ch.E[mr] = Em; }
                        if (!IDENT) { const i64 da = (aC + bS * (wt2 + wti)) * (wt2 - wti); ch.att[mc] += second ? -da : da; }
                        if (!CHIP && lg == 0 && n_acc < A.log_cap) A.log[(size_t)j * A.log_cap + n_acc] = make_uint2((u32)wi, other | (swap ? 0u : 0x80000000u));
                    }
                    n_acc += 1;
                    S0 = n0; S1 = n1; S2 = n2; Ecur = en;
                    if (A.lo.tr_digest) dig = (dig ^ (((u64)(swap ? 0 : 1) << 63) ^ ((u64)(u32)(kb + ls) << 40) ^ ((u64)(u32)wi << 20) ^ (u64)other)) * 0x100000001B3ull;
                    if (imp) {
                        B0 = n0; B1 = n1; B2 = n2;
                        best_step = kb + ls + 1; best_nlog = n_acc;
                        n_imp += 1;
                        if (CHIP) pend = pend || rp_lex_less(n0, n1, n2, inc_s[0], inc_s[1], inc_s[2]);
                    }
                    // the cached cells of the steps still to come follow the move (a relocation's targets are no sample's cells)
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        if (sr.i[x] == wi) sr.c[x] = w2p;
                        if (swap && sr.i[x] == wi2) sr.c[x] = w1p;          // (wi2 != wi, their cells differ)
                    }
                    __syncwarp(gmask);                              // the updates are visible
                    if (!IDENT && lg < 2 * dm.S) {
                        const bool b = lg >= dm.S;
                        const int c = b ? d2 : d1;
                        row_top_stage(dm, ch, dpl, dpo, rowbase[c], g_of[c], b ? r2 : r1, lg - (b ? dm.S : 0));
                    }
                    if (!IDENT) __syncwarp(gmask);
                }
            }
            const int upto = has ? ls : GL - 1;
            if (ok && lg >= pos && lg <= upto) { n_feas += 1; if (IDENT || (p1 >> 16) != (p2 >> 16)) n_rows += mi2 >= 0 ? 4 : 3; }
            pos = upto + 1;
            need = acc;
            pmask = has && !acc ? pmask & (pmask - 1) : 0;
        }
        if (live && lg == 0) { ch.Sc[0] = S0; ch.Sc[1] = S1; ch.Sc[2] = S2; ch.Sc[3] = Ecur; }
        __syncwarp();
    } else if (CHIP && warp >= cw && !last) make_recs(ln + 1, cw, NT / 32 - cw);

    // ---- epilogue of the level: the chain's report and terminal state ------------------------------
    const size_t rep = CHIP ? (size_t)(ln & 1) * P : 0;     // CHIP: two sets of reports taken in turn (a chain that
                                                            // runs ahead must not overwrite what a slower one still reads)
    i64 rows_all = 0;
    if (CHIP ? live : true) {
        n_feas = G::sum(n_feas);
        rows_all = G::sum((i64)n_rows);
    }
    if (live && lg == 0) {
        if (CHIP) {
            // what the level barrier reads first: the energy, and in its top bit whether the trajectory best beats the incumbent
            const bool beats = rp_lex_less(B0, B1, B2, inc_s[0], inc_s[1], inc_s[2]);
            A.lo.F[rep + j] = (u64)Ecur | (beats ? 1ull << 63 : 0ull);
        }
        if (!CHIP || A.lo.tr_term) { A.term[3 * (rep + j)] = S0; A.term[3 * (rep + j) + 1] = S1; A.term[3 * (rep + j) + 2] = S2; }
        A.best[3 * (rep + j)] = B0; A.best[3 * (rep + j) + 1] = B1; A.best[3 * (rep + j) + 2] = B2;
        if (!CHIP || A.lo.tr_term) { A.best_step[rep + j] = best_step; A.digest[rep + j] = dig; }
        if (!CHIP) A.best_nlog[j] = best_nlog;
        if (!CHIP && !A.last) { A.lo.F[j] = (u64)Ecur; atomicMin(A.lo.F + 2 * (size_t)P, (u64)Ecur); }
        sum_feas += n_feas; sum_acc += n_acc; sum_imp += n_imp; sum_rows += rows_all;
        if (!CHIP || last) {
            atomicAdd((u64 *)&A.counters[0], (u64)A.steps * n_levels);
            atomicAdd((u64 *)&A.counters[1], (u64)sum_feas);
            atomicAdd((u64 *)&A.counters[2], (u64)sum_acc);
            atomicAdd((u64 *)&A.counters[3], (u64)sum_imp);
            atomicAdd((u64 *)&A.counters[4], (u64)(sum_rows * dm.LP * 4));
        }
    }
    if (CHIP && live && (has_snap || pend)) {
        unsigned short *row = A.lo.cand_layout + (size_t)j * dm.N;
        const unsigned short *from = pend ? ch.cell : ch.snap;
        for (int x = lane; x < dm.N; x += 32) row[x] = from[x];
    }
    if (!CHIP) {
        if (!live) return;
        char *bdst = A.blob_dst + (size_t)j * A.bl.bytes;
        if (last) row_state_out(dm, A.bl, ch, bdst, lg, GL);
        else row_records_out(X, ch, bdst, lg, GL);
        int *td = (int *)(bdst + A.bl.off_wtab);
        for (int rg = lg; rg < dm.RG; rg += GL) { td[rg] = ch.ws[rg].x; X.F_dst[(size_t)j * dm.RG + rg] = ch.slack[rg]; }
        return;
    } else {
        // Meet the other chains: the reports are all they wait for, so arrive as soon as they are out.
        __syncthreads();
        if (tid == 0) {
            // (one thread's release covers what the CTA's threads wrote before they met)
            asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(A.sync) : "memory");
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
            const RowChain c = row_chain(dm, X, sm_chain, hw);
            char *bdst = buf_out + (size_t)jj * A.bl.bytes;
            int4 *wd = (int4 *)(X.Wr + (size_t)(half_w * P + jj) * dm.RG * X.rlp);
#pragma unroll 4
            for (int x = ht; x < nw; x += hn) wd[x] = c.W[x];
            if (last) row_state_out(dm, A.bl, c, bdst, ht, hn);
            else row_records_out(X, c, bdst, ht, hn);
            unsigned short *cd = (unsigned short *)(bdst + A.bl.off_cell);
            for (int x = ht; x < n4; x += hn) ((uint2 *)cd)[x] = ((const uint2 *)c.cell)[x];
            for (int i = (n4 << 2) + ht; i < dm.N; i += hn) cd[i] = c.cell[i];
            for (int rg = ht; rg < dm.RG; rg += hn) F_out[(size_t)jj * dm.RG + rg] = c.slack[rg];
            if (A.slices) {
                int *td = (int *)(bdst + A.bl.off_wtab);
                for (int rg = ht; rg < dm.RG; rg += hn) td[rg] = (half_w * P + jj) * dm.RG + rg;
            }
        }
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
        } else if (P <= NT) {
            // A member a thread: energies meet once, warps' weights once, and an ancestor is a count over the threads (five more
            // meetings of the CTA and a search of eight dependent steps as below: medium 849 us, here 807; two shards 859 and 816).
            const u64 r = tid < P ? __ldcg(eL + tid) : ~0ull >> 1;
            i64 e[1] = { (i64)(r & ~(1ull << 63)) };
            // (fetched beside the energy, whether its trajectory best beats the incumbent or not)
            const i64 b0 = tid < P ? __ldcg(bestL + 3 * tid) : 0, b1 = tid < P ? __ldcg(bestL + 3 * tid + 1) : 0, b2 = tid < P ? __ldcg(bestL + 3 * tid + 2) : 0;
            const int bj = r >> 63 ? tid : 0x7fffffff;
            const u32 hi = (u32)((u64)e[0] >> 32), mh = __reduce_min_sync(0xffffffffu, hi), ml = __reduce_min_sync(0xffffffffu, hi == mh ? (u32)e[0] : 0xffffffffu);
            if (lane == 0) { rmin[warp] = (i64)(((u64)mh << 32) | ml); rj[warp] = 0x7fffffff; }
            if (__any_sync(0xffffffffu, bj != 0x7fffffff)) {
                const int at = le_lexmin_lane(b0, b1, b2, bj);
                __syncwarp();
                if (lane == at) { r0[warp] = b0; r1s[warp] = b1; r2s[warp] = b2; rj[warp] = bj; }
            }
            if (tid == 0) win_s = -1;
            __syncthreads();
            i64 emin = rmin[0];
#pragma unroll
            for (int w = 1; w < NT / 32; ++w) emin = rmin[w] < emin ? rmin[w] : emin;
            if (warp == NT / 32 - 1) {                   // (the last warp: others may have fewer members to weigh, none has more)
                const int j0 = lane < NT / 32 ? rj[lane] : 0x7fffffff;
                if (__any_sync(0xffffffffu, j0 != 0x7fffffff)) {
                    const bool has = j0 != 0x7fffffff;
                    const i64 c0 = has ? r0[lane] : 0, c1 = has ? r1s[lane] : 0, c2 = has ? r2s[lane] : 0;
                    const int at = le_lexmin_lane(c0, c1, c2, j0);
                    // (all of them beat the incumbent)
                    if (lane == at) { inc_s[0] = c0; inc_s[1] = c1; inc_s[2] = c2; win_s = j0; }
                }
            }
            if (last) __syncthreads();
            else {
                const u64 M = (u64)(emin > dm.SC ? emin : dm.SC);
                u64 w[1] = { 0 };
                if (tid < P) le_weights<1>(e, emin, M, lv.cq, w);
                u64 F = w[0];
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) { const u64 x = __shfl_up_sync(0xffffffffu, F, o); if (lane >= o) F += x; }
                if (lane == 31) rsum[warp] = F;
                __syncthreads();
                u64 Ftot = 0;
#pragma unroll
                for (int x = 0; x < NT / 32; ++x) { const u64 y = rsum[x]; if (x < warp) F += y; Ftot += y; }
                const u64 u0 = (u64)(((unsigned __int128)lv.resample_x * Ftot) >> 32);
                const unsigned __int128 PF = (unsigned __int128)P * F;
                for (int m = m0; m < m1; ++m) {
                    // slots with P * F <= at
                    const int n = __syncthreads_count(tid < P && PF <= (unsigned __int128)u0 + (unsigned __int128)m * Ftot);
                    if (tid == 0) le_anc[m] = n;
                }
                __syncthreads();
            }
            if (win_s >= 0) inc_slot = win_s;
        } else {
        // incumbent: the lowest slot among the lexicographically best trajectory-best scores, if it beats it
        i64 b0 = inc_s[0], b1 = inc_s[1], b2 = inc_s[2], emin = 0x7fffffffffffffffll;
        int bj = 0x7fffffff;
        for (int m = tid; m < P; m += NT) {
            const u64 r = __ldcg(eL + m);
            const i64 e = (i64)(r & ~(1ull << 63));
            if (r >> 63) {
                const i64 s0 = __ldcg(bestL + 3 * m), s1 = __ldcg(bestL + 3 * m + 1), s2 = __ldcg(bestL + 3 * m + 2);
                if (rp_lex_less(s0, s1, s2, b0, b1, b2)) { b0 = s0; b1 = s1; b2 = s2; bj = m; }
            }
            emin = e < emin ? e : emin;
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
            if (P <= 2 * NT) le_prefix_weights_of<2>(P, en_of, lv.cq, tid, NT, emin, M, le_F, rsum, &carry_s);
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
            const RowChain c = row_chain(dm, X, sm_chain, hw);
            const char *bs = buf_out + (size_t)a * A.bl.bytes;
            const int4 *ws = (const int4 *)(X.Wr + (size_t)(half_w * P + a) * dm.RG * X.rlp);
            const unsigned short *cs = (const unsigned short *)(bs + A.bl.off_cell);
            // All of it in flight at once, past the L1 cache (four loops of loads one behind the other: medium 762 us, 743 here; tiny 314 and
            // 305; two shards the same).
            for (int x = ht; x < nw; x += hn) row_copy16(c.W + x, ws + x);
            for (int x = ht; x < (X.cs_bytes + 15) >> 4; x += hn) row_copy16((int4 *)c.base + x, (const int4 *)bs + x);
            if (A.bl.off_cell & 15) for (int x = ht; x < (dm.N + 3) >> 2; x += hn) ((uint2 *)c.cell)[x] = __ldcg((const uint2 *)cs + x);
            else for (int x = ht; x < (2 * dm.N + 15) >> 4; x += hn) row_copy16((int4 *)c.cell + x, (const int4 *)cs + x);
            // (both are padded to 16 bytes)
            for (int rg = ht; rg < dm.RG; rg += hn) c.slack[rg] = __ldcg(F_out + (size_t)a * dm.RG + rg);
            asm volatile("cp.async.wait_all;" ::: "memory");
            if (ht == 0) moved += 1;
        }
        half_w ^= 1;
        __syncthreads();
    }
    }
}

template <int GL, int LPL, int CPL, bool SPLIT, bool CHIP, bool COMP, bool IDENT>
static int launch_row_t(rp_ctx *c, const AnnealArgs &A, const RowArgs &X, int grid, int *done)
{
    constexpr bool TIGHT = !CHIP && ROW_WARPS_PER_SM(GL, LPL, CPL, IDENT) > 12;
    auto kern = k_anneal_row<GL, LPL, CPL, SPLIT, CHIP, COMP, IDENT, false>;
    // (or shared memory keeps no more than twelve resident anyway)
    constexpr bool LATE = !CHIP && !IDENT && GL == 32;
    if (LATE && !rp_row_starts_early(c)) kern = k_anneal_row<GL, LPL, CPL, SPLIT, CHIP, COMP, IDENT, LATE>;
    if (TIGHT && (grid <= 12 * rp_sms(c) || 228 * 1024 / (X.smem_bytes + 1024) <= 12)) kern = k_anneal_row<GL, LPL, CPL, SPLIT, CHIP, COMP, IDENT, TIGHT>;
    // (always the same value, above anything a launch asks for: contexts that plan different
    // windows at once on different host threads then never lower each other's limit)
    RP_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, ROW_SMEM_MAX));
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    *done = 0;
    if (CHIP && grid > rp_sms(c)) return RP_OK;
    cfg.gridDim = dim3(grid); cfg.blockDim = dim3(CHIP ? ROW_THREADS : 32);
    cfg.dynamicSmemBytes = X.smem_bytes; cfg.stream = c->stream;
    // Chains that start beside the launch before them (see rp_row_starts_early) go where there is room first: as much shared memory a CTA that
    // an SM takes its share of them and no more.  Nowhere else: other windows' chains have the room then (one launch per level each, 300 members
    // of 17 layers, two windows at once 896 -> 861 us a plan, four 513 -> 491; 512 of 24, four 548 -> 520).
    if (!CHIP && A.level > 0 && rp_row_starts_early(c)) {
        const size_t share = (grid + rp_sms(c) - 1) / rp_sms(c);
        cfg.dynamicSmemBytes = std::max(cfg.dynamicSmemBytes, (size_t)228 * 1024 / (share + 1) - 1024 + 256);
    }
    cudaLaunchAttribute at[1];
    if (CHIP) {
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
        cfg.attrs = at; cfg.numAttrs = 1;
    } else if (A.level > 0) {                       // behind the launch between two levels, see rp_level_turn.cu
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = at; cfg.numAttrs = 1;
    }
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, A, X);
    if (CHIP && e == cudaErrorCooperativeLaunchTooLarge) { cudaGetLastError(); return RP_OK; }
    RP_CUDA(e);
    ++g_rp_launches; ++c->n_queued;
    *done = 1;
    return RP_OK;
}

template <int GL, int LPL, int CPL, bool SPLIT, bool COMP, bool IDENT>
static int row_resident_t(const RowArgs &X, int *warps)
{
    auto kern = k_anneal_row<GL, LPL, CPL, SPLIT, false, COMP, IDENT, false>;
    RP_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, ROW_SMEM_MAX));
    RP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(warps, kern, 32, (size_t)X.smem_bytes));
    return RP_OK;
}
