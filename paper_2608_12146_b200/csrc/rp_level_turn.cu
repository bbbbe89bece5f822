// From one level of the population annealing to the next for the one-layer-per-lane kernel with one launch per level:
// incumbent, Boltzmann weights, ancestors, holders of the rank-load slices, list of free slices, in one cooperative launch.
//
// The three launches this replaces (a level barrier of one CTA, the holders, the free list) are short and one behind the
// other: what bounds them is latency, 34 us a level at 1024 members of 240 row-shards with the gaps.  Here the worker CTAs
// share the members out, meet once or twice and otherwise never wait; the last CTA looks after the incumbent (whose move log is
// replayed by a warp) beside them.  The chains leave their energies and the smallest of them behind.
//   1. weights, and all cumulative weights (every worker for itself).  Up to 1024 members every worker weighs them all, one or two a thread, and
//      there is no meeting (1024 members 2345 and 2324 us; four a thread at 1500 and 2048 gave nothing); more are shared out
//   2. ancestors of its members by 32 probes a step, the holders of the slices of each one that occurs
//   3. its piece of the slice table: free slices to the list, the counts of the level before back to zero (two tables taken in turn)
// In us a launch, 300 members of 100 row-shards 10.0 before, 9.0 here, 512 of 240 11.0 and 9.9, 1024 of 240 14, 4096 of 288 28 and 23.  What is left is
// trips to L2: two loads, a meeting of 2.5 k cycles and what the additions before it take to arrive, two loads and an addition.
#include <algorithm>
#include <string.h>
#include <type_traits>

#include "rp_level_end.cuh"
#include "rp_anneal_row.cuh"

#define TURN_THREADS 512
#define TURN_WARPS (TURN_THREADS / 32)
#define TURN_OWN 2                       // members a thread whose weights every worker works out for itself
#define TURN_ROWS 32
#define TURN_MAX_MEMBERS 16384           // cumulative weights on chip (with their padding, 136 KB)

struct TurnArgs {
    u64 *E, *weight;             // [P] energies of the terminal states, weights
    u64 *emin;                   // the smallest energy; left at its start value for the next level
    int *ref, *before, *list, *head;         // slices: counts (zero before), those of the level before (zero behind), free ones, cursors
    int ns;                      // slices
    int early;                   // the next level's chains may start
    int base;                    // arrivals at the meeting point of the launches before
};

__device__ __forceinline__ bool turn_meet(const AnnealArgs &A, int target)
{
    __shared__ int ok;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicAdd(A.sync, 1);
        ok = rp_wait_count(A.sync, target, A);
    }
    __syncthreads();
    return ok;
}

__global__ void __launch_bounds__(TURN_THREADS)
k_level_turn(const AnnealArgs A, const TurnArgs T)
{
    extern __shared__ __align__(16) unsigned char turn_smem[];
    __shared__ LeShared S;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int workers = (int)gridDim.x - 1, P = A.Ppop, RG = A.dm.RG;
    const bool own_weights = P <= TURN_OWN * TURN_THREADS;
    if (T.early) rp_let_next_launch_start();
    if ((int)blockIdx.x == workers) {
        if (__ldcg(&A.status[RP_SW_TIMEOUT])) return;
        i64 none;
        le_incumbent<false>(A, tid, TURN_THREADS, turn_smem, rp_le_ws_bytes(A, A.smem_bytes), S, none);
        return;
    }
    const int m0 = (int)((long long)P * blockIdx.x / workers), m1 = (int)((long long)P * (blockIdx.x + 1) / workers);

    // ---- 1: cumulative weights.  Up to TURN_OWN members a thread every worker weighs all members itself; more are shared out, and the
    // workers meet.  A thread adds up 2^lu consecutive members, place j of the table is j + (j >> lu) (no bank conflicts) ------------
    u64 *F = (u64 *)turn_smem;
    int lu = 0;
    const int late = __ldcg(&A.status[RP_SW_TIMEOUT]);
    const i64 emin = (i64)__ldcg(T.emin);
    const u64 M = (u64)(emin > A.dm.SC ? emin : A.dm.SC);
    while ((TURN_THREADS << lu) < P) ++lu;
    const int j0 = tid << lu, j1 = min(P, j0 + (1 << lu));
    u64 own = 0;
    auto weigh = [&](auto count) {                               // its own members, worked out here
        constexpr int U = decltype(count)::value;
        i64 e[U];
        u64 w[U];
#pragma unroll
        for (int u = 0; u < U; ++u) e[u] = j0 + u < P ? (i64)__ldcg(T.E + j0 + u) : emin;
        le_weights<U>(e, emin, M, A.cq, w);
#pragma unroll
        for (int u = 0; u < U; ++u) if (j0 + u < P) { own += w[u]; F[j0 + u + (j0 + u) / U] = own; }
    };
    if (own_weights) {
        if (late) return;
        if (lu == 0) weigh(std::integral_constant<int, 1>());
        else weigh(std::integral_constant<int, TURN_OWN>());
    } else {
        if (late) return;
        for (int m = m0 + tid; m < m1; m += TURN_THREADS) {
            const i64 e[1] = { (i64)__ldcg(T.E + m) };
            u64 w[1];
            le_weights<1>(e, emin, M, A.cq, w);
            T.weight[m] = w[0];
        }
        if (!turn_meet(A, T.base + workers)) { if (tid == 0) atomicExch(&A.status[RP_SW_TIMEOUT], 1); return; }
        for (int j = j0; j < j1; ++j) { own += __ldcg(T.weight + j); F[j + (j >> lu)] = own; }
    }
    u64 v = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const u64 x = __shfl_up_sync(0xffffffffu, v, o); if (lane >= o) v += x; }
    if (lane == 31) S.rsum[warp] = v;
    __syncthreads();
    u64 before = v - own;
#pragma unroll
    for (int x = 0; x < TURN_WARPS; ++x) { const u64 y = S.rsum[x]; if (x < warp) before += y; }
    for (int j = j0; j < j1; ++j) F[j + (j >> lu)] += before;
    __syncthreads();
    if (blockIdx.x == 0 && tid == 0) { T.head[0] = 0; T.head[1] = 0; }

    // ---- 2: ancestors, a warp per member: the slots with P * F <= at, by 32 probes a step ---------------------
    int *anc = (int *)(F + P + (P >> lu) + 1);                   // of this worker's members
    {
        const u64 Ftot = F[P - 1 + ((P - 1) >> lu)];
        const u64 u0 = (u64)(((unsigned __int128)A.resample_x * Ftot) >> 32);
        for (int m = m0 + warp; m < m1; m += TURN_WARPS) {
            const unsigned __int128 at = (unsigned __int128)u0 + (unsigned __int128)m * Ftot;
            int lo = 0, hi = P - 1;                     // smallest slot with P * F > at
            while (lo < hi) {
                const int n = hi - lo, j = lo + (int)(((long long)n * lane) >> 5);          // (rising with the lane, lo .. hi - 1)
                const unsigned low = __ballot_sync(0xffffffffu, (unsigned __int128)P * F[j + (j >> lu)] <= at);
                const int c = __popc(low);                                               // probes of the first c lanes are too low
                const int below = __shfl_sync(0xffffffffu, j, c ? c - 1 : 0), above = __shfl_sync(0xffffffffu, j, c < 32 ? c : 31);
                lo = c ? below + 1 : lo;
                hi = c < 32 ? above : hi;
            }
            if (lane == 0) {
                anc[m - m0] = lo;
                A.lo.anc_out[m] = lo;
                if (A.lo.tr_anc) A.lo.tr_anc[(size_t)A.level * P + m] = lo;
            }
        }
    }
    __syncthreads();
    // Ancestors rise with the member: each one that this worker's members have, once, and where its members start.
    int *who = anc + (m1 - m0) + 1, *start = who + (m1 - m0) + 1;
    if (warp == 0) {
        int k = 0;
        for (int x0 = 0; x0 < m1 - m0; x0 += 32) {
            const int x = x0 + lane;
            const bool head = x < m1 - m0 && (x == 0 || anc[x] != anc[x - 1]);
            const unsigned b = __ballot_sync(0xffffffffu, head);
            if (head) { const int at = k + __popc(b & ((1u << lane) - 1)); who[at] = anc[x]; start[at] = x; }
            k += __popc(b);
        }
        if (lane == 0) { start[k] = m1 - m0; S.win_n = k; }
    }
    __syncthreads();
    // Holders among the members that start the next level.  Most members share most slices for some levels, and additions to one
    // address queue up (one each: 14 k cycles at 1024 members of 240 row-shards, 60 k at 4096 of 288); so a thread takes one row-shard of
    // several ancestors and adds a run of equal slices at once, with the slice it saw first, the one nearly all of them share, counted
    // beside the runs.
    {
        const int groups = max(1, TURN_THREADS / RG), n = S.win_n;
        for (int x = tid; x < groups * RG; x += TURN_THREADS) {
            const int g = x / RG, rg = x - g * RG;
            const int a0 = n * g / groups, a1 = n * (g + 1) / groups;
            int first = -1, n_first = 0, run = -1, n_run = 0;
            for (int m = a0; m < a1; m += 8) {
                int s[8];
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    s[u] = m + u < a1 ? __ldcg((const int *)(A.blob_dst + (size_t)who[m + u] * A.bl.bytes + A.bl.off_wtab) + rg) : -1;
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    if (m + u >= a1) continue;
                    if ((unsigned)s[u] >= (unsigned)T.ns) { atomicExch(&A.status[RP_SW_POOL], 1); continue; }
                    const int c = start[m + u + 1] - start[m + u];
                    if (first < 0) first = s[u];
                    if (s[u] == first) { n_first += c; continue; }
                    if (s[u] != run) { if (n_run) atomicAdd(&T.ref[run], n_run); run = s[u]; n_run = 0; }
                    n_run += c;
                }
            }
            if (n_first) atomicAdd(&T.ref[first], n_first);
            if (n_run) atomicAdd(&T.ref[run], n_run);
        }
    }
    if (!turn_meet(A, T.base + (own_weights ? 1 : 2) * workers)) { if (tid == 0) atomicExch(&A.status[RP_SW_TIMEOUT], 1); return; }
    if (blockIdx.x == 0 && tid == 0) *T.emin = ~0ull >> 1;       // (every worker has read it)

    // ---- 3: free slices, and the counts of the level before back to zero.  A warp takes up to 32 * TURN_ROWS slices at a time, the CTA one
    // piece of the list for all of its warps; loads and stores of consecutive lanes are consecutive --------------------------
    const int rows = min(TURN_ROWS, (int)(((long long)T.ns + (long long)workers * TURN_THREADS - 1) / ((long long)workers * TURN_THREADS)));
    const int per = TURN_THREADS * rows;
    for (long long b0 = (long long)blockIdx.x * per; b0 < T.ns; b0 += (long long)workers * per) {
        const int s0 = (int)b0 + warp * 32 * rows + lane;
        unsigned isfree[TURN_ROWS];
        int n = 0;
#pragma unroll
        for (int rb = 0; rb < TURN_ROWS; rb += 8) {
            if (rb >= rows) break;
            int v[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) v[r] = rb + r < rows && s0 + 32 * (rb + r) < T.ns ? __ldcg(T.ref + s0 + 32 * (rb + r)) : 1;
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const int s = s0 + 32 * (rb + r);
                if (rb + r < rows && s < T.ns) T.before[s] = 0;
                isfree[rb + r] = __ballot_sync(0xffffffffu, v[r] == 0);
                n += __popc(isfree[rb + r]);
            }
        }
        __syncthreads();                             // (S.rj of the round before)
        if (lane == 0) S.rj[warp] = n;
        __syncthreads();
        if (warp == 0) {
            int w = lane < TURN_WARPS ? S.rj[lane] : 0;
            const int mine = w;
            for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(0xffffffffu, w, o); if (lane >= o) w += y; }
            int base = 0;
            if (lane == 31 && w) base = atomicAdd(&T.head[1], w);
            base = __shfl_sync(0xffffffffu, base, 31);
            if (lane < TURN_WARPS) S.rj[lane] = base + w - mine;
        }
        __syncthreads();
        int at = S.rj[warp];
#pragma unroll
        for (int r = 0; r < TURN_ROWS; ++r) {
            if (r >= rows) break;
            if ((isfree[r] >> lane) & 1u) T.list[at + __popc(isfree[r] & ((1u << lane) - 1))] = s0 + 32 * r;
            at += __popc(isfree[r]);
        }
    }
}

// Workers: as many as have something to do (a meeting costs the more the more there are); every one resident.
static int turn_workers(const rp_ctx *c)
{
    const int P = c->Ppop, ns = 2 * P * c->dm.RG;
    return std::max(4, std::min(rp_sms(c) - 1, std::max((P + 15) / 16, (ns + 4095) / 4096)));
}

// One launch per level asked for means that a caller plans several windows at once on separate streams: a launch whose CTAs wait
// for one another would make them wait for its SMs, so the parts then stay launches of their own, as beyond the table on chip and where a
// part of a GPU does not hold the workers and the CTA for the incumbent.
bool rp_row_turns(const rp_ctx *c) { return c->knob_level_launches != 1 && c->Ppop <= TURN_MAX_MEMBERS && turn_workers(c) < rp_sms(c); }

int rp_launch_level_end(rp_ctx *c, const AnnealArgs &A);

// Between level A.level of an rp_anneal call and the next one.
int rp_launch_level_turn(rp_ctx *c, const AnnealArgs &A0)
{
    const int P = c->Ppop, ns = 2 * P * c->dm.RG;
    AnnealArgs A = A0;
    TurnArgs T;
    T.E = c->d_F; T.weight = c->d_F + P; T.emin = c->d_F + 2 * (size_t)P;
    T.ref = c->d_wcount; T.before = c->d_wref; T.list = c->d_wfree; T.head = c->d_wfree_head;
    T.ns = ns; T.early = rp_row_starts_early(c);
    A.sync = c->d_sync;
    const int workers = turn_workers(c);
    T.base = A.level * (P <= TURN_OWN * TURN_THREADS ? 1 : 2) * workers;                  // (the count is zero when the call starts)
    int lu = 0;
    while ((TURN_THREADS << lu) < P) ++lu;
    const size_t ws_workers = sizeof(u64) * ((size_t)P + (P >> lu) + 1) + sizeof(int) * 3 * ((size_t)P / workers + 3);
    size_t ws = std::max((size_t)16 * 1024, std::min((size_t)2 * std::max((size_t)A.log_cap * 8, (size_t)c->dm.N * 3), (size_t)160 * 1024));
    ws = (std::max(ws, ws_workers) + 15) & ~(size_t)15;
    A.smem_bytes = (unsigned)ws;
    RP_CUDA(cudaFuncSetAttribute(k_level_turn, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = dim3(workers + 1); cfg.blockDim = dim3(TURN_THREADS); cfg.dynamicSmemBytes = ws; cfg.stream = c->stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at; cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_level_turn, A, T);
    if (e == cudaErrorCooperativeLaunchTooLarge) {        // a part of a GPU: the launches one by one, at every level
        cudaGetLastError();
        return rp_launch_level_end(c, A0);
    }
    RP_CUDA(e);
    ++g_rp_launches; ++c->n_queued;
    c->slices_listed = 1;
    std::swap(c->d_wref, c->d_wcount);               // the counts are the next level's holders
    return RP_OK;
}
