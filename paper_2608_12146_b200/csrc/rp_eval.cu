// Full evaluation of layouts (K4): cell statistics, per-row-shard rank loads W, expert and
// attention costs, shard work and the score tuple (Sections 3.4-3.5 of the paper).
//
// The work is the sum of the q rows of every row-shard's samples: N*L*P*4 bytes per layout, served by L2
// (q is shared by all layouts).  Two forms:
//  * few layouts of rows in whole 16-byte chunks (k_eval_few: the seed, the incumbent, diagnostics, small batches), bound by latency: a cluster of
//    CTAs per row-shard, each over its share of the samples, sixteen 16-byte loads in flight per lane; the CTAs'
//    sums meet through distributed shared memory;
//  * many layouts (k_eval_group, k_eval_slice or k_eval_sum, k_eval_score): the samples of a layout are grouped by row-shard once; then a
//    CTA keeps a slice of all samples' rows on chip and adds up the row-shards of many layouts from there (bound by shared memory), or,
//    where such a slice does not fit, warps stream through the rows in L2.
// In the first the cluster that finishes a layout last (atomic ticket) scores it.
#include <cooperative_groups.h>

#include <algorithm>

#include "rp_score.cuh"

namespace cg = cooperative_groups;

#define EVAL_THREADS 256
#define EVAL_SMEM_MAX (220 * 1024)

// What a launch scores and where its results go.
struct EvalArgs {
    RpDims dm;
    RpBlob bl;
    const int *lay32;                             // [n][N] layouts, or (null) the assignments of blobs[src[0..n-1]]
    const char *blobs;
    const int *src;
    const int *t, *q, *edp, *dp_list, *dp_off;
    int first;                                    // layouts of the call before this launch's
    int *W_out;                                   // [n][RG][LP], nullable
    char *blob_out;                               // [n] chain-state blobs (see RpBlob), nullable
    i64 *score_out, *score_out2;                  // [n][3], nullable
    double *f64_out;                              // [n][3], nullable
    int *bad;                                     // raised when a layout names a cell outside [0, K) (host memory; such a sample counts as cell 0)
    // Scores for a caller's device memory, which stays as it is if any layout of the call is bad: `bad_dev` is raised with `bad`
    // and zero before.  Many layouts: all are looked at before the first is scored.  Few: the CTA that finishes the last layout
    // (counter behind the tickets) copies them from score_out / f64_out.
    int *bad_dev;
    i64 *score_final;
    double *f64_final;
    int n;
    bool q_halves;                                // no cell's squared lengths add up to 2^48, whatever the layout
    i64 *cost;                                    // [n][RG] row-shard costs handed to the finishing CTA; zero between launches
    int *tickets;                                 // [n] arrival counters (many layouts: whether a cell is empty or overfull); zero between launches
    unsigned short *list;                         // [n][N] samples grouped by row-shard (k_eval_group)
    u32 *off;                                     // [n][RG+1] where a row-shard's samples start, and in the upper half which row-shard it is
    // Validation of the incumbent: with `host` set (pinned), the finishing CTA leaves the search's counters, the status
    // words, the incumbent's cached score, its full score, the best seed's and its layout there.
    i64 *host;
    const i64 *counters, *inc_score, *seed_score;
    const int *status;
    int *layout_host;
};

// Cell of sample i in layout lay.
struct EvalCells { const int *a; const unsigned short *b; };
__device__ __forceinline__ EvalCells eval_cells(const EvalArgs &A, int lay)
{
    EvalCells e;
    e.a = A.lay32 ? A.lay32 + (size_t)lay * A.dm.N : nullptr;
    e.b = A.lay32 ? nullptr : (const unsigned short *)(A.blobs + (size_t)A.src[lay] * A.bl.bytes + A.bl.off_cell);
    return e;
}
__device__ __forceinline__ int eval_cell(const EvalArgs &A, const EvalCells &e, int i)
{
    if (!e.a) return __ldg(e.b + i);
    const int c = __ldg(e.a + i);
    if ((unsigned)c < (unsigned)A.dm.K) return c;
    *A.bad = 1;
    if (A.bad_dev) *A.bad_dev = 1;
    return 0;
}

// Sum of one 16-byte column of the listed samples' rows, U loads in flight.
template <int U>
__device__ __forceinline__ int4 eval_sum_column(const int4 *__restrict__ col, size_t row4, const int *list, int m0, int m1)
{
    int4 a = make_int4(0, 0, 0, 0);
    for (int mb = m0; mb < m1; mb += U) {
        int4 v[U];
#pragma unroll
        for (int e = 0; e < U; ++e) v[e] = mb + e < m1 ? __ldg(col + (size_t)list[mb + e] * row4) : make_int4(0, 0, 0, 0);
#pragma unroll
        for (int e = 0; e < U; ++e) { a.x += v[e].x; a.y += v[e].y; a.z += v[e].z; a.w += v[e].w; }
    }
    return a;
}

// Rows of whole 16-byte chunks with at most 32 chunks per layer: a warp takes whole layers, chunk by lane.
__host__ __device__ static inline bool eval_vec(const RpDims &dm) { return (dm.P & 3) == 0 && dm.P <= 128; }
__device__ __forceinline__ int eval_layer_max(int m, int lane, int cpl)      // maximum over the cpl lanes of a layer, in its first lane
{
    if ((cpl & (cpl - 1)) == 0) { for (int o = cpl >> 1; o; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o)); }
    else { const int own = m; for (int o = 1; o < cpl; ++o) m = max(m, __shfl_down_sync(0xffffffffu, own, o)); }
    return m;
}

// Sums of squared lengths in shared memory: 64 bits, or (halves: no sum reaches 2^48) the lower 16 bits of each square and what lies
// above them added up in 32 bits each.  A 64-bit addition there is a loop, and the samples of a row-shard of few slots meet in it: 4000
// samples in six row-shards of one slot, 128 layouts 206 us and 147 in halves, one layout 48 and 41.
__device__ __forceinline__ void few_add(u64 *q, u32 low, u32 high, bool halves)
{
    if (halves) { atomicAdd((u32 *)q, low); atomicAdd((u32 *)q + 1, high); }
    else atomicAdd(q, ((u64)high << 32) | low);
}
__device__ __forceinline__ u64 few_square(u64 v, bool halves) { return halves ? ((v >> 32) << 16) + (u32)v : v; }
__device__ __forceinline__ void few_add_square(u64 *q, int t, bool halves)
{
    const u64 sq = (u64)t * (u64)t;
    if (halves) few_add(q, (u32)sq & 0xffffu, (u32)(sq >> 16), true);
    else few_add(q, (u32)sq, (u32)(sq >> 32), false);
}

// Many layouts, first kernel (one CTA per layout): its samples grouped by row-shard, the cells' statistics and from them the
// attention part of every row-shard's cost.  by_length: the row-shards in order of decreasing sample counts (equal from
// GROUP_BINS - 1 on), so that those summed side by side are of nearly the same length.
#define GROUP_THREADS 512
#define GROUP_BINS GROUP_THREADS
static inline size_t eval_group_bytes(const RpDims &dm)
{
    return (sizeof(u64) * (size_t)dm.K + sizeof(int) * 2 * ((size_t)dm.RG + (size_t)dm.K) + 2 * ((size_t)dm.K + dm.N) + 15) & ~(size_t)15;
}
__global__ void __launch_bounds__(GROUP_THREADS)
k_eval_group(const EvalArgs A, bool by_length)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    const RpDims &dm = A.dm;
    u64 *Q = (u64 *)smraw;                                              // [K] statistics
    int *T = (int *)(Q + dm.K), *cnt = T + dm.K;
    int *off = cnt + dm.K;                                              // [RG] counts, then fill pointers
    int *end = off + dm.RG;                                             // [RG] the same from the other end
    unsigned short *rg_of = (unsigned short *)(end + dm.RG);            // [K]
    unsigned short *rgs = rg_of + dm.K;                                 // [N]
    __shared__ int wsum[GROUP_THREADS / 32], bins[GROUP_BINS];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, lay = blockIdx.x;
    for (int x = tid; x < dm.RG; x += GROUP_THREADS) off[x] = 0;
    for (int c = tid; c < dm.K; c += GROUP_THREADS) { rg_of[c] = (unsigned short)rp_rowshard(dm, A.edp, c); Q[c] = 0; T[c] = 0; cnt[c] = 0; }
    bins[tid] = 0;
    __syncthreads();
    const EvalCells e = eval_cells(A, lay);
    char *b = A.blob_out ? A.blob_out + (size_t)lay * A.bl.bytes : nullptr;
#pragma unroll 4
    for (int i = tid; i < dm.N; i += GROUP_THREADS) {
        const int c = eval_cell(A, e, i), rg = rg_of[c], t = __ldg(A.t + i);
        rgs[i] = (unsigned short)rg;
        atomicAdd(&off[rg], 1);
        atomicAdd(&T[c], t); atomicAdd(&cnt[c], 1);
        few_add_square(&Q[c], t, A.q_halves);
        if (b) ((unsigned short *)(b + A.bl.off_cell))[i] = (unsigned short)c;
    }
    __syncthreads();
    u32 *go = A.off + (size_t)lay * (dm.RG + 1);
    // exclusive sums over the CTA of one number per thread
    auto before = [&](int own) {
        int v = own;
        for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(0xffffffffu, v, o); if (lane >= o) v += y; }
        if (lane == 31) wsum[warp] = v;
        __syncthreads();
        int run = v - own;
        for (int w = 0; w < warp; ++w) run += wsum[w];
        return run;
    };
    if (by_length) {
        // the row-shards of one length lie together, the lengths in decreasing order: where the samples and the row-shards
        // of a length start (a thread per length)
        for (int x = tid; x < dm.RG; x += GROUP_THREADS) atomicAdd(&bins[min(off[x], GROUP_BINS - 1)], 1);
        __syncthreads();
        const int len = GROUP_BINS - 1 - tid, first = before(bins[len]);
        __syncthreads();
        bins[len] = first;
        __syncthreads();
        // (a row-shard's place is handed to the prefix sums through the list of places)
        for (int x = tid; x < dm.RG; x += GROUP_THREADS) go[atomicAdd(&bins[min(off[x], GROUP_BINS - 1)], 1)] = (u32)x << 16;
        __syncthreads();
    }
    {   // exclusive prefix sums: a thread takes consecutive places
        const int chunk = (dm.RG + GROUP_THREADS - 1) / GROUP_THREADS, x0 = min(dm.RG, tid * chunk), x1 = min(dm.RG, x0 + chunk);
        int sum = 0;
        for (int x = x0; x < x1; ++x) sum += off[by_length ? go[x] >> 16 : x];
        int run = before(sum);
        for (int x = x0; x < x1; ++x) {
            const int rg = by_length ? go[x] >> 16 : x, c = off[rg];
            off[rg] = run; go[x] = (u32)run | (u32)rg << 16; run += c;
            end[rg] = run;
        }
        if (tid == 0) go[dm.RG] = (u32)dm.N;
    }
    __syncthreads();
    unsigned short *list = A.list + (size_t)lay * dm.N;
    for (int i = tid; i < dm.N; i += GROUP_THREADS) {
        if (!by_length || !(i & 1)) list[atomicAdd(&off[rgs[i]], 1)] = (unsigned short)i;
        else list[atomicSub(&end[rgs[i]], 1) - 1] = (unsigned short)i;                 // odd ones from the end (see k_eval_slice)
    }
    for (int rg = tid; rg < dm.RG; rg += GROUP_THREADS) {
        const int r = rg / dm.G, g = rg % dm.G, d0 = __ldg(A.dp_off + g), d1 = __ldg(A.dp_off + g + 1);
        i64 Af = 0;
        for (int s = 0; s < dm.S; ++s) {
            const i64 ca = dm.ahat[s] * dm.C, cb = dm.bhat[s];
            i64 worst = 0;
            for (int x = d0; x < d1; ++x) {
                const int c = r * dm.D + __ldg(A.dp_list + x);
                const i64 v = ca * T[c] + cb * (i64)few_square(Q[c], A.q_halves);
                worst = v > worst ? v : worst;
            }
            Af += worst;
        }
        A.cost[(size_t)lay * dm.RG + rg] = Af;                          // the sums add the expert part
        if (b) {
            ((i64 *)(b + A.bl.off_Afx))[rg] = Af;
            if (A.bl.off_wtab >= 0)        // the pool holds the call's layouts as RG consecutive slices each
                ((int *)(b + A.bl.off_wtab))[rg] = (A.first + lay) * dm.RG + rg;
        }
    }
    int wrong = 0;
    for (int c = tid; c < dm.K; c += GROUP_THREADS) {
        wrong |= cnt[c] < 1 || T[c] > dm.C;
        if (b) { ((u64 *)(b + A.bl.off_Q))[c] = few_square(Q[c], A.q_halves); ((int *)(b + A.bl.off_T))[c] = T[c]; ((int *)(b + A.bl.off_cnt))[c] = cnt[c]; }
    }
    wrong = __syncthreads_or(wrong);
    if (tid == 0) A.tickets[lay] = wrong;
}

// Many layouts, second kernel where N rows of at least one 16-byte chunk fit on chip.  A CTA holds `w` consecutive chunks of every
// sample's row, `lps` whole layers or one of `parts` pieces of a layer, and adds up the row-shards of a share of the layouts
// from there: teams of TW lanes, a row-shard each and a chunk a lane, read their samples' ids sixteen bits at a time and then the
// rows from shared memory; a team that has finished reads the row of zeros behind the last sample.  Every sample's row crosses
// L2 once a CTA instead of once a layout; bound by its instructions and by shared memory alike (a quarter warp reads 128 bytes at a
// time, two rows of 64 bytes collide where both are even or odd): 256 layouts of 2048 samples in 240 row-shards, 24 layers of 16 ranks, 136 us
// with the streaming sums, 80 with a division and a multiplication per row-shard and sample left in, 66 (a call 161, and 93 now).
#define SLICE_THREADS 1024
#define SLICE_MAX (1 << 12)           // row-shards whose busiest loads are kept between the pieces of a layer
struct SlicePlan { int tw, w, parts, lps, slices, groups, batch; size_t smem; };
template <int TW>
__global__ void __launch_bounds__(SLICE_THREADS)
k_eval_slice(const EvalArgs A, const SlicePlan S, int n)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    const RpDims &dm = A.dm;
    constexpr int TPW = 32 / TW, IDS = TW < 4 ? 4 : TW, PER = IDS / TW;          // teams of a warp; samples a round, ids of a lane
    int4 *rows = (int4 *)smraw;                                                 // [N + 1][w]
    const int N = dm.N, RG = dm.RG, cpl = dm.P >> 2, rc = dm.LP >> 2, w = S.w;
    int *top = (int *)(rows + (size_t)(N + 1) * w);                             // parts > 1: [batch * RG] busiest loads so far
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, team = lane / TW, k = lane & (TW - 1);
    const int slice = blockIdx.x % S.slices, group = blockIdx.x / S.slices, layer = slice * S.lps;
    const bool first_of_layer = k % cpl == 0;
    const int nl = min(S.lps, dm.L - layer), used = S.parts > 1 ? w : nl * cpl;        // chunks that exist
    const int last = (int)((long long)n * (group + 1) / S.groups);
    for (int lay0 = (int)((long long)n * group / S.groups); lay0 < last; lay0 += S.batch) {
        const u32 nrg = min(S.batch, last - lay0) * RG;                         // row-shards of this batch of layouts
        for (int part = 0; part < S.parts; ++part) {
            const int first = layer * cpl + part * w;                           // first chunk
            if (part || S.parts > 1 || lay0 == (int)((long long)n * group / S.groups)) {
                __syncthreads();
                const int4 *q4 = (const int4 *)A.q + first;
                for (int x = tid; x < N * w; x += SLICE_THREADS) {
                    const int i = x / w, c = x - i * w;
                    if (c < used) {
                        const unsigned dst = (unsigned)__cvta_generic_to_shared(rows + x);
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(q4 + (size_t)i * rc + c) : "memory");
                    } else rows[x] = make_int4(0, 0, 0, 0);
                }
                if (tid < w) rows[(size_t)N * w + tid] = make_int4(0, 0, 0, 0);
                asm volatile("cp.async.wait_all;" ::: "memory");
                __syncthreads();
            }
            const int4 *col = rows + min(k, w - 1);
            constexpr int STRIDE = SLICE_THREADS / TW;
            // This team's row-shard of the batch: place `hi` of layout `lo` of the batch (across), or place `lo` of layout `hi`.  Across, the
            // teams of a warp have row-shards of one place, which are of nearly the same length in all layouts, and the longest come first:
            // few long row-shards of a layout differ much (3300 samples in 32, 47 layers of 16 ranks, 500 layouts 1152 us one layout after the other, 310
            // across; in 208, 383 and 379).  With one or two lanes a team a warp's ids then lie in 32 or 16 lists at a time, which only pays
            // where there are several rounds (6900 in 24, 11 of 8, 64 layouts 140 and 160, 500 405 and 259), with one lane hardly ever (13000 in
            // 240, 24 of 4, 500 layouts 692 and 990).
            const bool across = TW > 2 || (TW == 2 && nrg >= (u32)STRIDE);
            const u32 inner = across ? nrg / RG : RG, dh = STRIDE / inner, dl = STRIDE % inner;
            u32 f = warp * TPW + team, hi = f / inner, lo = f - hi * inner;
            u32 o0 = 0, o1 = 0;
            if (f < nrg) { const u32 *go = A.off + (lay0 + (across ? lo : hi)) * (RG + 1u) + (across ? hi : lo); o0 = __ldg(go); o1 = __ldg(go + 1); }
            while (f - team < nrg) {
                const bool on = f < nrg;
                const int p = (int)(o0 & 0xffffu), len = (int)(o1 & 0xffffu) - p;
                const u32 lay = lay0 + (across ? lo : hi), at = lay * (u32)RG + (o0 >> 16), here = f;
                // Odd teams walk their list from its end: a list holds its even samples first, and rows of 64 bytes that a
                // quarter warp reads together collide where both are even or both odd.
                const unsigned short *list = A.list + lay * (u32)N + ((team & 1) ? p + len - 1 : p);
                const int step = (team & 1) ? -1 : 1;
                f += STRIDE; hi += dh; lo += dl;                                // the next one's offsets under this one's sums
                if (lo >= inner) { lo -= inner; ++hi; }
                o0 = o1 = 0;
                if (f < nrg) { const u32 *go = A.off + (lay0 + (across ? lo : hi)) * (RG + 1u) + (across ? hi : lo); o0 = __ldg(go); o1 = __ldg(go + 1); }
                const int most = (int)__reduce_max_sync(0xffffffffu, len);
                int4 a = make_int4(0, 0, 0, 0);
                int id[PER];
#pragma unroll
                for (int m = 0; m < PER; ++m) { const int e = m * TW + k; id[m] = w * (e < len ? (int)__ldg(list + e * step) : N); }
                for (int done = 0; done < most; done += IDS) {
                    int now[PER];
#pragma unroll
                    for (int m = 0; m < PER; ++m) { const int e = done + IDS + m * TW + k; now[m] = id[m]; id[m] = w * (e < len ? (int)__ldg(list + e * step) : N); }
#pragma unroll
                    for (int u = 0; u < IDS; u += 2) {
                        if (done + u >= most) break;
                        const int i0 = TW == 1 ? now[u] : __shfl_sync(0xffffffffu, now[u / TW], u % TW, TW),
                                  i1 = TW == 1 ? now[u + 1] : __shfl_sync(0xffffffffu, now[(u + 1) / TW], (u + 1) % TW, TW);
                        const int4 v = col[i0], z = col[i1];
                        a.x += v.x + z.x; a.y += v.y + z.y; a.z += v.z + z.z; a.w += v.w + z.w;
                    }
                }
                const bool mine = on && k < used;
                if (A.W_out && mine) ((int4 *)(A.W_out + (size_t)at * dm.LP))[first + k] = a;
                int m = mine ? max(max(a.x, a.y), max(a.z, a.w)) : 0;
                i64 es;
                if (S.lps == 1) {                                               // (a piece of) one layer
#pragma unroll
                    for (int o = 1; o < TW; o <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
                    if (S.parts > 1 && on && k == 0) {
                        if (part) m = max(m, top[here]);
                        top[here] = m;
                    }
                    es = m;
                } else {                                                        // whole layers: maximum over cpl lanes, sum over the layers
                    const int own = m;
                    for (int o = 1; o < cpl; ++o) m = max(m, __shfl_down_sync(0xffffffffu, own, o, TW));
                    es = mine && first_of_layer ? (i64)m : 0;
#pragma unroll
                    for (int o = 1; o < TW; o <<= 1) es += __shfl_xor_sync(0xffffffffu, es, o);
                }
                if (on && k == 0 && part + 1 == S.parts) atomicAdd((u64 *)A.cost + at, (u64)(dm.EC * es));
            }
        }
    }
}

// How k_eval_slice divides the rows (tw = 0: not at all).  As many chunks of a row as fit, up to eight, a CTA to an SM; the SMs
// are shared out so that their busiest has the least to do.  A layer in pieces is read a piece at a time, over again for every batch of layouts,
// and pieces of one or two chunks are slower than the streaming sums.  Calls in us, streaming and from slices: whole layers, 2048 samples in 240
// row-shards, 24 layers of 16 ranks, n = 256 159 and 102; 13000 in 96, 8 of 4, n = 16 181 and 142; 700 in 48, 48 of 24, n = 256 163 and 121;
// pieces of four chunks, 3000 in 192, 24 of 32, n = 4 62 and 60, 64 128 and 93, 256 274 and 234; of two, 6000 in 96, 48 of 32, n = 4 146
// and 192, 256 855 and 1726; of one, 8192 in 448, 24 of 16, n = 4 84 and 117, 256 344 and 1033.
static SlicePlan eval_slice_plan(const RpDims &dm, int n)
{
    SlicePlan S = {};
    const int cpl = dm.P >> 2;
    if ((dm.P & 3) || dm.N > 65534) return S;
    auto fits = [&](int w, int parts) { return 16 * (size_t)w * (dm.N + 1) + (parts > 1 ? 4 * (size_t)SLICE_MAX : 0) <= EVAL_SMEM_MAX; };
    S.parts = 1;
    while (S.parts <= cpl && !(cpl % S.parts == 0 && cpl / S.parts <= 8 && fits(cpl / S.parts, S.parts))) ++S.parts;
    if (S.parts > cpl || (S.parts > 1 && (cpl / S.parts < 3 || dm.RG > SLICE_MAX))) return SlicePlan{};
    S.lps = 1;
    if (S.parts == 1) while (S.lps < dm.L && cpl * (S.lps + 1) <= 8 && fits(cpl * (S.lps + 1), 1)) ++S.lps;
    S.w = cpl * S.lps / S.parts;
    S.tw = 1;
    while (S.tw < S.w) S.tw *= 2;
    S.slices = (dm.L + S.lps - 1) / S.lps;
    double best = 1e300;
    for (int g = 1; g <= std::min(n, 32); ++g) {
        // per CTA: loading its slice, then its layouts, in units of a layout's samples (64 bytes a cycle and SM from L2, 90 from shared memory)
        const double cost = std::ceil((double)S.slices * g / 148) * (1.5 + (double)((n + g - 1) / g));
        if (cost < best) { best = cost; S.groups = g; }
    }
    // Narrow slices collide in shared memory (rows of 16 or 32 bytes) and pay a trip through the lists per layer, in ps a sample and layer 4.0 and
    // 3.6; rows that stream fill a warp's strips whatever a layer has, 80, 104 and 140 ps a sample for one to three of them.  With enough layouts
    // for both rates: 13000 samples in 240 row-shards, 47 layers of 4 ranks, 500 layouts 1182 us from slices and 697 streaming, 24 layers
    // 692 and 531, 11 394 and 526; 6900 in 240, 47 of 8, 622 and 568, 24 357 and 427.  Few long row-shards stream badly (6900 in 24, 47 of 8,
    // 1008 and, across, 713).
    if (S.tw <= 2 && (long long)n * S.slices >= 6000) {
        const int used = 32 / cpl * cpl, strips = ((dm.LP >> 2) + used - 1) / used, ns = std::min(3, strips);
        const double row = S.slices * (S.tw == 1 ? 4.0 : 3.6), streamed = (strips + ns - 1) / ns * (ns == 1 ? 80.0 : ns == 2 ? 104.0 : 140.0);
        if (row > streamed && (S.tw == 1 || dm.N <= 128ll * dm.RG)) return SlicePlan{};
    }
    S.batch = S.parts > 1 ? std::max(1, SLICE_MAX / dm.RG) : n;
    S.smem = 16 * (size_t)S.w * (dm.N + 1) + (S.parts > 1 ? 4 * (size_t)SLICE_MAX : 0);
    return S;
}

// Many layouts, second kernel elsewhere.  A task is NS strips of 32 chunks (whole layers) of `rpt` consecutive row-shards of one
// layout: a warp streams through their samples, which lie one after the other in the list, with U*NS loads in flight
// whatever row-shard they belong to, and closes a row-shard when its last sample has been added.  Bound by its
// instructions before it is by L2: row-shards hold 8.5 samples on average on large, and loops over one row-shard, or
// one strip, at a time took 127 to 175 us for 256 layouts (46 instructions per sample and strip; 20 per sample and three strips here).
template <int NS, int U>
__global__ void __launch_bounds__(EVAL_THREADS, NS == 1 ? 4 : (NS == 2 ? 3 : 2))
k_eval_sum(const EvalArgs A, int n, int sgroups, int rpt, bool sum32)
{
    const RpDims &dm = A.dm;
    const int lane = threadIdx.x & 31, RG = dm.RG, rc = dm.LP >> 2;
    const bool vec = eval_vec(dm);
    const int groups = (RG + rpt - 1) / rpt, per = groups * sgroups;
    const int cpl = dm.P >> 2, used = vec ? (32 / cpl) * cpl : 32;
    for (unsigned task = blockIdx.x * (EVAL_THREADS / 32) + (threadIdx.x >> 5); task < (unsigned)n * (unsigned)per; task += gridDim.x * (EVAL_THREADS / 32)) {
        const int lay = (int)(task / (unsigned)per), r = (int)(task - (unsigned)lay * per), sg = r % sgroups, rg0 = r / sgroups * rpt, nr = min(rpt, RG - rg0);
        const u32 *go = A.off + (size_t)lay * (RG + 1) + rg0;
        const unsigned short *list = A.list + (size_t)lay * dm.N;
        const int ends = (int)(__ldg(go + min(lane + 1, nr)) & 0xffffu), s0 = (int)(__ldg(go) & 0xffffu);        // lane x: where row-shard rg0 + x ends
        if (!vec) {
            int m0 = s0;
            for (int x = 0; x < nr; ++x) {
                const int m1 = __shfl_sync(0xffffffffu, ends, x);
                int *wout = A.W_out ? A.W_out + ((size_t)lay * RG + rg0 + x) * dm.LP : nullptr;
                const i64 es = rp_warp_layer_max_sum(dm, lane, [&](int e) {
                    int sum = 0;
                    for (int m = m0; m < m1; ++m) sum += __ldg(A.q + (size_t)__ldg(list + m) * dm.LP + e);
                    if (wout) wout[e] = sum;
                    return sum;
                });
                if (lane == 0) A.cost[(size_t)lay * RG + rg0 + x] += dm.EC * es;
                m0 = m1;
            }
            continue;
        }
        int4 a[NS];
        const int4 *col[NS];                // (lanes and strips past the row's end read its first chunk and are ignored)
        unsigned on = 0;
#pragma unroll
        for (int z = 0; z < NS; ++z) {
            const int c = (sg * NS + z) * used + lane;
            a[z] = make_int4(0, 0, 0, 0);
            if (lane < used && c < rc) on |= 1u << z;
            col[z] = (const int4 *)A.q + (((on >> z) & 1u) ? c : 0);
        }
        const int s1 = __shfl_sync(0xffffffffu, ends, nr - 1);
        int x = 0, end = __shfl_sync(0xffffffffu, ends, 0);
        auto close = [&]() {                // row-shard rg0 + x is complete
            const size_t at = (size_t)lay * RG + rg0 + x;
            u32 own = 0, high = 0;          // sum of this lane's layers (see eval_launch); where it may pass 32 bits, its 16-bit halves
#pragma unroll
            for (int z = 0; z < NS; ++z) {
                const bool o = (on >> z) & 1u;
                if (A.W_out && o) ((int4 *)(A.W_out + at * dm.LP))[(sg * NS + z) * used + lane] = a[z];
                const int m = eval_layer_max(o ? max(max(a[z].x, a[z].y), max(a[z].z, a[z].w)) : 0, lane, cpl);
                const u32 v = o && lane % cpl == 0 ? (u32)m : 0u;
                if (sum32) own += v;
                else { own += v & 0xffffu; high += v >> 16; }
                a[z] = make_int4(0, 0, 0, 0);
            }
            i64 es = (i64)__reduce_add_sync(0xffffffffu, own);
            if (!sum32) es += (i64)__reduce_add_sync(0xffffffffu, high) << 16;
            if (lane == 0) atomicAdd((u64 *)A.cost + at, (u64)(dm.EC * es));
            ++x;
            end = __shfl_sync(0xffffffffu, ends, x);
        };
        int next = s0 + lane < s1 ? (int)__ldg(list + s0 + lane) : 0;
        for (int p = s0; p < s1; p += 32) {
            const int id = next, nm = min(32, s1 - p);
            next = p + 32 + lane < s1 ? (int)__ldg(list + p + 32 + lane) : 0;
            for (int y = 0; y < nm; y += U) {
                int4 v[U][NS];
#pragma unroll
                for (int u = 0; u < U; ++u) {               // (past the end: sample 0, not counted)
                    const size_t at = (size_t)(u32)__shfl_sync(0xffffffffu, id, y + u) * (u32)rc;
#pragma unroll
                    for (int z = 0; z < NS; ++z) v[u][z] = __ldg(col[z] + at);
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (y + u < nm) {
                        while (p + y + u == end) close();
#pragma unroll
                        for (int z = 0; z < NS; ++z) { a[z].x += v[u][z].x; a[z].y += v[u][z].y; a[z].z += v[u][z].z; a[z].w += v[u][z].w; }
                    }
                }
            }
        }
        while (x < nr) close();             // the last ones (no sample lies beyond s1)
    }
}

// Of 32 lanes' non-negative numbers: the largest, by its upper and its lower word; the sum (below 2^63), 21 bits of each at a time.
__device__ __forceinline__ i64 few_warp_max(i64 v)
{
    const u32 hi = (u32)((u64)v >> 32), mh = __reduce_max_sync(0xffffffffu, hi);
    return (i64)(((u64)mh << 32) | __reduce_max_sync(0xffffffffu, hi == mh ? (u32)v : 0u));
}
__device__ __forceinline__ i64 few_warp_sum(i64 v)
{
    const u64 lo = __reduce_add_sync(0xffffffffu, (u32)v & 0x1fffffu), mid = __reduce_add_sync(0xffffffffu, (u32)(v >> 21) & 0x1fffffu),
              hi = __reduce_add_sync(0xffffffffu, (u32)(v >> 42));
    return (i64)(lo + (mid << 21) + (hi << 42));
}

// Many layouts, last kernel: the scores from the row-shards' costs, and what is left of the blob.
__global__ void __launch_bounds__(EVAL_THREADS)
k_eval_score(const EvalArgs A)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    const RpDims &dm = A.dm;
    i64 *U = (i64 *)smraw;                                               // [G]
    __shared__ i64 top_s[EVAL_THREADS / 32];
    const int tid = threadIdx.x, lane = tid & 31, lay = blockIdx.x;
    i64 *cost = A.cost + (size_t)lay * dm.RG;
    char *b = A.blob_out ? A.blob_out + (size_t)lay * A.bl.bytes : nullptr;
    for (int g = tid; g < dm.G; g += EVAL_THREADS) U[g] = 0;
    __syncthreads();
    i64 top = 0;
    for (int rg = tid; rg < dm.RG; rg += EVAL_THREADS) {
        const i64 J = __ldcg(cost + rg);
        cost[rg] = 0;
        top = J > top ? J : top;
        atomicAdd((u64 *)&U[rg % dm.G], (u64)J);
        if (b) {
            ((i64 *)(b + A.bl.off_Jfx))[rg] = J;
            ((i64 *)(b + A.bl.off_Esum))[rg] = (J - ((const i64 *)(b + A.bl.off_Afx))[rg]) / dm.EC;
        }
    }
    top = few_warp_max(top);
    if (lane == 0) top_s[tid >> 5] = top;
    const int wrong = A.tickets[lay];
    __syncthreads();
    if (tid == 0) A.tickets[lay] = 0;
    if (A.host) {          // coverage is checked by the caller's `bad` flag: every sample sits in one cell by construction
        if (tid < 8) A.host[tid] = A.counters[tid];
        if (tid < 3) { A.host[16 + tid] = A.inc_score[tid]; A.host[22 + tid] = A.seed_score[tid]; }
        if (tid < RP_SW_COUNT) ((int *)(A.host + 56))[tid] = A.status[tid] | (tid == RP_SW_VALIDATE && wrong ? 1 : 0);
        if (A.layout_host) for (int i = tid; i < dm.N; i += EVAL_THREADS) A.layout_host[i] = __ldg(A.lay32 + i);
    }
    if (b) for (int g = tid; g < dm.G; g += EVAL_THREADS) ((i64 *)(b + A.bl.off_U))[g] = U[g];
    if (tid >= 32) return;
    const bool refused = A.bad_dev && __ldcg(A.bad_dev);
    i64 s0 = 0, s1 = 0, s2 = lane < EVAL_THREADS / 32 ? top_s[lane] : 0;
    for (int g = lane; g < dm.G; g += 32) { const i64 u = U[g]; s1 += u; s0 = u > s0 ? u : s0; }
    for (int o = 16; o; o >>= 1) s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    s0 = few_warp_max(s0); s2 = few_warp_max(s2);
    if (lane == 0) {
        const i64 sc[3] = { s0, s1, s2 };
        for (int x = 0; x < 3; ++x) {
            if (refused) continue;
            if (A.score_out) A.score_out[(size_t)lay * 3 + x] = sc[x];
            if (A.score_out2) A.score_out2[(size_t)lay * 3 + x] = sc[x];
            if (A.f64_out) A.f64_out[(size_t)lay * 3 + x] = (double)sc[x] / (double)dm.SC;
        }
        if (b) { i64 *S = (i64 *)(b + A.bl.off_S); S[0] = s0; S[1] = s1; S[2] = s2; S[3] = rp_energy(s0, s1, s2); }
    }
}

// grid = (MS, row-shards, layouts), clusters of MS CTAs along x: CTA x of a row-shard takes the samples of
// range x, then the layers of range x of the summed row.  The row-shard's cell statistics and cost are worked out by its own
// cluster beside the sums, so that what is left for the CTA that finishes a layout is a sum over its row-shards (with the statistics of
// all samples added up there, one CTA took two thirds of the time on heavy's 8192; with the one launch of the metrics behind it a call
// of rp_diagnostics on heavy 90 -> 47 us).  Where there are more CTAs than the SMs hold it matters how many those are: 48 registers
// and five to an SM (the loop over the cluster's sums unrolled twice; 62 and four when it and the statistics were unrolled four times: two
// layouts of 2048 samples in 240 row-shards 38.4 and 32.4 us, 69 of 401 in ten 53.4 and 48.3).
static inline size_t eval_few_smem(const RpDims &dm, int MS)
{
    const size_t part = (sizeof(int) * ((size_t)dm.LP + dm.N / MS + 2) + 7) & ~(size_t)7;
    return std::max(part + (size_t)16 * dm.D, (size_t)8 * dm.RG);
}
template <bool WIDE>            // more than 32 chunks in a layer
__global__ void __launch_bounds__(EVAL_THREADS)
k_eval_few(const EvalArgs A)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    rp_let_next_launch_start();                                          // (the diagnostics' coefficients need nothing of this)
    const RpDims &dm = A.dm;
    const cg::cluster_group cl = cg::this_cluster();
    const int MS = gridDim.x, ms = blockIdx.x, rg = blockIdx.y, lay = blockIdx.z;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = EVAL_THREADS / 32;
    int *part = (int *)smraw;                                           // [LP] this CTA's share of the sum
    int *list = part + dm.LP;                                           // [N / MS + 1] its samples
    u64 *Q = (u64 *)(smraw + ((sizeof(int) * ((size_t)dm.LP + dm.N / MS + 2) + 7) & ~(size_t)7));      // [D] statistics of the row's cells on
    int *T = (int *)(Q + dm.D), *cnt = T + dm.D;                        // this shard, by slot
    __shared__ int n_s, last_s, wrong_s;
    __shared__ i64 of_warp[3][EVAL_THREADS / 32], es_of[8];                      // (a place a warp: 64-bit additions to one address queue up)
    const EvalCells cells = eval_cells(A, lay);
    char *b = A.blob_out ? A.blob_out + (size_t)lay * A.bl.bytes : nullptr;
    if (tid == 0) n_s = 0;
    const int row = rg / dm.G, g = rg % dm.G, first = row * dm.D;
    // (a slot of another shard has a negative count: which slots are the row-shard's is looked up in global memory only here)
    for (int d = tid; d < dm.D; d += EVAL_THREADS) { Q[d] = 0; T[d] = 0; cnt[d] = __ldg(A.edp + d) == g ? 0 : (int)0x80000000; }
    __syncthreads();
    const int i0 = (int)((long long)dm.N * ms / MS), i1 = (int)((long long)dm.N * (ms + 1) / MS);
#pragma unroll 8
    for (int i = i0 + tid; i < i1; i += EVAL_THREADS) {
        const int c = eval_cell(A, cells, i), d = c - first;
        if ((unsigned)d >= (unsigned)dm.D || cnt[d] < 0) continue;
        const int ti = __ldg(A.t + i);
        list[atomicAdd(&n_s, 1)] = i;
        atomicAdd(&T[d], ti); atomicAdd(&cnt[d], 1);
        few_add_square(&Q[d], ti, A.q_halves);
        if (b) ((unsigned short *)(b + A.bl.off_cell))[i] = (unsigned short)c;
    }
    if (A.layout_host && rg == 0) for (int i = i0 + tid; i < i1; i += EVAL_THREADS) A.layout_host[i] = __ldg(A.lay32 + i);
    __syncthreads();
    const int cpl = dm.P >> 2, rc = dm.LP >> 2, n = n_s;
    for (int c0 = 32 * warp; c0 < rc; c0 += 32 * nwarps) {
        const int c = c0 + lane;
        const int4 a = eval_sum_column<16>((const int4 *)A.q + (c < rc ? c : 0), rc, list, 0, n);
        if (c < rc) ((int4 *)part)[c] = a;
    }
    cl.sync();
    const int l0 = dm.L * ms / MS, l1 = dm.L * (ms + 1) / MS, lps = WIDE ? 1 : 32 / cpl, used = WIDE ? 32 : lps * cpl;
    int4 *wout = A.W_out ? (int4 *)(A.W_out + ((size_t)lay * dm.RG + rg) * dm.LP) : nullptr;
    i64 es = 0;
    if (WIDE) {                                           // a layer per warp
        for (int l = l0 + warp; l < l1; l += nwarps) {
            int m = 0;
            for (int c = l * cpl + lane; c < (l + 1) * cpl; c += 32) {
                int4 a = make_int4(0, 0, 0, 0);
                for (int x = 0; x < MS; ++x) {
                    const int4 v = ((const int4 *)cl.map_shared_rank(part, x))[c];
                    a.x += v.x; a.y += v.y; a.z += v.z; a.w += v.w;
                }
                if (wout) wout[c] = a;
                m = max(m, max(max(a.x, a.y), max(a.z, a.w)));
            }
            m = __reduce_max_sync(0xffffffffu, m);
            if (lane == 0) es += m;
        }
    } else
    for (int c0 = l0 * cpl + warp * used; c0 < l1 * cpl; c0 += nwarps * used) {
        const int c = c0 + lane;
        const bool on = lane < used && c < l1 * cpl;
        int4 a = make_int4(0, 0, 0, 0);
        if (on)
#pragma unroll 2
            for (int x = 0; x < MS; ++x) {
                const int4 v = ((const int4 *)cl.map_shared_rank(part, x))[c];
                a.x += v.x; a.y += v.y; a.z += v.z; a.w += v.w;
            }
        if (wout && on) wout[c] = a;
        const int m = eval_layer_max(on ? max(max(a.x, a.y), max(a.z, a.w)) : 0, lane, cpl);
        if (on && lane % cpl == 0) es += m;
    }
    es = few_warp_sum(es);
    if (lane == 0) of_warp[0][warp] = es;
    // Statistics of all of the cluster's samples meet in its first CTA: a lane there for every CTA of a slot, which fetches; more slots
    // than it has lanes for are added to it from afar (diagnostics of 6000 samples in four row-shards of 256 slots 56.5 us fetched, 55 so).
    if (dm.D * MS <= EVAL_THREADS) {
        if (ms == 0 && MS > 1) {
            const int d = tid / MS, x = tid & (MS - 1);
            const bool on = d < dm.D && cnt[d < dm.D ? d : 0] >= 0;
            int t = 0, m = 0;
            u64 q = 0;
            if (on) { t = cl.map_shared_rank(T, x)[d]; m = cl.map_shared_rank(cnt, x)[d]; q = cl.map_shared_rank(Q, x)[d]; }
            for (int o = 1; o < MS; o <<= 1) {
                t += __shfl_xor_sync(0xffffffffu, t, o); m += __shfl_xor_sync(0xffffffffu, m, o); q += __shfl_xor_sync(0xffffffffu, q, o);
            }
            if (on && x == 0) { T[d] = t; cnt[d] = m; Q[d] = q; }
        }
    } else if (ms) {
        int *T0 = cl.map_shared_rank(T, 0), *cnt0 = cl.map_shared_rank(cnt, 0);
        u64 *Q0 = cl.map_shared_rank(Q, 0);
        for (int d = tid; d < dm.D; d += EVAL_THREADS)
            if (cnt[d] > 0) { atomicAdd(T0 + d, T[d]); atomicAdd(cnt0 + d, cnt[d]); few_add(Q0 + d, (u32)Q[d], (u32)(Q[d] >> 32), A.q_halves); }
    }
    __syncthreads();
    if (tid == 0) {
        i64 sum = 0;
#pragma unroll
        for (int w = 0; w < EVAL_THREADS / 32; ++w) sum += of_warp[0][w];
        cl.map_shared_rank(es_of, 0)[ms] = sum;
    }
    cl.sync();                                            // nobody reads another CTA's shared memory from here on
    if (ms) return;
    if (b)
        for (int d = tid; d < dm.D; d += EVAL_THREADS) {
            if (cnt[d] < 0) continue;
            ((u64 *)(b + A.bl.off_Q))[first + d] = few_square(Q[d], A.q_halves);
            ((int *)(b + A.bl.off_T))[first + d] = T[d];
            ((int *)(b + A.bl.off_cnt))[first + d] = cnt[d];
        }
    if (warp == 0) {
        i64 Af = 0, E = 0;
        for (int x = 0; x < MS; ++x) E += es_of[x];
        bool wrong = false;
        for (int d = lane; d < dm.D; d += 32) wrong |= cnt[d] == 0 || (cnt[d] > 0 && T[d] > dm.C);
        wrong = __any_sync(0xffffffffu, wrong);
        for (int s = 0; s < dm.S; ++s) {
            const i64 ca = dm.ahat[s] * dm.C, cb = dm.bhat[s];
            i64 v = 0;
            for (int d = lane; d < dm.D; d += 32) { const i64 w = cnt[d] < 0 ? 0 : ca * T[d] + cb * (i64)few_square(Q[d], A.q_halves); v = w > v ? w : v; }
            Af += few_warp_max(v);
        }
        if (lane == 0) {
            const i64 J = Af + dm.EC * E;
            if (b) {
                ((i64 *)(b + A.bl.off_Esum))[rg] = E; ((i64 *)(b + A.bl.off_Afx))[rg] = Af; ((i64 *)(b + A.bl.off_Jfx))[rg] = J;
                if (A.bl.off_wtab >= 0) ((int *)(b + A.bl.off_wtab))[rg] = (A.first + lay) * dm.RG + rg;      // the pool holds the call's layouts as RG slices each
            }
            A.cost[(size_t)lay * dm.RG + rg] = J;
            __threadfence();
            // arrivals in the lower half, row-shards with an empty or overfull cell in the upper one
            const unsigned before = atomicAdd((unsigned *)&A.tickets[lay], 1u | (wrong ? 1u << 16 : 0u));
            last_s = (before & 0xffffu) == (unsigned)dm.RG - 1;
            if (last_s) { wrong_s = wrong || before >> 16; A.tickets[lay] = 0; }
        }
    }
    __syncthreads();
    if (!last_s) return;
    __threadfence();
    // costs of the row-shards on chip, one trip; a thread adds up a shard's rows
    i64 *Js = (i64 *)smraw;                                              // [RG]
    i64 top = 0, sum = 0, most = 0;
    {
        i64 *eg = A.cost + (size_t)lay * dm.RG;
#pragma unroll 4
        for (int x = tid; x < dm.RG; x += EVAL_THREADS) {
            const i64 J = __ldcg(eg + x);
            eg[x] = 0;
            Js[x] = J;
            top = J > top ? J : top;
        }
    }
    __syncthreads();
    for (int x = tid; x < dm.G; x += EVAL_THREADS) {
        i64 u = 0;
#pragma unroll 4
        for (int r = 0; r < dm.R; ++r) u += Js[r * dm.G + x];
        sum += u; most = u > most ? u : most;
        if (b) ((i64 *)(b + A.bl.off_U))[x] = u;
    }
    top = few_warp_max(top); most = few_warp_max(most); sum = few_warp_sum(sum);
    if (lane == 0) { of_warp[0][warp] = most; of_warp[1][warp] = sum; of_warp[2][warp] = top; }
    __syncthreads();
    i64 sc[3] = { 0, 0, 0 };
#pragma unroll
    for (int w = 0; w < EVAL_THREADS / 32; ++w) {
        const i64 m = of_warp[0][w], n = of_warp[2][w];
        sc[0] = m > sc[0] ? m : sc[0]; sc[1] += of_warp[1][w]; sc[2] = n > sc[2] ? n : sc[2];
    }
    if (A.host) {          // coverage is checked by the caller's `bad` flag: every sample sits in one cell by construction
        if (tid < 8) A.host[tid] = A.counters[tid];
        if (tid < 3) { A.host[16 + tid] = A.inc_score[tid]; A.host[22 + tid] = A.seed_score[tid]; }
        if (tid < RP_SW_COUNT) ((int *)(A.host + 56))[tid] = A.status[tid] | (tid == RP_SW_VALIDATE && wrong_s ? 1 : 0);
    }
    if (tid < 3) {
        const i64 v = tid == 0 ? sc[0] : (tid == 1 ? sc[1] : sc[2]);
        if (A.score_out) A.score_out[(size_t)lay * 3 + tid] = v;
        if (A.score_out2) A.score_out2[(size_t)lay * 3 + tid] = v;
        if (A.f64_out) A.f64_out[(size_t)lay * 3 + tid] = (double)v / (double)dm.SC;
        if (b) { i64 *S = (i64 *)(b + A.bl.off_S); S[tid] = v; if (tid == 0) S[3] = rp_energy(sc[0], sc[1], sc[2]); }
    }
    if (!A.score_final && !A.f64_final) return;
    if (tid < 32) __threadfence();
    __syncthreads();
    if (A.n > 1) {
        if (tid == 0) {
            last_s = (atomicAdd(&A.tickets[A.n], 1) == A.n - 1);
            if (last_s) A.tickets[A.n] = 0;
        }
        __syncthreads();
        if (!last_s) return;
        __threadfence();
    }
    if (__ldcg(A.bad_dev)) return;
#pragma unroll 4
    for (int x = tid; x < 3 * A.n; x += EVAL_THREADS) {
        if (A.score_final) A.score_final[x] = __ldcg(A.score_out + x);
        if (A.f64_final) A.f64_final[x] = __ldcg(A.f64_out + x);
    }
}

// Windows are scored up to this measure of their size.  It is the shared memory of a scoring kernel that is gone, no kernel here needs as much,
// and stays as what callers have been told: what was refused with RP_ERR_RANGE is refused.
static size_t eval_smem_bytes(const RpDims &dm)
{
    const size_t cells = (sizeof(u64) * dm.K + sizeof(i64) * (2 * (size_t)dm.RG + dm.G) + sizeof(int) * 2 * (size_t)dm.K + 2 * (size_t)dm.N + 15) & ~(size_t)15;
    return (cells + sizeof(int) * (2 * (size_t)dm.RG + 1 + dm.N) + 15) & ~(size_t)15;
}

// Whether n layouts take the few-layouts form.  It has a cluster per row-shard and layout, which scans the whole assignment; the other
// form groups an assignment once, but in one CTA, and has three launches where this has one.  Both add up the same rows, so that what counts
// is the scans (left) against the grouping, the launches and the slices' loading (right); drawn through 1760 calls of 900 windows timed in both
// forms, the chosen one is 0.8 % above the better one on average.  Calls in us, few and many: 512 samples in 32 row-shards, 16 layers of 8
// ranks, n = 8 37.0 and 36.6, 64 49 and 37, 512 204 and 54; 2048 in 240, 24 of 16, n = 4 36.9 and 41.5, 6 44.7 and 42.5, 64 172 and 54; 1808 in
// 18, 28 of 32, n = 27 54 and 70; 227 in 6, 30 of 32, n = 53 34 and 42; 5430 in 32, 32 chunks a row, n = 32 98 and 142; 4000 in 6, 16 of 8, n = 64
// 96 and 138, 128 148 and 141, 512 307 and 233; 8192 in 448, 24 of 16 (no slice on chip), n = 2 63 and 95; 30000 in 160, n = 3 142 and 270, 4 335
// and 267.  (With the rows among the scans, and no row-shards on the right: 1.3 % above on average, 1.4 times at worst where few row-shards are
// long.)  One layout: 8192 in 448 47.6 and 94, 4000 in 2000 44.8 and 46.3, 8000 in 1920 51.8 and 71.
static bool eval_is_few(const RpDims &dm, int n)
{
    if ((dm.P & 3) || n >= 65536 || dm.RG >= 65536 || dm.LP > 16384 || eval_few_smem(dm, 8) > EVAL_SMEM_MAX) return false;
    const double N = dm.N, RG = dm.RG;
    if (n == 1) return RG * N <= 5e6;
    return n * RG * (8.5 + N / 480.0) <= 5e3 + 2.8 * std::min(N, 1e4) + 38.0 * RG + dm.LP;
}
size_t rp_eval_list_len(const RpDims &dm, int n) { return eval_is_few(dm, n) ? 0 : (size_t)n * dm.N; }
size_t rp_eval_off_len(const RpDims &dm, int n) { return eval_is_few(dm, n) ? 0 : (size_t)n * (dm.RG + 1); }

// The scratch (Esum, tickets) is zero before and after a launch.
static int eval_launch(rp_ctx *c, EvalArgs &A, int n)
{
    const RpDims &dm = c->dm;
    if (eval_smem_bytes(dm) > EVAL_SMEM_MAX) return RP_ERR_RANGE;
    A.dm = dm; A.bl = c->bl; A.t = c->d_t; A.q = c->d_q; A.edp = c->d_edp; A.dp_list = c->d_dp_list; A.dp_off = c->d_dp_off;
    A.n = n;
    A.q_halves = (double)dm.C * (double)c->tokens < 281474976710656.0;         // (and N < 65536: see eval_smem_bytes)
    if (eval_is_few(dm, n)) {
        int MS = 1;
        while (MS < 8 && (long long)n * dm.RG * MS < 148 * 4 && dm.N >= 64 * MS) MS *= 2;
        while (MS < 8 && eval_few_smem(dm, MS) > EVAL_SMEM_MAX) MS *= 2;
        const size_t sm = eval_few_smem(dm, MS);
        auto few = eval_vec(dm) ? k_eval_few<false> : k_eval_few<true>;
        if (sm > 32 * 1024) RP_CUDA(cudaFuncSetAttribute(few, cudaFuncAttributeMaxDynamicSharedMemorySize, EVAL_SMEM_MAX));
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(MS, dm.RG, n); cfg.blockDim = dim3(EVAL_THREADS);
        cfg.dynamicSmemBytes = sm; cfg.stream = c->stream;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = MS; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
        cfg.attrs = at; cfg.numAttrs = 1;
        RP_CUDA(cudaLaunchKernelEx(&cfg, few, A));
    } else {
        const size_t gm = eval_group_bytes(dm), fm = sizeof(i64) * (size_t)dm.G;
        if (gm > EVAL_SMEM_MAX || dm.N > 65535) return RP_ERR_RANGE;
        if (gm > 32 * 1024) RP_CUDA(cudaFuncSetAttribute(k_eval_group, cudaFuncAttributeMaxDynamicSharedMemorySize, EVAL_SMEM_MAX));
        if (fm > 32 * 1024) RP_CUDA(cudaFuncSetAttribute(k_eval_score, cudaFuncAttributeMaxDynamicSharedMemorySize, EVAL_SMEM_MAX));
        const int cpl = dm.P >> 2, used = eval_vec(dm) ? 32 / cpl * cpl : 32, strips = eval_vec(dm) ? ((dm.LP >> 2) + used - 1) / used : 1;
        const int ns = std::min(3, strips), sgroups = (strips + ns - 1) / ns, warps = ns == 1 ? 32 : (ns == 2 ? 24 : 16);     // per SM
        // What a warp adds up for a row-shard: the busiest loads of its layers, each at most k times the tokens of the window
        // (a layout handed in may put them all into one cell).
        const bool sum32 = eval_vec(dm) && (double)std::min(dm.L, ns * used / cpl) * dm.k * (double)c->tokens < 4294967296.0;
        if (A.score_final) A.score_out = A.score_final;
        if (A.f64_final) A.f64_out = A.f64_final;
        auto part = [&](int first) {                       // (16384 layouts: bounds the task numbers of a launch)
            EvalArgs B = A;
            B.first = first;
            if (B.lay32) B.lay32 += (size_t)first * dm.N; else B.src += first;
            if (B.W_out) B.W_out += (size_t)first * dm.RG * dm.LP;
            if (B.blob_out) B.blob_out += (size_t)first * c->bl.bytes;
            if (B.score_out) B.score_out += 3 * (size_t)first;
            if (B.f64_out) B.f64_out += 3 * (size_t)first;
            B.cost += (size_t)first * dm.RG; B.tickets += first; B.list += (size_t)first * dm.N; B.off += (size_t)first * (dm.RG + 1);
            return B;
        };
        const SlicePlan S = eval_slice_plan(dm, std::min(n, 16384));
        auto slice = S.tw == 1 ? k_eval_slice<1> : S.tw == 2 ? k_eval_slice<2> : S.tw == 4 ? k_eval_slice<4> : k_eval_slice<8>;
        if (S.tw) RP_CUDA(cudaFuncSetAttribute(slice, cudaFuncAttributeMaxDynamicSharedMemorySize, EVAL_SMEM_MAX));
        for (int first = 0; first < n; first += 16384) {
            k_eval_group<<<std::min(16384, n - first), GROUP_THREADS, gm, c->stream>>>(part(first), S.tw != 0);
            ++g_rp_launches;
        }
        for (int first = 0; first < n; first += 16384) {
            const EvalArgs B = part(first);
            const int m = std::min(16384, n - first);
            if (S.tw) {
                SlicePlan P = S;
                P.groups = std::min(P.groups, m);
                slice<<<P.slices * P.groups, SLICE_THREADS, P.smem, c->stream>>>(B, P, m);
                k_eval_score<<<m, EVAL_THREADS, fm, c->stream>>>(B);
                g_rp_launches += 2;
                continue;
            }
            // several tasks for each warp the SMs hold, of at most 31 row-shards
            const int rpt = (int)std::max<long long>(1, std::min<long long>(31, (long long)m * dm.RG * sgroups / (148 * warps * 6)));
            const long long want = ((long long)m * ((dm.RG + rpt - 1) / rpt) * sgroups + 7) / 8;
            const int grid = (int)std::min<long long>(want, 148 * warps / 8);
            if (ns == 1) k_eval_sum<1, 8><<<grid, EVAL_THREADS, 0, c->stream>>>(B, m, sgroups, rpt, sum32);
            else if (ns == 2) k_eval_sum<2, 4><<<grid, EVAL_THREADS, 0, c->stream>>>(B, m, sgroups, rpt, sum32);
            else k_eval_sum<3, 4><<<grid, EVAL_THREADS, 0, c->stream>>>(B, m, sgroups, rpt, sum32);
            k_eval_score<<<m, EVAL_THREADS, fm, c->stream>>>(B);
            g_rp_launches += 2;
        }
        --g_rp_launches;                                   // (one is counted below)
    }
    ++g_rp_launches;
    RP_CUDA(cudaGetLastError());
    return RP_OK;
}

// n layouts lay [n][N] (null: the assignments of the current buffer's blobs that src names) with the context's scratch.
// score_final, f64_final: see EvalArgs; score_out / f64_out are then scratch.
int rp_launch_eval(rp_ctx *c, const int *lay, const int *src, int n, int *W_out, char *blob_out, i64 *score_out, double *f64_out,
                   i64 *score_final, double *f64_final)
{
    EvalArgs A = {};
    A.lay32 = lay; A.blobs = c->buf[c->cur].blob; A.src = src;
    A.W_out = W_out; A.blob_out = blob_out; A.score_out = score_out; A.f64_out = f64_out;
    A.bad = rp_pin_bad(c);
    if (score_final || f64_final) { A.score_final = score_final; A.f64_final = f64_final; A.bad_dev = c->d_status + RP_SW_BAD_LAYOUT; }
    A.cost = c->d_eval_Esum; A.tickets = c->d_eval_tickets; A.list = c->d_eval_list; A.off = (u32 *)c->d_eval_off;
    return eval_launch(c, A, n);
}

// One layout with the population's own scratch.
static void eval_one(rp_ctx *c, EvalArgs &A)
{
    A.bad = rp_pin_bad(c);
    A.cost = c->d_one_Esum; A.tickets = c->d_one_ticket; A.list = c->d_one_list; A.off = (u32 *)c->d_one_off;
}
int rp_launch_eval_seed(rp_ctx *c)
{
    EvalArgs A = {};
    eval_one(c, A);
    A.lay32 = c->d_seed_layout; A.W_out = c->d_W; A.blob_out = c->buf[0].blob; A.score_out = c->d_inc_score; A.score_out2 = c->d_seed_score;
    return eval_launch(c, A, 1);
}
// Validate(x*) and the full rescoring of the incumbent; the results go to the pinned block (see EvalArgs::host).
int rp_launch_eval_incumbent(rp_ctx *c)
{
    EvalArgs A = {};
    eval_one(c, A);
    A.lay32 = c->d_inc_layout;
    A.score_out = c->h_pin + 19; A.f64_out = (double *)(c->h_pin + 25);
    A.host = c->h_pin; A.counters = c->d_counters; A.inc_score = c->d_inc_score; A.seed_score = c->d_seed_score; A.status = c->d_status;
    A.layout_host = rp_mail_layout(c);
    return eval_launch(c, A, 1);
}

// ---------------------------------------------------------------------------------------------
// Layout of the chain-state blob and of the per-plan static tables; the static block itself.
// ---------------------------------------------------------------------------------------------
void rp_make_layouts(const RpDims &dm, RpBlob *bl, RpStatic *sl)
{
    int o = 0;
    bl->off_Q = o;    o += 8 * dm.K;
    bl->off_Esum = o; o += 8 * dm.RG;
    bl->off_Afx = o;  o += 8 * dm.RG;
    bl->off_Jfx = o;  o += 8 * dm.RG;
    bl->off_U = o;    o += 8 * dm.G;
    bl->off_S = o;    o += 8 * 4;
    bl->off_T = o;    o += 4 * dm.K;
    bl->off_cnt = o;  o += 4 * dm.K;
    bl->off_cell = o; o += 2 * dm.N;
    bl->off_wtab = -1;
    if (rp_uses_slices(dm)) { o = (o + 3) & ~3; bl->off_wtab = o; o += 4 * dm.RG; }
    bl->bytes = (o + 15) & ~15;
    sl->t_staged = dm.N <= 2048;
    o = 0;
    sl->off_dpl = o;  o += 4 * dm.D;
    sl->off_dpo = o;  o += 4 * (dm.G + 1);
    sl->off_t = o;    o += sl->t_staged ? 4 * dm.N : 0;
    sl->off_rg = o;   o += 2 * dm.K;
    sl->off_g = o;    o += 2 * dm.K;
    sl->off_row = o;  o += 2 * dm.K;
    sl->bytes = (o + 15) & ~15;
}

// A fresh population in one launch: the static tables; every member descends from slot 0, whose rank loads sit in cell 0 and
// are copied into a cell of the member's own (P + m) at level 0; the seed is the incumbent; counters, scratch and the
// slices' holder counts at zero.
struct SetupArgs {
    RpDims dm;
    RpStatic sl;
    const int *t, *edp, *dp_list, *dp_off, *seed_layout;
    char *blk;
    int P, *anc, *wloc, *wloc_next, *done, *inc_layout, *one_ticket, *wcount, *undecided, *inc_slot, *sync, *status;
    i64 *one_Esum, *counters;
    u64 *emin;
};
__global__ void __launch_bounds__(256)
k_setup_population(const SetupArgs A)
{
    const RpDims &dm = A.dm;
    const RpStatic &sl = A.sl;
    const int tid = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
    for (int d = tid; d < dm.D; d += nt) ((int *)(A.blk + sl.off_dpl))[d] = A.dp_list[d];
    for (int g = tid; g <= dm.G; g += nt) ((int *)(A.blk + sl.off_dpo))[g] = A.dp_off[g];
    if (sl.t_staged) for (int i = tid; i < dm.N; i += nt) ((int *)(A.blk + sl.off_t))[i] = A.t[i];
    for (int c = tid; c < dm.K; c += nt) {
        const int r = c / dm.D, g = A.edp[c % dm.D];
        ((unsigned short *)(A.blk + sl.off_rg))[c] = (unsigned short)(r * dm.G + g);
        ((unsigned short *)(A.blk + sl.off_g))[c] = (unsigned short)g;
        ((unsigned short *)(A.blk + sl.off_row))[c] = (unsigned short)(r * dm.D);
    }
    for (int m = tid; m < A.P; m += nt) { A.anc[m] = 0; A.wloc[m] = 0; A.wloc_next[m] = A.P + m; }
    for (int i = tid; i < dm.N; i += nt) A.inc_layout[i] = A.seed_layout[i];
    for (int x = tid; x < dm.RG + 3; x += nt) A.one_Esum[x] = 0;      // (three sums of the diagnostics behind them)
    for (int x = tid; x <= A.P; x += nt) A.sync[x] = 0;
    if (A.wcount) for (size_t x = tid; x < 2 * (size_t)A.P * dm.RG; x += nt) A.wcount[x] = 0;
    if (tid < 7) A.counters[tid] = 0;                      // (the eighth is the window's token total)
    if (tid < RP_SW_COUNT) A.status[tid] = 0;
    if (tid == 0) { *A.done = 0; *A.one_ticket = 0; *A.undecided = 0; *A.inc_slot = -1; *A.emin = ~0ull >> 1; }
}

int rp_launch_setup_population(rp_ctx *c)
{
    const RpDims &dm = c->dm;
    SetupArgs A = {};
    A.dm = dm; A.sl = c->sl; A.t = c->d_t; A.edp = c->d_edp; A.dp_list = c->d_dp_list; A.dp_off = c->d_dp_off; A.seed_layout = c->d_seed_layout;
    A.blk = c->d_static; A.P = c->Ppop; A.anc = c->d_anc; A.wloc = c->d_wloc; A.wloc_next = c->d_wloc_next; A.done = c->d_done;
    A.inc_layout = c->d_inc_layout; A.one_ticket = c->d_one_ticket; A.wcount = c->d_wcount; A.undecided = c->d_undecided;
    A.inc_slot = c->d_inc_slot; A.sync = c->d_sync; A.status = c->d_status; A.one_Esum = c->d_one_Esum; A.counters = c->d_counters;
    A.emin = c->d_F + 2 * (size_t)c->Ppop;
    const size_t most = std::max((size_t)std::max(c->Ppop + 1, dm.N), c->d_wcount ? 2 * (size_t)c->Ppop * dm.RG / 8 : 0);
    const int grid = (int)std::min<size_t>(148 * 4, (most + 255) / 256);
    k_setup_population<<<grid, 256, 0, c->stream>>>(A);
    ++g_rp_launches;
    RP_CUDA(cudaGetLastError());
    return RP_OK;
}

// ---------------------------------------------------------------------------------------------
// Load-balance diagnostics (evaluation section of the paper): coefficient of variation of the
// aggregate rank loads, EP peak sum, tail peak, EP balance efficiency, attention and joint proxies.
// ---------------------------------------------------------------------------------------------
struct RpDiagDev { double cv_identity, cv_placed; i64 s_ep, t_ep, n_ep; i64 afx_sum, s0; };

// One launch: the last CTA works out the coefficients of variation, the others the peaks (the two have nothing to do with one
// another; as launches of their own, and with 64-bit shuffles for the peaks, they took 27 us behind the scoring).
#define DIAG_THREADS 512
#define DIAG_PEAK_CTAS 148
// Coefficients: one warp per layer; the lanes fetch the rank loads, one lane adds them up with plain sequential IEEE sums (no fused
// multiply-add); then thread 0 averages the layers in order.
__device__ __forceinline__ void diag_cv(const i64 *__restrict__ Lagg, const i64 *__restrict__ rank_load, const RpDims &dm,
                                        double *cvs, RpDiagDev *__restrict__ out)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double *G = cvs + 2 * dm.L + (size_t)warp * dm.P;
    for (int x = warp; x < 2 * dm.L; x += DIAG_THREADS / 32) {
        const int l = x >> 1, which = x & 1;
        for (int p = lane; p < dm.P; p += 32) {
            i64 g = 0;
            if (which) g = __ldg(rank_load + (size_t)l * dm.P + p);
            else {
#pragma unroll 4
                for (int n = 0; n < dm.H; ++n) g += __ldg(Lagg + (size_t)l * dm.E + p * dm.H + n);
            }
            G[p] = (double)g;
        }
        __syncwarp();
        if (lane == 0) {
            double mean = 0.0, var = 0.0;
            for (int p = 0; p < dm.P; ++p) mean = __dadd_rn(mean, G[p]);
            mean = __ddiv_rn(mean, (double)dm.P);
            for (int p = 0; p < dm.P; ++p) {
                const double d = __dsub_rn(G[p], mean);
                var = __dadd_rn(var, __dmul_rn(d, d));
            }
            var = __ddiv_rn(var, (double)dm.P);
            cvs[which * dm.L + l] = (mean > 0.0) ? __ddiv_rn(__dsqrt_rn(var), mean) : 0.0;
        }
        __syncwarp();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0;
        for (int x = 0; x < dm.L; ++x) { a = __dadd_rn(a, cvs[x]); b = __dadd_rn(b, cvs[dm.L + x]); }
        out->cv_identity = __ddiv_rn(a, (double)dm.L);
        out->cv_placed = __ddiv_rn(b, (double)dm.L);
    }
}

// Peaks: one warp per (row, layer): lanes over ranks, loop over shards; integer results by atomics on `sums` (s_ep, n_ep, t_ep; zero
// between launches, as the ticket is).  W and blob are written by the scoring, beside which this launch starts: neither __ldg nor __restrict__.
__global__ void __launch_bounds__(DIAG_THREADS)
k_diagnose(const i64 *__restrict__ Lagg, const i64 *__restrict__ rank_load, const int *W, const char *blob,
           RpBlob bl, RpDims dm, i64 *__restrict__ sums, int *__restrict__ ticket, RpDiagDev *__restrict__ out)
{
    extern __shared__ double cvs[];          // [2][L], then one row of rank loads per warp
    if (blockIdx.x == DIAG_PEAK_CTAS) { diag_cv(Lagg, rank_load, dm, cvs, out); return; }
    rp_wait_for_launch_before();
    const int lane = threadIdx.x & 31;
    const int wid = (int)(threadIdx.x >> 5) * DIAG_PEAK_CTAS + (int)blockIdx.x, nw = DIAG_PEAK_CTAS * DIAG_THREADS / 32;
    i64 s_ep = 0, n_ep = 0, t_ep = 0;
    for (int rl = wid; rl < dm.R * dm.L; rl += nw) {
        const int r = rl / dm.L, l = rl % dm.L;
        const int *w0 = W + ((size_t)r * dm.G * dm.L + l) * dm.P;
        int peak = 0;
        i64 best_sum = 0;
        for (int g0 = 0; g0 < dm.G; g0 += 4) {
            int mx[4] = { 0, 0, 0, 0 };
            i64 sum[4] = { 0, 0, 0, 0 };
            for (int p = lane; p < dm.P; p += 32)
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int v = g0 + u < dm.G ? w0[(size_t)(g0 + u) * dm.LP + p] : 0;
                    sum[u] += v; mx[u] = max(mx[u], v);
                }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                // (32 lanes' sums of 21 bits at a time)
                const u64 lo = __reduce_add_sync(0xffffffffu, (u32)sum[u] & 0x1fffffu), mid = __reduce_add_sync(0xffffffffu, (u32)(sum[u] >> 21) & 0x1fffffu),
                          hi = __reduce_add_sync(0xffffffffu, (u32)(sum[u] >> 42));
                const i64 all = (i64)(lo + (mid << 21) + (hi << 42));
                peak = max(peak, (int)__reduce_max_sync(0xffffffffu, mx[u]));
                best_sum = all > best_sum ? all : best_sum;
            }
        }
        s_ep += peak; n_ep += best_sum; t_ep = peak > t_ep ? peak : t_ep;
    }
    if (lane == 0) {
        if (s_ep) atomicAdd((u64 *)&sums[0], (u64)s_ep);
        if (n_ep) atomicAdd((u64 *)&sums[1], (u64)n_ep);
        if (t_ep) atomicMax(&sums[2], t_ep);
        __threadfence();
    }
    if (blockIdx.x == 0 && threadIdx.x < 32) {      // attention total and joint from the layout's blob
        const i64 *Afx = (const i64 *)(blob + bl.off_Afx);
        i64 a = 0;
        for (int x = lane; x < dm.RG; x += 32) a += Afx[x];
        for (int o = 16; o; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (lane == 0) { out->afx_sum = a; out->s0 = ((const i64 *)(blob + bl.off_S))[0]; }
    }
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(ticket, 1) == DIAG_PEAK_CTAS - 1) {
        __threadfence();
        out->s_ep = __ldcg(sums); out->n_ep = __ldcg(sums + 1); out->t_ep = __ldcg(sums + 2);
        sums[0] = 0; sums[1] = 0; sums[2] = 0; *ticket = 0;
    }
}

extern "C" int rp_diagnostics(rp_ctx *c, const int32_t *layout, rp_diag *out)
{
    if (!c || !out) return RP_ERR_ARG;
    if (c->stage < 3) return RP_ERR_STATE;
    const RpDims &dm = c->dm;
    if (dm.L > 1024) return RP_ERR_RANGE;
    cudaMemPool_t pool;
    RP_TRY(rp_get_pool(c->device, &pool));
    // scratch: a copy of a layout that is not in this GPU's memory, W, one blob
    const size_t wn = (size_t)dm.RG * dm.LP;
    const size_t off_W = ((size_t)dm.N * 4 + 255) & ~(size_t)255, off_blob = off_W + ((wn * 4 + 255) & ~(size_t)255);
    // (a row of P rank loads per warp: 144 KB with 1024 layers of 1024 ranks, the most there are)
    const size_t cv_smem = sizeof(double) * (2 * (size_t)dm.L + DIAG_THREADS / 32 * (size_t)dm.P);
    char *buf = nullptr;
    RP_CUDA(cudaMallocFromPoolAsync((void **)&buf, off_blob + (size_t)c->bl.bytes + 256, pool, c->stream));
    int st = RP_OK;
    cudaError_t e = cudaSuccess;
    do {
        const int *dl = layout ? layout : c->d_inc_layout;
        if (layout && rp_ptr_kind(c, layout) != 2) {
            e = cudaMemcpyAsync(buf, layout, sizeof(int) * dm.N, cudaMemcpyDefault, c->stream);
            if (e != cudaSuccess) break;
            dl = (const int *)buf;
        }
        int *bad = rp_pin_bad(c);
        *bad = 0;
        EvalArgs A = {};
        eval_one(c, A);
        A.lay32 = dl; A.W_out = (int *)(buf + off_W); A.blob_out = buf + off_blob;
        st = eval_launch(c, A, 1);
        if (st != RP_OK) break;
        // the record goes to the pinned block: its sums by the last CTA of the peaks, the rest by the first
        RpDiagDev *host = (RpDiagDev *)(c->h_pin + 32);
        if (cv_smem > 32 * 1024) {
            e = cudaFuncSetAttribute(k_diagnose, cudaFuncAttributeMaxDynamicSharedMemorySize, EVAL_SMEM_MAX);
            if (e != cudaSuccess) break;
        }
        // (started beside the scoring: what the peaks read of it they wait for, the coefficients are of the placement alone)
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(DIAG_PEAK_CTAS + 1); cfg.blockDim = dim3(DIAG_THREADS); cfg.dynamicSmemBytes = cv_smem; cfg.stream = c->stream;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = at; cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, k_diagnose, (const i64 *)c->d_Lagg, (const i64 *)c->d_rank_load, (const int *)(buf + off_W), (const char *)(buf + off_blob),
                               c->bl, dm, c->d_one_Esum + dm.RG, c->d_one_ticket, host);
        if (e != cudaSuccess) break;
        ++g_rp_launches;
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
        if (e != cudaSuccess) break;
        if (*bad) { st = RP_ERR_ARG; break; }
        const RpDiagDev h = *host;
        out->cv_identity = h.cv_identity; out->cv_placed = h.cv_placed;
        out->s_ep = h.s_ep; out->t_ep = h.t_ep; out->n_ep = h.n_ep;
        out->eta_ep = h.s_ep > 0 ? (double)h.n_ep / ((double)dm.P * (double)h.s_ep) : 1.0;
        out->attention = (double)h.afx_sum / (double)dm.SC;
        out->joint = (double)h.s0 / (double)dm.SC;
    } while (0);
    cudaFreeAsync(buf, c->stream);
    if (e != cudaSuccess) return rp_fail(e);
    return st;
}

// ---------------------------------------------------------------------------------------------
// Scoring layouts without allocating: the kernels above, with their scratch (samples grouped by
// row-shard, row-shard sums, arrival counters) taken from a fixed array that is part of the library image
// instead of from the context's allocator.
// ---------------------------------------------------------------------------------------------
#define RP_NOALLOC_MAX_LAYOUTS 1024            // layouts per call
#define RP_NOALLOC_MAX_CELLS (1 << 19)         // n * N          (1 MiB of 16-bit cell ids)
#define RP_NOALLOC_MAX_ROWSHARDS (1 << 15)     // n * R * G      (256 KiB of 64-bit sums)

struct RpNoAllocScratch {
    int tickets[RP_NOALLOC_MAX_LAYOUTS];           // (next to the sums: cleared together)
    i64 esum[RP_NOALLOC_MAX_ROWSHARDS];
    int off[RP_NOALLOC_MAX_ROWSHARDS + RP_NOALLOC_MAX_LAYOUTS];
    unsigned short list[RP_NOALLOC_MAX_CELLS];
};
// About 1.4 MiB on every GPU that loads the library, held until the process exits.
static __device__ __align__(256) unsigned char g_noalloc_scratch[sizeof(RpNoAllocScratch)];
// Device address of the array above, per device (in host code the symbol itself is only a
// stand-in, never a device address).
static void *g_noalloc_addr[64];

extern "C" int rp_eval_layouts_noalloc(rp_ctx *c, const int32_t *layouts, int32_t n, int64_t *score_fx,
                                       double *score_f64)
{
    if (!c || !layouts || n < 1) return RP_ERR_ARG;
    if (c->stage < 3) return RP_ERR_STATE;
    const RpDims &dm = c->dm;
    if (n > RP_NOALLOC_MAX_LAYOUTS || (long long)n * dm.N > RP_NOALLOC_MAX_CELLS ||
        (long long)n * dm.RG > RP_NOALLOC_MAX_ROWSHARDS)
        return RP_ERR_RANGE;                  // beyond the fixed scratch: use rp_eval_population
    const size_t smem = eval_smem_bytes(dm);
    if (smem > 220 * 1024) return RP_ERR_RANGE;   // nothing has been queued yet
    int cur = -1;
    RP_CUDA(cudaGetDevice(&cur));
    if (cur != c->device || cur < 0 || cur >= 64) return RP_ERR_STATE;
    // every array must already be on the device: staging a host array would need memory
    const void *ptrs[3] = { layouts, score_fx, score_f64 };
    for (int x = 0; x < 3; ++x) {
        if (!ptrs[x]) continue;
        cudaPointerAttributes at;
        if (cudaPointerGetAttributes(&at, ptrs[x]) != cudaSuccess) { cudaGetLastError(); return RP_ERR_ARG; }
        if (at.type != cudaMemoryTypeDevice && at.type != cudaMemoryTypeManaged) return RP_ERR_ARG;
        if (at.type == cudaMemoryTypeDevice && at.device != c->device) return RP_ERR_ARG;    // another GPU's memory
    }
    if (!g_noalloc_addr[cur]) {               // set-up, once per device, with that device current
        void *p = nullptr;
        RP_CUDA(cudaGetSymbolAddress(&p, g_noalloc_scratch));
        g_noalloc_addr[cur] = p;
    }
    RpNoAllocScratch *sc = (RpNoAllocScratch *)g_noalloc_addr[cur];
    // the array keeps what the previous call left: the arrival counters and the row-shard sums must start at zero
    RP_CUDA(cudaMemsetAsync(sc, 0, sizeof(sc->tickets) + sizeof(i64) * (size_t)n * dm.RG, c->stream));
    int *bad = rp_pin_bad(c);
    *bad = 0;
    EvalArgs A = {};
    A.lay32 = layouts; A.score_out = (i64 *)score_fx; A.f64_out = score_f64; A.bad = bad;
    A.cost = sc->esum; A.tickets = sc->tickets; A.list = sc->list; A.off = (u32 *)sc->off;
    RP_TRY(eval_launch(c, A, n));
    RP_CUDA(cudaStreamSynchronize(c->stream));
    return *bad ? RP_ERR_ARG : RP_OK;
}
