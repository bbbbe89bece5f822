// Randomized fixed-row seeds (Algorithm 2 of the paper, trial loop): one warp per trial.
//
// WindowShuffle keeps the window of the next `width` samples (decreasing length) in the
// registers of `width` lanes; RandomizedBestFit ranks the cells a sample fits in by one 64-bit
// key (remaining capacity, then sample count, then index: smaller = fuller, fewer, lower).
// Random words: Philox(h, 0, trial, 4) for the shuffle, (h, 0, trial, 5) for the fit, h = position
// of the sample in the emitted order.
//
// A trial is a chain of N steps, so its latency is what counts.  The warp keeps the keys of the cells sorted: the cells a
// sample fits in are the keys from (length, 0, 0) on, the r-th of them is taken out, and its smaller new key goes in front of
// those it passes, which move up by one.  Up to 512 cells a lane holds E consecutive keys in registers (a position is one
// warp-wide sum of compares, the move one shuffle and a compare a key: 520 cycles a sample at 240 cells, 600 with a second sum; 435 with keys
// of 32 bits, which pass by a minimum and a maximum: a warp alone pays two to three cycles an instruction); beyond, the keys lie in shared memory
// (two searches of two ballots: 1100 cycles).  Ranking by r + 1 passes over all cells took 4400.  What does not depend on the
// fit runs 32 samples at a time: a lane draws the random words of its sample, then the shuffle emits the 32 samples.
#include <algorithm>

#include "rp_common.cuh"

#define SEED_WARPS 4

// Keys sorted in blocks of 2^lb: block x of the 32 starts at x * (2^lb + 1), so that the last keys of all blocks lie in
// different banks.  Unused places hold ~0.
__device__ __forceinline__ int seed_at(int x, int lb) { return x + (x >> lb); }

// Number of keys below v; `top` is the last key of this lane's block.
__device__ __forceinline__ int seed_below(const u64 *keys, int lb, u64 top, u64 v, int lane)
{
    const int w = __popc(__ballot_sync(0xffffffffu, top < v)), B = 1 << lb;
    if (w == 32) return 32 << lb;
    int n = w << lb;
    for (int e0 = 0; e0 < B; e0 += 32)
        n += __popc(__ballot_sync(0xffffffffu, e0 + lane < B && keys[(w << lb) + w + min(e0 + lane, B - 1)] < v));
    return n;
}

// The samples of positions h0 .. h0+nb-1 (lane x: `em` of position h0 + x, with the random word of its fit) and the window behind them.
__device__ __forceinline__ void seed_emit(const int *__restrict__ order, const RpDims &dm, int width, u32 key0, u32 key1, int j, int h0, int nb, int lane,
                                          int &win, int &em, u32 &xf)
{
    const int h = h0 + lane;
    const int ahead = width + h < dm.N ? order[width + h] : -1;      // enters the window after step h
    // the window holds min(width, N - h) samples at step h
    const int pos = rp_pick(rp_philox((u32)h, 0u, (u32)j, 4u, key0, key1).x, min(width, dm.N - h));
    xf = rp_philox((u32)h, 0u, (u32)j, 5u, key0, key1).x;
    em = 0;
#pragma unroll 4
    for (int u = 0; u < nb; ++u) {
        const int at = __shfl_sync(0xffffffffu, pos, u), in = __shfl_sync(0xffffffffu, ahead, u);
        const int s = __shfl_sync(0xffffffffu, win, at), up = __shfl_down_sync(0xffffffffu, win, 1);
        if (lane >= at) win = lane == width - 1 ? in : up;           // close the gap, order kept
        if (lane == u) em = s;
    }
}

// Widths of the fields of a key: remaining capacity on top, samples, index + 1.
// The capacity's field holds what an open cell can have left, one less than the cap at most.  A length can be the cap itself: where that is a power
// of two as large as the field, the length shifted there is 2^32 (2^64), which is zero.  A cell that such a sample opens has nothing left, as the
// subtraction says anyway; behind the opening samples it fits nowhere, which every comparison with a shifted length has to say.
struct SeedKey { int rem, index; };              // (shifts of the capacity and of the samples)

// A key that passes `from` places on its way down: keys that are not below it move up by one as far as place `from`.
template <int E>
__device__ __forceinline__ void seed_insert(u64 (&v)[E], u64 key, int top, u64 below, int lane)
{
    // where a key moves from one that is below the new one, the new key comes in
    bool lt[E + 1];                                  // key of the place before; of place e at e + 1
    lt[0] = lane == 0 || below < key;
#pragma unroll
    for (int e = 0; e < E; ++e) lt[e + 1] = v[e] < key;
#pragma unroll
    for (int e = E - 1; e >= 0; --e)
        if (!lt[e + 1] && e <= top) v[e] = lt[e] ? key : (e ? v[e ? e - 1 : 0] : below);
}
template <int E>
__device__ __forceinline__ void seed_insert(u32 (&v)[E], u32 key, int top, u32 below, int lane)
{
    // the larger of what comes from the place before and the new key, unless what is there is smaller still
    if (lane == 0) below = 0;
#pragma unroll
    for (int e = E - 1; e >= 0; --e) v[e] = min(v[e], max(e ? v[e ? e - 1 : 0] : below, e <= top ? key : 0xffffffffu));
}

// A trial with the keys in registers, E a lane (K <= 32 * E).  1: done, 0: a sample fits nowhere, -1: a cell has more samples than a
// key of this width counts.
template <int E, class Key>
__device__ __forceinline__ int seed_trial(const int *__restrict__ t, const int *__restrict__ order, const RpDims &dm, int width, u32 key0, u32 key1,
                                          int j, int *lay, SeedKey sk, int lane)
{
    Key v[E];                                        // keys of places lane * E .. + E-1, unused places ~0
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = (Key)~(Key)0;
    const Key one = (Key)1 << sk.index, full = ((Key)1 << sk.rem) - one;       // a sample; as many as there is room for
    int win = lane < dm.N ? order[lane] : -1;        // lane x < width: the x-th sample of the window
    for (int h0 = 0; h0 < dm.N; h0 += 32) {
        const int nb = min(32, dm.N - h0);
        int em;
        u32 xf;
        seed_emit(order, dm, width, key0, key1, j, h0, nb, lane, win, em, xf);
        const int len = lane < nb ? t[em] : 0;
        // the length as a capacity of a key (its upper word; there is nothing in the lower one of 64 bits), less one: zero less one is all ones
        const u32 lim = (sizeof(Key) == 4 ? (u32)len << sk.rem : (u32)len << (sk.rem - 32)) - 1u;
        int place = 0;
        bool over = false;
        for (int u = 0; u < nb; ++u) {
            const u32 under = __shfl_sync(0xffffffffu, lim, u);
            const Key ts = sizeof(Key) == 4 ? (Key)(under + 1u) : (Key)((u64)(under + 1u) << 32);
            const u32 x = __shfl_sync(0xffffffffu, xf, u);
            Key key;
            int from;                                // place the new key comes from
            if (h0 + u < dm.K) {
                from = h0 + u;                       // cell h opens
                key = (Key)((u64)(u32)dm.C << sk.rem) - ts;
                key |= one | (Key)(u32)(from + 1);
            } else {
                int n = 0;                           // keys below ts: all of them, unused places too, where ts is zero
#pragma unroll
                for (int e = 0; e < E; ++e) n += (u32)(sizeof(Key) == 4 ? (u64)v[e] : (u64)v[e] >> 32) <= under;
                const int p0 = __reduce_add_sync(0xffffffffu, n), nc = dm.K - p0;        // feasible cells
                if (nc <= 0) return over ? -1 : 0;
                from = p0 + rp_pick(x, nc < width ? nc : width);
                Key m[E];                            // key number from % E of every lane by halving
#pragma unroll
                for (int e = 0; e < E; ++e) m[e] = v[e];
#pragma unroll
                for (int half = E / 2; half; half /= 2)
#pragma unroll
                    for (int e = 0; e < half; ++e) m[e] = (from & half) ? m[e + half] : m[e];
                key = __shfl_sync(0xffffffffu, m[0], from / E);
                over |= (key & full) == full;
                key = key - ts + one;
            }
            seed_insert(v, key, from - lane * E, (Key)__shfl_up_sync(0xffffffffu, v[E - 1], 1), lane);
            if (lane == u) place = (int)(key & (one - 1)) - 1;
        }
        if (over) return -1;
        if (lane < nb) lay[em] = place;
    }
    return 1;
}

// E > 0: E keys a lane in registers (K <= 32 * E), NARROW: of 32 bits as long as those hold every cell's samples; E = 0: in shared memory,
// blocks of 2^lb.
template <int E, bool NARROW>
__global__ void __launch_bounds__(SEED_WARPS * 32)
k_seed_trials(const int *__restrict__ t, const int *__restrict__ order, const int *__restrict__ seed_layout, RpDims dm,
              int width, int lb, SeedKey sk, u32 key0, u32 key1, int Ppop, int *__restrict__ layouts, int *__restrict__ ok)
{
    extern __shared__ __align__(16) u64 seed_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int places = (32 << lb) + 32;
    u64 *keys = seed_smem + (size_t)warp * places;
    const int j = blockIdx.x * SEED_WARPS + warp;
    if (j >= Ppop) return;
    int *lay = layouts + (size_t)j * dm.N;
    if (j == 0) {                                    // member 0 is the length-only seed
        for (int i = lane; i < dm.N; i += 32) lay[i] = seed_layout[i];
        if (lane == 0) ok[0] = 1;
        return;
    }
    bool good = true;
    if constexpr (E > 0) {
        int st = -1;
        if (NARROW) st = seed_trial<E, u32>(t, order, dm, width, key0, key1, j, lay, sk, lane);
        if (st < 0) st = seed_trial<E, u64>(t, order, dm, width, key0, key1, j, lay, SeedKey{ 40, 20 }, lane);
        good = st == 1;
    } else {
        for (int x = lane; x < places; x += 32) keys[x] = ~0ull;
        __syncwarp();
        const int last = (lane << lb) + lane + (1 << lb) - 1;        // last key of this lane's block
        int win = lane < dm.N ? order[lane] : -1;    // lane x < width: the x-th sample of the window
        for (int h0 = 0; h0 < dm.N && good; h0 += 32) {
            const int nb = min(32, dm.N - h0);
            int em;
            u32 xf;
            seed_emit(order, dm, width, key0, key1, j, h0, nb, lane, win, em, xf);
            const int len = lane < nb ? t[em] : 0;
            int place = 0;
            for (int u = 0; u < nb; ++u) {
                const u64 ts = (u64)(u32)__shfl_sync(0xffffffffu, len, u) << 40;
                const u32 x = __shfl_sync(0xffffffffu, xf, u);
                u64 key;
                int from;                            // place the new key comes from
                const u64 top = keys[last];
                if (h0 + u < dm.K) {
                    from = h0 + u;
                    key = (((u64)(u32)dm.C << 40) - ts) | (1ull << 20) | (u64)(u32)(from + 1);
                } else {
                    const int p0 = ts ? seed_below(keys, lb, top, ts, lane) : dm.K, nc = dm.K - p0;        // (ts = 0: see SeedKey)
                    if (nc == 0) { good = false; break; }
                    from = p0 + rp_pick(x, nc < width ? nc : width);
                    key = keys[seed_at(from, lb)] - ts + (1ull << 20);
                }
                const int to = seed_below(keys, lb, top, key, lane);
                __syncwarp();
                for (int hi = from; hi > to; hi -= 128) {        // from the top
                    u64 w[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) { const int y = hi - 32 * e - lane; if (y > to) w[e] = keys[seed_at(y - 1, lb)]; }
                    __syncwarp();
#pragma unroll
                    for (int e = 0; e < 4; ++e) { const int y = hi - 32 * e - lane; if (y > to) keys[seed_at(y, lb)] = w[e]; }
                    __syncwarp();
                }
                if (lane == 0) keys[seed_at(to, lb)] = key;
                __syncwarp();
                if (lane == u) place = (int)(key & 0xFFFFFu) - 1;
            }
            if (lane < nb && good) lay[em] = place;
        }
    }
    __syncwarp();
    if (!good) for (int i = lane; i < dm.N; i += 32) lay[i] = seed_layout[i];
    if (lane == 0) ok[j] = good ? 1 : 0;
}

int rp_launch_seed_trials(rp_ctx *c, int width, int *layouts, int *ok)
{
    const RpDims &dm = c->dm;
    int lb = 0;
    while ((32 << lb) < dm.K) ++lb;
    const size_t smem = lb > 4 ? sizeof(u64) * (size_t)SEED_WARPS * ((32 << lb) + 32) : 0;
    if (smem > 200 * 1024) return RP_ERR_RANGE;
    if (smem > 32 * 1024) RP_CUDA(cudaFuncSetAttribute(k_seed_trials<0, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, RP_SMEM_LIMIT));
    // Keys of 32 bits where the capacity (below the cap once a cell is open) and the index leave room for four times the samples an average
    // cell has; a trial that comes upon a cell with more starts over with 64.
    auto bits = [](u32 x) { int n = 0; while (x >> n) ++n; return n; };
    SeedKey sk;
    sk.index = bits((u32)dm.K);
    const int cb = 32 - std::max(1, bits((u32)dm.C - 1)) - sk.index;
    sk.rem = sk.index + cb;
    const bool narrow = lb <= 4 && cb > 0 && 4ll * dm.N / dm.K < (1ll << cb);
#define SEED_FN(E_) (narrow ? k_seed_trials<E_, true> : k_seed_trials<E_, false>)
    auto fn = lb > 4 ? k_seed_trials<0, false> : lb == 4 ? SEED_FN(16) : lb == 3 ? SEED_FN(8) : lb == 2 ? SEED_FN(4) : SEED_FN(2);
#undef SEED_FN
    const int grid = (c->Ppop + SEED_WARPS - 1) / SEED_WARPS;
    fn<<<grid, SEED_WARPS * 32, smem, c->stream>>>(c->d_t, c->d_order, c->d_seed_layout, dm, width, lb, sk,
                                                  (u32)c->cfg.seed, (u32)(c->cfg.seed >> 32), c->Ppop, layouts, ok);
    ++g_rp_launches;
    RP_CUDA(cudaGetLastError());
    return RP_OK;
}

// Best member of a scored population (lexicographic, lowest index on ties): becomes the incumbent.
__global__ void __launch_bounds__(1024)
k_pick_best(const i64 *__restrict__ scores, const int *__restrict__ layouts, int n, int N, int *__restrict__ anc,
            int *__restrict__ inc_layout, i64 *__restrict__ inc_score, i64 *__restrict__ best_out)
{
    __shared__ i64 r0[32], r1[32], r2[32];
    __shared__ int rj[32], win;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    i64 b0 = 0x7fffffffffffffffll, b1 = b0, b2 = b0;
    int bj = 0x7fffffff;
    for (int j = tid; j < n; j += 1024) {
        const i64 s0 = scores[3 * (size_t)j], s1 = scores[3 * (size_t)j + 1], s2 = scores[3 * (size_t)j + 2];
        if (rp_lex_less(s0, s1, s2, b0, b1, b2)) { b0 = s0; b1 = s1; b2 = s2; bj = j; }
        anc[j] = j;                                  // every member continues from its own state
    }
    for (int o = 16; o; o >>= 1) {
        const i64 o0 = __shfl_xor_sync(0xffffffffu, b0, o), o1 = __shfl_xor_sync(0xffffffffu, b1, o);
        const i64 o2 = __shfl_xor_sync(0xffffffffu, b2, o);
        const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
        if (rp_lex_less(o0, o1, o2, b0, b1, b2) || (o0 == b0 && o1 == b1 && o2 == b2 && oj < bj)) { b0 = o0; b1 = o1; b2 = o2; bj = oj; }
    }
    if (lane == 0) { r0[warp] = b0; r1[warp] = b1; r2[warp] = b2; rj[warp] = bj; }
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < 32; ++w)
            if (rp_lex_less(r0[w], r1[w], r2[w], b0, b1, b2) || (r0[w] == b0 && r1[w] == b1 && r2[w] == b2 && rj[w] < bj)) {
                b0 = r0[w]; b1 = r1[w]; b2 = r2[w]; bj = rj[w];
            }
        win = bj;
        inc_score[0] = b0; inc_score[1] = b1; inc_score[2] = b2;
        best_out[0] = b0; best_out[1] = b1; best_out[2] = b2;
    }
    __syncthreads();
    const int *src = layouts + (size_t)win * N;
    for (int i = tid; i < N; i += 1024) inc_layout[i] = src[i];
}

int rp_launch_pick_best(rp_ctx *c, const i64 *scores, const int *layouts, int n, i64 *best_score_out)
{
    k_pick_best<<<1, 1024, 0, c->stream>>>(scores, layouts, n, c->dm.N, c->d_anc, c->d_inc_layout, c->d_inc_score, best_score_out);
    ++g_rp_launches;
    RP_CUDA(cudaGetLastError());
    return RP_OK;
}
