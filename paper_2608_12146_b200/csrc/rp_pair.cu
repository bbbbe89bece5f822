// EDPAwarePair (Section 4.1.1; Algorithm 2, third construction operator): every completed cell
// stays the same set of samples, only the (row, DP slot) it occupies changes.
//
//   profile of cell b      w_b[l][p] = sum of q[i][l][p] over its samples; peak_b = max w_b
//   order                  cells by decreasing peak, ties by lower cell index
//   insertion key of an empty slot s (row r, shard g) for the cell in hand:
//                          (sum_l max_p (V+w_b) - sum_l max_p V,  max_{l,p} (V+w_b)),
//                          V the rank load of row-shard (r, g) from the cells placed so far;
//                          slots ranked by ascending key, ties by lower slot index
//   rank-decaying sampling rho = min(min(w, #empty) - 1, leading zero bits of the draw),
//                          draw = Philox(h, 0, member, 6).x for the h-th cell placed
//
// One CTA per population member (member 0, the length-only seed, is left alone).  Empty slots of
// one row-shard share their key, so the key is computed once per row-shard that has both placed
// cells and an empty slot, one warp per row-shard, lanes over layers; one without placed cells has
// the cell's own sums as its key.
//
// A chain of K steps per member, so a step's latency decides.  With one slot per row-shard (EDP width = DP width) all
// empty slots rank by their index alone: no rank loads, one warp draws from the 32 lowest empty slots kept in its lanes.
// With more, a round of the ranking is two sets of four warp-wide minima and one barrier (a serial pass of one thread over
// the warps' results and two barriers before: 22 k cycles a step at 240 slots).  255 members of 240 cells, 24 layers of 16
// ranks, one slot per row-shard: 2.77 ms -> 0.10 ms, most of it now the sums of the cells' samples.
#include "rp_common.cuh"

#define PAIR_THREADS 256
#define PAIR_WARPS (PAIR_THREADS / 32)

struct __align__(16) PairKey { u64 d; u32 p, s; };

// Smallest (d, p, s) of the warp.
__device__ __forceinline__ PairKey pair_min(const PairKey &k)
{
    const u32 hi = (u32)(k.d >> 32), lo = (u32)k.d;
    const u32 mh = __reduce_min_sync(0xffffffffu, hi);
    bool in = hi == mh;
    const u32 ml = __reduce_min_sync(0xffffffffu, in ? lo : 0xffffffffu);
    in = in && lo == ml;
    const u32 mp = __reduce_min_sync(0xffffffffu, in ? k.p : 0xffffffffu);
    in = in && k.p == mp;
    PairKey r;
    r.d = ((u64)mh << 32) | ml; r.p = mp;
    r.s = __reduce_min_sync(0xffffffffu, in ? k.s : 0xffffffffu);
    return r;
}

__device__ __forceinline__ int pair_ld(const int *p, int) { return __ldg(p); }
__device__ __forceinline__ int4 pair_ld(const int *p, int4) { return __ldg((const int4 *)p); }
__device__ __forceinline__ int pair_add(int a, int b) { return a + b; }
__device__ __forceinline__ int4 pair_add(int4 a, int4 b) { return make_int4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
__device__ __forceinline__ int pair_top(int a) { return a; }
__device__ __forceinline__ int pair_top(int4 a) { return max(max(a.x, a.y), max(a.z, a.w)); }

// Profile of one cell (sum over its n samples) by one warp, written to `prof` unless that is null; returns this lane's peak.
template <typename T>
__device__ __forceinline__ int pair_profile(const int *__restrict__ q, const int *list, int n, int LP, int *prof, int lane)
{
    constexpr int VEC = sizeof(T) / 4;
    int pk = 0;
    for (int x = lane * VEC; x < LP; x += 32 * VEC) {
        T acc = T();
        int e = 0;
        for (; e + 4 <= n; e += 4) {                 // four loads in flight
            const T a = pair_ld(q + (size_t)list[e] * LP + x, T()), b = pair_ld(q + (size_t)list[e + 1] * LP + x, T());
            const T c = pair_ld(q + (size_t)list[e + 2] * LP + x, T()), d = pair_ld(q + (size_t)list[e + 3] * LP + x, T());
            acc = pair_add(acc, pair_add(pair_add(a, b), pair_add(c, d)));
        }
        for (; e < n; ++e) acc = pair_add(acc, pair_ld(q + (size_t)list[e] * LP + x, T()));
        if (prof) *(T *)(prof + x) = acc;
        pk = max(pk, pair_top(acc));
    }
    return pk;
}

__global__ void __launch_bounds__(PAIR_THREADS)
k_edp_pair(RpDims dm, const int *__restrict__ q, const unsigned short *__restrict__ rg_of,
           const int *__restrict__ lay_in, int *__restrict__ lay_out, int *__restrict__ prof_all,
           int *__restrict__ V_all, int first_member, int width, u32 key0, u32 key1)
{
    extern __shared__ __align__(16) unsigned char pair_smem[];
    const int N = dm.N, K = dm.K, RG = dm.RG, LP = dm.LP, L = dm.L, P = dm.P;
    const bool one_slot = RG == K;                 // every row-shard has one slot
    i64 *e_old = (i64 *)pair_smem;                 // [RG] sum_l max_p V
    i64 *kd = e_old + RG;                          // [RG] increase of that sum for the cell in hand
    int *kp = (int *)(kd + RG);                    // [RG] largest peak after insertion
    int *free_rg = kp + RG;                        // [RG] empty slots left in the row-shard
    int *peak = free_rg + RG;                      // [K]
    int *order = peak + K;                         // [K] cells by (-peak, index)
    int *slot_of = order + K;                      // [K]
    int *cstart = slot_of + K;                     // [K + 1] first entry of each cell in `list`
    int *fillp = cstart + K + 1;                   // [K] fill pointers, then draws | row-shard of the slot << 8
    int *list = fillp + K;                         // [N] samples grouped by cell
    i64 *eself = (i64 *)(((size_t)(list + N) + 7) & ~(size_t)7);   // [K] sum_l max_p of the cell's own profile
    __shared__ PairKey red[2][PAIR_WARPS];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int j = first_member + blockIdx.x;
    const int *lay = lay_in + (size_t)j * N;
    int *prof = prof_all + (size_t)blockIdx.x * K * LP;
    int *V = V_all + (size_t)j * RG * LP;

    // ---- samples grouped by cell (counting sort) ----------------------------------------------
    for (int b = tid; b <= K; b += PAIR_THREADS) cstart[b] = 0;
    for (int x = tid; x < RG; x += PAIR_THREADS) { e_old[x] = 0; free_rg[x] = 0; }
    __syncthreads();
    for (int i = tid; i < N; i += PAIR_THREADS) atomicAdd(&cstart[lay[i] + 1], 1);
    for (int s = tid; s < K; s += PAIR_THREADS) atomicAdd(&free_rg[rg_of[s]], 1);
    __syncthreads();
    if (warp == 0) {                               // inclusive prefix of the counts
        int run = 0;
        for (int b0 = 1; b0 <= K; b0 += 32) {
            const int b = b0 + lane;
            int v = b <= K ? cstart[b] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(0xffffffffu, v, o); if (lane >= o) v += y; }
            if (b <= K) cstart[b] = run + v;
            run += __shfl_sync(0xffffffffu, v, 31);
        }
    }
    __syncthreads();
    for (int b = tid; b < K; b += PAIR_THREADS) fillp[b] = cstart[b];
    __syncthreads();
    for (int i = tid; i < N; i += PAIR_THREADS) list[atomicAdd(&fillp[lay[i]], 1)] = i;
    __syncthreads();

    // ---- cell profiles and peaks: one warp per cell, lanes over (layer, rank) -------------------
    for (int b = warp; b < K; b += PAIR_WARPS) {
        const int *lb = list + cstart[b];
        const int n = cstart[b + 1] - cstart[b];
        int *pb = one_slot ? nullptr : prof + (size_t)b * LP;
        int pk = LP % 4 == 0 ? pair_profile<int4>(q, lb, n, LP, pb, lane) : pair_profile<int>(q, lb, n, LP, pb, lane);
        pk = __reduce_max_sync(0xffffffffu, pk);
        if (lane == 0) peak[b] = pk;
        if (one_slot) continue;
        __syncwarp();                              // the profile row is complete before it is read back per layer
        i64 es = 0;
        for (int l = lane; l < L; l += 32) {
            int mn = 0;
            for (int p = 0; p < P; ++p) mn = max(mn, pb[l * P + p]);
            es += mn;
        }
        for (int o = 16; o; o >>= 1) es += __shfl_xor_sync(0xffffffffu, es, o);
        if (lane == 0) eself[b] = es;
    }
    __syncthreads();
    // ---- order by (-peak, index): rank by counting; the draws of all steps -----------------------
    for (int b = tid; b < K; b += PAIR_THREADS) {
        const int pb = peak[b];
        int r = 0;
        for (int o = 0; o < K; ++o) { const int po = peak[o]; r += (po > pb) || (po == pb && o < b); }
        order[r] = b;
        const int lz = __clz((int)rp_philox((u32)b, 0u, (u32)j, 6u, key0, key1).x);
        const int ne = K - b, m = ne < width ? ne : width;
        fillp[b] = (lz < m - 1 ? lz : m - 1) | ((int)rg_of[b] << 8);
    }
    __syncthreads();

    if (one_slot) {
        // The rho-th lowest empty slot; rho < 32, so the 32 lowest in the lanes of one warp are enough.
        if (warp == 0) {
            int win = lane;                        // slots from K on never come up: rho < number of empty slots
            for (int h0 = 0; h0 < K; h0 += 32) {
                const int nb = min(32, K - h0);
                const int draw = lane < nb ? fillp[h0 + lane] & 255 : 0, b = lane < nb ? order[h0 + lane] : 0;
                int mine = 0;
                for (int u = 0; u < nb; ++u) {
                    const int rho = __shfl_sync(0xffffffffu, draw, u);
                    const int s = __shfl_sync(0xffffffffu, win, rho), up = __shfl_down_sync(0xffffffffu, win, 1);
                    if (lane >= rho) win = lane == 31 ? h0 + u + 32 : up;
                    if (lane == u) mine = s;
                }
                if (lane < nb) slot_of[b] = mine;
            }
        }
        __syncthreads();
    } else {
        u32 gone = 0;                              // bit m: slot tid + m * PAIR_THREADS is taken (K < 32 * PAIR_THREADS)
        int par = 0;
        // ---- place the cells one by one --------------------------------------------------------
        for (int h = 0; h < K; ++h) {
            const int b = order[h];
            const int *wb = prof + (size_t)b * LP;
            const i64 es = eself[b];
            const int pkb = peak[b];
            // keys of the row-shards that still have an empty slot, 32 row-shards of a warp looked at at a time
            for (int r0 = 0; r0 < RG; r0 += 32 * PAIR_WARPS) {
                const int mine = r0 + lane * PAIR_WARPS + warp;
                bool part = false;
                if (mine < RG && free_rg[mine] > 0) {
                    part = e_old[mine] != 0;
                    if (!part) { kd[mine] = es; kp[mine] = pkb; }      // nothing placed there yet: the cell's own sums
                }
                for (unsigned todo = __ballot_sync(0xffffffffu, part); todo; todo &= todo - 1) {
                    const int rg = r0 + (__ffs(todo) - 1) * PAIR_WARPS + warp;
                    const int *v = V + (size_t)rg * LP;
                    i64 en = 0;
                    int pk = 0;
                    for (int l = lane; l < L; l += 32) {
                        int mn = 0;
                        if (P % 4 == 0) {
                            for (int p = 0; p < P; p += 4)
                                mn = max(mn, pair_top(pair_add(*(const int4 *)(v + l * P + p), *(const int4 *)(wb + l * P + p))));
                        } else {
                            for (int p = 0; p < P; ++p) mn = max(mn, v[l * P + p] + wb[l * P + p]);
                        }
                        en += mn;
                        pk = max(pk, mn);
                    }
                    for (int o = 16; o; o >>= 1) en += __shfl_xor_sync(0xffffffffu, en, o);
                    pk = __reduce_max_sync(0xffffffffu, pk);
                    if (lane == 0) { kd[rg] = en - e_old[rg]; kp[rg] = pk; }
                }
            }
            __syncthreads();
            // the rho-th ranked empty slot: rho + 1 rounds of a block-wide minimum, earlier picks left out
            const int rho = fillp[h] & 255;
            u32 out = gone;
            int s = 0;
            for (int round = 0; round <= rho; ++round) {
                PairKey best = { ~0ull, 0xffffffffu, 0xffffffffu };
                for (int m = 0, x = tid; x < K; ++m, x += PAIR_THREADS) {
                    if ((out >> m) & 1) continue;
                    const int rg = fillp[x] >> 8;
                    const u64 d = (u64)kd[rg];
                    const u32 p = (u32)kp[rg];
                    if (d < best.d || (d == best.d && p < best.p)) { best.d = d; best.p = p; best.s = (u32)x; }
                }
                best = pair_min(best);
                if (lane == 0) red[par][warp] = best;
                __syncthreads();
                const PairKey none = { ~0ull, 0xffffffffu, 0xffffffffu };
                s = (int)pair_min(lane < PAIR_WARPS ? red[par][lane] : none).s;
                par ^= 1;
                if ((s & (PAIR_THREADS - 1)) == tid) out |= 1u << (s / PAIR_THREADS);
            }
            if ((s & (PAIR_THREADS - 1)) == tid) gone |= 1u << (s / PAIR_THREADS);
            const int rg = fillp[s] >> 8;
            if (free_rg[rg] > 1) {                 // of a full row-shard nothing is asked any more
                int *v = V + (size_t)rg * LP;
                if (e_old[rg] == 0) for (int x = tid; x < LP; x += PAIR_THREADS) v[x] = wb[x];
                else for (int x = tid; x < LP; x += PAIR_THREADS) v[x] += wb[x];
            }
            __syncthreads();
            if (tid == 0) {
                slot_of[b] = s;
                free_rg[rg] -= 1;
                e_old[rg] += kd[rg];
            }
            __syncthreads();
        }
    }
    for (int i = tid; i < N; i += PAIR_THREADS) lay_out[(size_t)j * N + i] = slot_of[lay[i]];
}

size_t rp_pair_smem_bytes(const RpDims &dm)
{
    return sizeof(i64) * 2 * dm.RG + sizeof(int) * 2 * dm.RG + sizeof(int) * ((size_t)5 * dm.K + 1) + sizeof(int) * (dm.N + 1) +
           sizeof(i64) * dm.K + 16;
}

// Pairs members [first, first + count) of lay_in into lay_out; prof is scratch for `count`
// members ([count][K][LP] ints), V the rank-load cells of the members ([P_pop][RG][LP], overwritten).
int rp_launch_edp_pair(rp_ctx *c, const int *lay_in, int *lay_out, int *prof, int first, int count, int width)
{
    const RpDims &dm = c->dm;
    const size_t smem = rp_pair_smem_bytes(dm);
    if (smem > 200 * 1024) return RP_ERR_RANGE;
    if (smem > 32 * 1024)
        RP_CUDA(cudaFuncSetAttribute(k_edp_pair, cudaFuncAttributeMaxDynamicSharedMemorySize, RP_SMEM_LIMIT));
    const unsigned short *rg_of = (const unsigned short *)(c->d_static + c->sl.off_rg);
    k_edp_pair<<<count, PAIR_THREADS, smem, c->stream>>>(dm, c->d_q, rg_of, lay_in, lay_out, prof, c->d_W, first, width,
                                                         (u32)c->cfg.seed, (u32)(c->cfg.seed >> 32));
    ++g_rp_launches;
    RP_CUDA(cudaGetLastError());
    return RP_OK;
}
