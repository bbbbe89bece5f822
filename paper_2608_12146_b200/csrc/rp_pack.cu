// Row count R* and the length-only seed layout (Section 3.2 of the paper; first line of
// Algorithm 2), as one CTA on the GPU so that the whole plan stays stream-ordered.
//
// The samples are sorted by (-t_i, i) (by counting on the whole GPU, small and very large windows with a bitonic sort
// on 64-bit keys in the packing CTA), then for
// R = R_lb, R_lb+1, ... first-fit-decreasing is tried into K = R*D cells: the K longest
// samples open the cells, each later sample goes to the lowest-numbered cell it still fits
// in.  The fit search is done by one warp, 32 cells per ballot.
#include "rp_common.cuh"

#define PACK_THREADS 1024
#define FFD_MAX_CELLS 4096

// First fit of the samples keys[K..N) into K <= 1024*E cells by one warp, a run of samples at a time.
//
// Lane w keeps the largest remaining capacity of block w (32*E consecutive cells): a ballot finds the block, a second one
// the cell c that takes the next sample.  M, the largest remaining capacity below c, is what rejected it.  The samples
// behind it are no longer than it; they go to c as well as long as they are longer than M (no lower cell takes them) and
// fit after the ones before (prefix sums of the lengths, worked out once per 32 samples): one ballot gives the length of
// the run, and only then does a cell change.  Bound by the chain of warp-wide operations: about 440 cycles a run (38 runs
// for the 42 samples behind the first of a 64-sample window, 619 for 1808 at 2048, 349 for 8144 at 8192) instead of 170 to
// 250 a sample: 2048 samples in 270 k cycles, 4096 in 374 k (639 k with a tree of maxima searched by 32 samples at once,
// which placed 7 to 28 samples in 1800 cycles; 487 k and 393 k at 2048 and 8192, now 270 k and 228 k).
template <int E>
__device__ __forceinline__ bool first_fit_runs(const RpDims &dm, const u64 *keys, int *rem, int *cell_of, int K, int lane)
{
    // rem[32*32*E]: remaining capacities, -1 past the last cell
    int bm = -1;
    for (int x = 0; x < 32 * E; ++x) bm = max(bm, rem[lane * 32 * E + x]);
    for (int x0 = K; x0 < dm.N; x0 += 32) {
        const int nb = min(32, dm.N - x0);
        const u64 key = lane < nb ? keys[x0 + lane] : 0;
        const int len = lane < nb ? dm.C - (int)(key >> 32) : 0, id = (int)(u32)key;
        u32 pre = (u32)len;                         // at most 32*C, C <= 2^24
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const u32 y = __shfl_up_sync(0xffffffffu, pre, o); if (lane >= o) pre += y; }
        int p = 0;
        while (p < nb) {
            const int ts = __shfl_sync(0xffffffffu, len, p);
            const u32 base = __shfl_sync(0xffffffffu, pre, p) - (u32)ts;
            const unsigned m = __ballot_sync(0xffffffffu, bm >= ts);
            if (!m) return true;                    // the sample fits nowhere
            const int w = __ffs(m) - 1;
            int v[E];
            if (E == 1) v[0] = rem[w * 32 + lane];
            else {
                const int4 q = ((const int4 *)rem)[w * 32 + lane];
                v[0] = q.x; v[E > 1 ? 1 : 0] = q.y; v[E > 2 ? 2 : 0] = q.z; v[E > 3 ? 3 : 0] = q.w;
            }
            int big = v[0];
#pragma unroll
            for (int e = 1; e < E; ++e) big = max(big, v[e]);
            const int i = __ffs(__ballot_sync(0xffffffffu, big >= ts)) - 1;
            // first cell of lane i that takes it, what is left there, and the largest before it
            int f = E - 1, rc = 0, low = 0;
#pragma unroll
            for (int e = E - 1; e >= 0; --e) if (v[e] >= ts) f = e;
#pragma unroll
            for (int e = 0; e < E; ++e) { if (e == f) rc = v[e]; if (e < f) low = max(low, v[e]); }
            rc = __shfl_sync(0xffffffffu, rc, i);
            const unsigned below = (unsigned)max(lane < w ? bm : 0, lane < i ? max(big, 0) : (lane == i ? low : 0));
            const int M = (int)__reduce_max_sync(0xffffffffu, below);
            const bool in = lane < nb && len > M && pre - base <= (u32)rc;
            const unsigned out = __ballot_sync(0xffffffffu, lane > p && !in);      // p itself is always placed
            const int e1 = out ? __ffs(out) - 1 : 32;           // the run is p .. e1-1
            const int used = (int)(__shfl_sync(0xffffffffu, pre, e1 - 1) - base);
            const int ff = E == 1 ? 0 : __shfl_sync(0xffffffffu, f, i);
            if (lane >= p && lane < e1) cell_of[id] = (w * 32 + i) * E + ff;
            if (lane == i) {
#pragma unroll
                for (int e = 0; e < E; ++e) if (e == f) { v[e] = rc - used; rem[(w * 32 + i) * E + e] = v[e]; }
            }
            big = v[0];
#pragma unroll
            for (int e = 1; e < E; ++e) big = max(big, v[e]);
            const int nm = __reduce_max_sync(0xffffffffu, big);
            if (lane == w) bm = nm;
            __syncwarp();
            p = e1;
        }
    }
    return false;
}

__device__ __forceinline__ bool first_fit_smem(const RpDims &dm, const u64 *keys, int *fill, int *cell_of, int K, int B, int tid)
{
    const int b0 = tid * B, b1 = min(K, b0 + B);
    int blockmax = -1;
    for (int b = b0; b < b1; ++b) blockmax = max(blockmax, dm.C - fill[b]);
    for (int x = K; x < dm.N; ++x) {
        const u64 key = keys[x];
        const int ts = dm.C - (int)(key >> 32);
        const unsigned m = __ballot_sync(0xffffffffu, blockmax >= ts);
        if (!m) return true;
        if (tid == __ffs(m) - 1) {
            int found = -1, nm = -1;
            for (int b = b0; b < b1; ++b) {
                int rem = dm.C - fill[b];
                if (found < 0 && rem >= ts) { found = b; rem -= ts; fill[b] += ts; }
                nm = max(nm, rem);
            }
            blockmax = nm;
            cell_of[(u32)key] = found;
        }
    }
    return false;
}

// Packing runs beside the checks of the window: lengths outside [1, C] are still possible (the window is then refused).
// Kept within [0, C] they harm nobody here.
__device__ __forceinline__ int pack_len(const RpDims &dm, int t) { return min(max(t, 0), dm.C); }

// Position of every sample in the order (-t, i) by counting, over the whole GPU: RANK_PER samples per CTA, four threads
// each over a quarter of the lengths in shared memory.  N^2 comparisons (67 million at 8192 samples, a few microseconds);
// the one-CTA sort takes 82 us there.
#define RANK_THREADS 256
#define RANK_PER (RANK_THREADS / 4)
__global__ void __launch_bounds__(RANK_THREADS)
k_pack_rank(RpDims dm, const int *__restrict__ t, u64 *__restrict__ keys, int *__restrict__ order)
{
    extern __shared__ __align__(16) int len[];              // [N rounded up to 16], padded with -1 (shorter than any sample)
    const int tid = threadIdx.x, n16 = (dm.N + 15) & ~15;
    for (int i = tid; i < n16; i += RANK_THREADS) len[i] = i < dm.N ? pack_len(dm, __ldg(t + i)) : -1;
    __syncthreads();
    const int i = blockIdx.x * RANK_PER + (tid >> 2), part = tid & 3;
    const int ti = i < dm.N ? len[i] : 0x7fffffff;
    int before = 0;
    // chunks of four, dealt to the four threads in turn; a sample of the same length comes first if its index is lower
    for (int c = part; c < n16 / 4; c += 4) {
        const int4 v = ((const int4 *)len)[c];
        const int j = 4 * c;
        before += (v.x > ti || (v.x == ti && j < i)) + (v.y > ti || (v.y == ti && j + 1 < i))
                + (v.z > ti || (v.z == ti && j + 2 < i)) + (v.w > ti || (v.w == ti && j + 3 < i));
    }
    before += __shfl_xor_sync(0xffffffffu, before, 1);
    before += __shfl_xor_sync(0xffffffffu, before, 2);
    if (part == 0 && i < dm.N) { keys[before] = ((u64)(u32)(dm.C - ti) << 32) | (u32)i; order[before] = i; }
}

__global__ void __launch_bounds__(PACK_THREADS)
k_pack_ffd(RpDims dm, const int *__restrict__ t, int min_rows, u64 *keys_g, int n_pow2,
           int *__restrict__ fill_g, int *__restrict__ cell_of, int *__restrict__ out, int *__restrict__ order_out, const u64 *sorted)
{
    extern __shared__ __align__(16) u64 keys_s[];
    u64 *keys = keys_g ? keys_g : keys_s;
    int *fill = fill_g ? fill_g : (int *)(keys_s + (keys_g ? 0 : n_pow2));
    int *rem = fill;                               // remaining capacities (cells of the run-at-a-time form), else fills
    __shared__ i64 total_s;
    __shared__ int fail_s;
    const int tid = threadIdx.x, nt = (int)blockDim.x;
    if (tid == 0) total_s = 0;
    __syncthreads();
    i64 part = 0;
    for (int i = tid; i < n_pow2; i += nt) {
        if (i < dm.N) {
            part += t[i];
            const int ti = pack_len(dm, t[i]);
            keys[i] = sorted ? sorted[i] : ((u64)(u32)(dm.C - ti) << 32) | (u32)i;     // ascending = longest first, then id
        } else {
            keys[i] = ~0ull;
        }
    }
    for (int o = 16; o; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if ((tid & 31) == 0 && part) atomicAdd((u64 *)&total_s, (u64)part);
    __syncthreads();
    // Bitonic sort.  Element i sits with thread i % nt, so partners closer than 32 are
    // lanes of one warp: those exchanges run on registers with shuffles (no block-wide barrier),
    // the wider ones through the key array.
    constexpr int SORT_E = 8;                      // elements per thread at most (n_pow2 <= 8192 on this path)
    const bool in_regs = n_pow2 <= SORT_E * nt;
    for (int k = 2; k <= n_pow2 && !sorted; k <<= 1) {
        int j = k >> 1;
        for (; j >= 32 || (j > 0 && !in_regs); j >>= 1) {
            for (int i = tid; i < n_pow2; i += nt) {
                int ixj = i ^ j;
                if (ixj > i) {
                    u64 a = keys[i], b = keys[ixj];
                    bool up = ((i & k) == 0);
                    if ((a > b) == up) { keys[i] = b; keys[ixj] = a; }
                }
            }
            __syncthreads();
        }
        if (j > 0) {
            // all remaining distances of this k (and, while k <= 32, of the following k as well)
            u64 r[SORT_E];
#pragma unroll
            for (int m = 0; m < SORT_E; ++m) { const int i = m * nt + tid; r[m] = i < n_pow2 ? keys[i] : ~0ull; }
            int kk = k;
            for (;;) {
                for (int jj = min(kk >> 1, 16); jj > 0; jj >>= 1) {
#pragma unroll
                    for (int m = 0; m < SORT_E; ++m) {
                        const int i = m * nt + tid;
                        if (m * nt >= n_pow2) break;          // uniform: no element of this slot exists
                        const u64 o = __shfl_xor_sync(0xffffffffu, r[m], jj);
                        const bool up = ((i & kk) == 0), lower = ((tid & jj) == 0);
                        const u64 lo = r[m] < o ? r[m] : o, hi = r[m] < o ? o : r[m];
                        r[m] = (lower == up) ? lo : hi;
                    }
                }
                if (kk >= 32 || (kk << 1) > n_pow2) break;
                kk <<= 1;                                       // the next k still fits inside a warp
            }
            k = kk;
#pragma unroll
            for (int m = 0; m < SORT_E; ++m) { const int i = m * nt + tid; if (i < n_pow2) keys[i] = r[m]; }
            __syncthreads();
        }
    }
    if (!sorted) for (int x = tid; x < dm.N; x += nt) order_out[x] = (int)(u32)keys[x];   // samples by (-t, i)
    const i64 cap_row = (i64)dm.C * dm.D;
    i64 Rlb = (total_s + cap_row - 1) / cap_row;
    if (Rlb < 1) Rlb = 1;
    if (Rlb < min_rows) Rlb = min_rows;
    int Rstar = 0;
    for (i64 R = Rlb; R * dm.D <= dm.N && !Rstar; ++R) {
        const int K = (int)(R * dm.D);
        if (tid == 0) fail_s = 0;
        // the K longest samples open the cells
        for (int x = tid; x < K; x += nt) {
            const u64 key = keys[x];
            if (K > FFD_MAX_CELLS) fill[x] = dm.C - (int)(key >> 32);
            else rem[x] = (int)(key >> 32);                          // what is left of the cell
            cell_of[(u32)key] = x;
        }
        if (K <= FFD_MAX_CELLS) for (int x = K + tid; x < (K <= 1024 ? 1024 : FFD_MAX_CELLS); x += nt) rem[x] = -1;
        __syncthreads();
        if (tid < 32) {
            // First fit = the lowest cell whose remaining capacity takes the sample.
            const bool failed = K > FFD_MAX_CELLS ? first_fit_smem(dm, keys, fill, cell_of, K, (K + 31) / 32, tid)
                              : K <= 1024 ? first_fit_runs<1>(dm, keys, rem, cell_of, K, tid)
                                          : first_fit_runs<4>(dm, keys, rem, cell_of, K, tid);
            if (failed && tid == 0) fail_s = 1;
        }
        __syncthreads();
        if (!fail_s) Rstar = (int)R;
        __syncthreads();
    }
    if (tid == 0) {
        out[0] = Rstar;
        out[1] = (Rstar != 0 && Rstar == Rlb) ? 1 : 0;
        out[2] = (int)(Rlb > 0x7fffffff ? 0x7fffffff : Rlb);
        out[3] = (Rstar == 0);
    }
}

int rp_launch_pack(rp_ctx *c, int /*unused*/) { return rp_launch_pack_on(c, c->stream); }

int rp_launch_pack_on(rp_ctx *c, cudaStream_t stream)
{
    const RpDims &dm = c->dm;
    int n_pow2 = 1;
    while (n_pow2 < dm.N) n_pow2 <<= 1;
    // sort keys (8 bytes each) and cell fills (4 bytes per cell: at most N cells, or the padded blocks of the run-at-a-time
    // form) on chip when they fit
    const size_t fills = dm.N > (dm.N <= 1024 ? 1024 : FFD_MAX_CELLS) ? dm.N : (dm.N <= 1024 ? 1024 : FFD_MAX_CELLS);
    size_t smem = (size_t)n_pow2 * sizeof(u64) + fills * sizeof(int);
    u64 *keys_g = nullptr;
    int *fill_g = nullptr;
    if (smem > 160 * 1024) { keys_g = c->d_sort_keys; fill_g = (int *)(c->d_sort_keys + n_pow2); smem = 0; }
    if (smem > 32 * 1024)
        RP_CUDA(cudaFuncSetAttribute(k_pack_ffd, cudaFuncAttributeMaxDynamicSharedMemorySize, RP_SMEM_LIMIT));
    // small windows: fewer warps make the block-wide barriers of the sort cheaper
    const int threads = n_pow2 >= PACK_THREADS ? PACK_THREADS : (n_pow2 < 256 ? 256 : n_pow2);
    // The order by counting on the whole GPU from 513 samples (below, the sort in the packing kernel is cheaper than a
    // launch: 6.5 us at 512, 21 us at 2048) to 32768 (its work grows with the square).
    const u64 *sorted = nullptr;
    if (dm.N > 512 && dm.N <= 32768) {
        const size_t rs = sizeof(int) * (size_t)((dm.N + 15) & ~15);
        if (rs > 32 * 1024) RP_CUDA(cudaFuncSetAttribute(k_pack_rank, cudaFuncAttributeMaxDynamicSharedMemorySize, 128 * 1024));
        k_pack_rank<<<(dm.N + RANK_PER - 1) / RANK_PER, RANK_THREADS, rs, stream>>>(dm, c->d_t, c->d_sort_keys, c->d_order);
        ++g_rp_launches;
        sorted = c->d_sort_keys;
    }
    k_pack_ffd<<<1, threads, smem, stream>>>(dm, c->d_t, c->cfg.min_rows, keys_g, n_pow2, fill_g,
                                                    c->d_seed_layout, (int *)(c->h_pin + 10), c->d_order, sorted);
    ++g_rp_launches;
    RP_CUDA(cudaGetLastError());
    return RP_OK;
}
