// Row count R* and the length-only seed layout (Section 3.2 of the paper; first line of
// Algorithm 2), as one CTA on the GPU so that the whole plan stays stream-ordered.
//
// The samples are sorted by (-t_i, i) (by counting on the whole GPU, small and very large windows with a bitonic sort
// on 64-bit keys in the packing CTA), then for
// R = R_lb, R_lb+1, ... first-fit-decreasing is tried into K = R*D cells: the K longest
// samples open the cells, each later sample goes to the lowest-numbered cell it still fits in (first_fit_flow).
#include "rp_common.cuh"

#define PACK_THREADS 1024
#define FLOW_PHASE 8                  // cells between two meetings of the warps
#define FLOW_LAG (32 / FLOW_PHASE + 1)
#define FLOW_GONE 0x40000000u         // a sample that has found its cell, with the cell below (no cell has as much left)
#define FLOW_FEW 5120                 // samples up to which a lane holds eight of them, not sixteen
#define FLOW_PAD 48                   // zeros behind the capacities: the cells a warp's lanes see behind the last one

// First fit of 32*G samples a warp, in decreasing order over the lanes and warps, into K cells of `rest` (what is left of each; FLOW_PAD
// zeros behind them), the lowest cell first.
//
// Which samples a cell takes depends on nothing but the samples that no lower cell has taken, so the samples are a pipeline that the
// cells run through: a lane holds G consecutive samples, the capacity of a cell moves from lane to lane with one shuffle a step, and
// a sample that is taken keeps the cell's number in place of its length.  Between warps a cell goes through `rest` itself: warp w starts
// FLOW_LAG phases behind warp w-1, whose last lane has written a cell 31 steps after the first has read it.  About 100 cycles a step
// with eight samples a lane and 180 with sixteen (their chain of subtractions and minima, the shuffle), for N/G + K steps and the
// lags, whatever the lengths are; in cycles, 8 and 16 samples a lane: 512 samples in 72 cells 12 k and 15 k, 2048 in 240 56 k
// and 56 k, 4096 in 288 100 k and 112 k, 8192 in 48 120 k and 100 k.  (Samples that move through lanes of cells need a shuffle for every
// sample: 32 k, 97 k, 206 k and 261 k.  One warp that placed a run of samples at a time, before: 440 cycles a run, 270 k, 374 k and 228 k
// for the last three.)
template <int G>
__device__ __forceinline__ void first_fit_flow(u32 (&x)[G], u32 *rest, int K, int warp, int n_warps, int lane)
{
    const int phases = (K + 31 + FLOW_PHASE - 1) / FLOW_PHASE, all = phases + FLOW_LAG * (n_warps - 1);
    u32 r = 0;
    for (int ph = 0; ph < all; ++ph) {
        const int p = ph - FLOW_LAG * warp;
        if (p >= 0 && p < phases) {
            u32 in[FLOW_PHASE];
#pragma unroll
            for (int u = 0; u < FLOW_PHASE; u += 4) {
                const uint4 v = *(const uint4 *)(rest + p * FLOW_PHASE + u);
                in[u] = v.x; in[u + 1] = v.y; in[u + 2] = v.z; in[u + 3] = v.w;
            }
#pragma unroll
            for (int u = 0; u < FLOW_PHASE; ++u) {
                const int c = p * FLOW_PHASE + u;                       // lane 0 has cell c, the others the cells before it
                const u32 y = __shfl_up_sync(0xffffffffu, r, 1), tag = FLOW_GONE + (u32)(c - lane);
                r = lane ? y : in[u];
#pragma unroll
                for (int k = 0; k < G; ++k) {
                    const u32 left = r - x[k];                          // (more than r where it does not fit)
                    x[k] = x[k] <= r ? tag : x[k];
                    r = min(r, left);
                }
                if (lane == 31 && c >= 31 && c - 31 < K) rest[c - 31] = r;
            }
        }
        if (n_warps > 1) asm volatile("bar.sync 1, %0;" ::"r"(32 * n_warps) : "memory");
    }
}

// The samples behind the K longest, as many at a time as the CTA's lanes hold; whether one of this thread's has found no cell.
template <int G>
__device__ __forceinline__ bool first_fit(const RpDims &dm, const u64 *keys, u32 *rest, int *cell_of, int K, int tid, int nt)
{
    bool left = false;
    for (int b = K; b < dm.N; b += nt * G) {
        const int n_warps = (min(dm.N - b, nt * G) + 32 * G - 1) / (32 * G), first = b + tid * G;
        if (b > K) __syncthreads();                                     // the cells as the samples before have left them
        if (tid >> 5 >= n_warps) continue;
        u32 x[G];
#pragma unroll
        for (int k = 0; k < G; ++k) x[k] = first + k < dm.N ? max(1u, (u32)dm.C - (u32)(keys[first + k] >> 32)) : FLOW_GONE;
        first_fit_flow<G>(x, rest, K, tid >> 5, n_warps, tid & 31);
#pragma unroll
        for (int k = 0; k < G; ++k)
            if (first + k < dm.N) {
                left |= x[k] < FLOW_GONE;
                cell_of[(u32)keys[first + k]] = (int)(x[k] - FLOW_GONE);
            }
    }
    return left;
}

// Whether K cells are too few for the samples longer than a third of the cap, by this thread's share of them.  Among them the K longest open the
// cells and a cell takes one more at most.  Sample K + i fits beside the openers of up to C less its length, and so do all samples before
// it, i + 1 with it: there have to be i + 1 such openers, the last of which is opener K - 1 - i.  Where that holds for all of them the
// first fit places them all (it takes the longest opener that a sample fits beside); where it does not, it fails.  With more cells samples and
// openers of the same i are shorter: what holds for K cells holds for more.
__device__ __forceinline__ bool too_few_cells(const u64 *keys, int N, int C, int K, int tid, int nt)
{
    bool bad = false;
    for (int i = tid; i < min(N - K, K); i += nt) {
        const int s = C - (int)(keys[K + i] >> 32);
        if (3ll * s <= C) break;                                     // (nor is any behind it longer)
        bad |= s > (int)(keys[K - 1 - i] >> 32);
    }
    // a sample more than two to a cell, still that long
    if (tid == 0 && N - K > K) bad |= 3ll * (C - (int)(keys[2 * (size_t)K] >> 32)) > C;
    return bad;
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
k_pack_ffd(RpDims dm, const int *__restrict__ t, int min_rows, u64 *keys_g, int n_pow2, u32 *rest_g,
           int *__restrict__ cell_of, int *__restrict__ out, int *__restrict__ order_out, const u64 *sorted)
{
    extern __shared__ __align__(16) u64 keys_s[];
    u64 *sort = keys_g ? keys_g : keys_s;
    const u64 *keys = sorted ? sorted : sort;
    u32 *rest = rest_g ? rest_g : (u32 *)(keys_s + (sorted ? 0 : n_pow2));           // what is left of the cells
    __shared__ i64 total_s;
    __shared__ int fail_s;
    const int tid = threadIdx.x, nt = (int)blockDim.x;
    if (tid == 0) total_s = 0;
    __syncthreads();
    i64 part = 0;
    for (int i = tid; i < n_pow2; i += nt) {
        if (i < dm.N) {
            const int ti = t[i];
            part += ti;
            if (!sorted) sort[i] = ((u64)(u32)(dm.C - pack_len(dm, ti)) << 32) | (u32)i;     // ascending = longest first, then id
        } else if (!sorted) {
            sort[i] = ~0ull;
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
                    u64 a = sort[i], b = sort[ixj];
                    bool up = ((i & k) == 0);
                    if ((a > b) == up) { sort[i] = b; sort[ixj] = a; }
                }
            }
            __syncthreads();
        }
        if (j > 0) {
            // all remaining distances of this k (and, while k <= 32, of the following k as well)
            u64 r[SORT_E];
#pragma unroll
            for (int m = 0; m < SORT_E; ++m) { const int i = m * nt + tid; r[m] = i < n_pow2 ? sort[i] : ~0ull; }
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
            for (int m = 0; m < SORT_E; ++m) { const int i = m * nt + tid; if (i < n_pow2) sort[i] = r[m]; }
            __syncthreads();
        }
    }
    if (!sorted) for (int x = tid; x < dm.N; x += nt) order_out[x] = (int)(u32)keys[x];   // samples by (-t, i)
    const i64 cap_row = (i64)dm.C * dm.D;
    i64 Rlb = (total_s + cap_row - 1) / cap_row;
    if (Rlb < 1) Rlb = 1;
    if (Rlb < min_rows) Rlb = min_rows;
    int Rstar = 0;
    // Row counts that the samples of more than a third of the cap rule out are passed over, by halving: up to `low` rows are too few, `high` are
    // not, or more than there are samples for.  An attempt that fails costs as much as one that does not, and with such samples there
    // are many.  In us, every row count tried and so: 2000 samples of 17000 to 30000 tokens, cap 32768, 8 slots, 5390 and 26 (one run of samples at a
    // time, which ended at the first that fits nowhere, 419); 2048 of 34000 to 60000, 65536, 16, 2880 and 24 (232); 2000 of 12000 to 30000, 32768, 8,
    // 2070 and 95 (359); half of them 20000, half short 2325 and 77 (214).  Without such samples 52 and 52, 83 and 83 (2048 and 4096).  (Leaving the
    // pipeline as soon as a warp's samples have passed the last cell, too: 4 to 12 % on all packings for its test, little to gain.)
    i64 R0 = Rlb;
    const auto too_few = [&](i64 R) { return __syncthreads_or(too_few_cells(keys, dm.N, dm.C, (int)(R * dm.D), tid, nt)); };
    if (Rlb * dm.D < dm.N && 3ll * (dm.C - (int)(keys[Rlb * dm.D] >> 32)) > dm.C && too_few(Rlb)) {
        i64 low = Rlb, high = dm.N / dm.D + 1;
        while (high - low > 1) {
            const i64 mid = (low + high) / 2;
            if (too_few(mid)) low = mid; else high = mid;
        }
        R0 = high;
    }
    for (i64 R = R0; R * dm.D <= dm.N && !Rstar; ++R) {
        const int K = (int)(R * dm.D);
        if (tid == 0) fail_s = 0;
        // the K longest samples open the cells
        for (int x = tid; x < K + FLOW_PAD; x += nt) {
            const u64 key = x < K ? keys[x] : 0;
            rest[x] = (u32)(key >> 32);
            if (x < K) cell_of[(u32)key] = x;
        }
        __syncthreads();
        if (dm.N - K <= FLOW_FEW ? first_fit<8>(dm, keys, rest, cell_of, K, tid, nt) : first_fit<16>(dm, keys, rest, cell_of, K, tid, nt)) fail_s = 1;
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
    // On chip where they fit: the keys to sort (8 bytes each) and what is left of the cells (4; at most as many as samples).  Beyond,
    // in the two halves of the scratch.
    size_t smem = (sorted ? 0 : (size_t)n_pow2 * sizeof(u64)) + sizeof(u32) * ((size_t)dm.N + FLOW_PAD);
    u64 *keys_g = nullptr;
    u32 *rest_g = nullptr;
    if (smem > 160 * 1024) { keys_g = c->d_sort_keys; rest_g = (u32 *)(c->d_sort_keys + n_pow2); smem = 0; }
    if (smem > 32 * 1024)
        RP_CUDA(cudaFuncSetAttribute(k_pack_ffd, cudaFuncAttributeMaxDynamicSharedMemorySize, RP_SMEM_LIMIT));
    k_pack_ffd<<<1, threads, smem, stream>>>(dm, c->d_t, c->cfg.min_rows, keys_g, n_pow2, rest_g,
                                                    c->d_seed_layout, (int *)(c->h_pin + 10), c->d_order, sorted);
    ++g_rp_launches;
    RP_CUDA(cudaGetLastError());
    return RP_OK;
}
