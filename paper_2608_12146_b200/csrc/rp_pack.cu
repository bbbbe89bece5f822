// Row count R* and the length-only seed layout (Section 3.2 of the paper; first line of
// Algorithm 2), as one CTA on the GPU so that the whole plan stays stream-ordered.
//
// The samples are sorted by (-t_i, i) with a bitonic sort on 64-bit keys, then for
// R = R_lb, R_lb+1, ... first-fit-decreasing is tried into K = R*D cells: the K longest
// samples open the cells, each later sample goes to the lowest-numbered cell it still fits
// in.  The fit search is done by one warp, 32 cells per ballot.
#include "rp_common.cuh"

#define PACK_THREADS 1024

// First fit of the samples keys[K..N) into K cells by one warp, 32 samples at a time.
//
// Every lane looks up the lowest cell that takes its own sample, against the same state, in a tree of maxima (eight
// children per node, two 16-byte loads a level).  Samples come longest first, so the cells found do not increase from
// lane to lane and samples that found the same cell are neighbours: a segmented sum tells which of them still fit after
// the ones before; these are placed.  The others (and those behind them in their group) stay for the next round, ahead
// of new samples.  The order of placement does not matter: a sample that waits found a higher cell than every later
// sample placed meanwhile, so it does not fit where those went, and wherever it goes in the end lies higher.  A sample
// for which no cell is left has none in the one-by-one order either.
// One sample at a time cost 250 cycles (524 us on wide's 4096 samples); see k_pack_ffd for now.
#define FFD_LEVELS 4                        // 8^4 cells
#define FFD_MAX_CELLS 4096
__device__ __forceinline__ int max8(const int *p)
{
    const int4 a = ((const int4 *)p)[0], b = ((const int4 *)p)[1];
    return max(max(max(a.x, a.y), max(a.z, a.w)), max(max(b.x, b.y), max(b.z, b.w)));
}
__device__ __forceinline__ int first8(const int *p, int t)              // first of eight entries that is at least t
{
    const int4 a = ((const int4 *)p)[0], b = ((const int4 *)p)[1];
    const unsigned m = (a.x >= t ? 1u : 0u) | (a.y >= t ? 2u : 0u) | (a.z >= t ? 4u : 0u) | (a.w >= t ? 8u : 0u) |
                       (b.x >= t ? 16u : 0u) | (b.y >= t ? 32u : 0u) | (b.z >= t ? 64u : 0u) | (b.w >= t ? 128u : 0u);
    return __ffs(m) - 1;
}
// tree: levels from the leaves (remaining capacity, padded with -1) up; lev[x] = start of level x; depth levels, the last of at most 8 entries.
__device__ __forceinline__ bool first_fit_rounds(const RpDims &dm, const u64 *keys, int *tree, const int *lev, int depth, int *queue,
                                                 int *cell_of, int K, int lane)
{
    int len = 0, id = 0, kept = 0, next = K;
    bool have = false;
    for (;;) {
        // samples left over from the last round first, then new ones
        if (lane >= kept) {
            const int x = next + lane - kept;
            have = x < dm.N;
            if (have) { const u64 key = keys[x]; len = dm.C - (int)(key >> 32); id = (int)(u32)key; }
        }
        next += 32 - kept;
        if (!__any_sync(0xffffffffu, have)) return false;
        const int want = have ? len : 0x7fffffff;
        int c = 0;
        for (int l = depth - 1; l >= 0; --l) {
            const int f = first8(tree + lev[l] + 8 * c, want);
            c = 8 * c + (f < 0 ? 0 : f);
            if (l == depth - 1 && __any_sync(0xffffffffu, have && f < 0)) return true;           // nowhere to go
        }
        if (!have) c = -1;
        // length of the group before this lane
        const int before_c = __shfl_up_sync(0xffffffffu, c, 1);
        const bool head = lane == 0 || before_c != c;
        const unsigned heads = __ballot_sync(0xffffffffu, head);
        const int h = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));
        int sum = have ? len : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(0xffffffffu, sum, o); if (lane - o >= h) sum += y; }
        const int rem = have ? tree[lev[0] + c] : 0;
        const bool fits = have && sum <= rem;                        // sums grow along a group: true up to a lane, then false
        const unsigned ok = __ballot_sync(0xffffffffu, fits), wait = __ballot_sync(0xffffffffu, have && !fits);
        __syncwarp();
        if (fits) {
            cell_of[id] = c;
            const bool lastly = lane == 31 || ((heads >> (lane + 1)) & 1u) || !((ok >> (lane + 1)) & 1u);
            if (lastly) tree[lev[0] + c] = rem - sum;
        } else if (have) {
            const int at = __popc(wait & ((1u << lane) - 1u));
            queue[2 * at] = len; queue[2 * at + 1] = id;
        }
        __syncwarp();
        // maxima above the changed cells, level by level (several lanes may write the same value)
        for (int l = 1, n = c >> 3; l < depth; ++l, n >>= 3) {
            const int m = fits ? max8(tree + lev[l - 1] + 8 * n) : 0;
            __syncwarp();
            if (fits) tree[lev[l] + n] = m;
            __syncwarp();
        }
        kept = __popc(wait);
        if (lane < kept) { len = queue[2 * lane]; id = queue[2 * lane + 1]; have = true; }
        __syncwarp();
    }
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

__global__ void __launch_bounds__(PACK_THREADS)
k_pack_ffd(RpDims dm, const int *__restrict__ t, int min_rows, u64 *__restrict__ keys_g, int n_pow2,
           int *__restrict__ fill_g, int *__restrict__ cell_of, int *__restrict__ out, int *__restrict__ order_out)
{
    extern __shared__ __align__(16) u64 keys_s[];
    u64 *keys = keys_g ? keys_g : keys_s;
    int *fill = fill_g ? fill_g : (int *)(keys_s + (keys_g ? 0 : n_pow2));
    __shared__ __align__(16) int tree[FFD_MAX_CELLS + FFD_MAX_CELLS / 8 + FFD_MAX_CELLS / 64 + 8];
    __shared__ int queue[64], lev[FFD_LEVELS];
    __shared__ i64 total_s;
    __shared__ int fail_s;
    const int tid = threadIdx.x, nt = (int)blockDim.x;
    if (tid == 0) total_s = 0;
    __syncthreads();
    i64 part = 0;
    for (int i = tid; i < n_pow2; i += nt) {
        if (i < dm.N) {
            int ti = t[i];
            part += ti;
            keys[i] = ((u64)(u32)(dm.C - ti) << 32) | (u32)i;     // ascending = longest first, then id
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
    for (int k = 2; k <= n_pow2; k <<= 1) {
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
    for (int x = tid; x < dm.N; x += nt) order_out[x] = (int)(u32)keys[x];   // samples by (-t, i)
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
            else tree[x] = (int)(key >> 32);                         // what is left of the cell
            cell_of[(u32)key] = x;
        }
        int depth = 1;
        if (K <= FFD_MAX_CELLS) {
            int n = (K + 7) & ~7, at = 0;                             // entries of a level, padded to whole nodes
            for (int x = K + tid; x < n; x += nt) tree[x] = -1;
            if (tid == 0) lev[0] = 0;
            __syncthreads();
            for (; n > 8; ++depth) {
                const int up = n >> 3, upn = (up + 7) & ~7;
                for (int x = tid; x < upn; x += nt) tree[at + n + x] = x < up ? max8(tree + at + 8 * x) : -1;
                if (tid == 0) lev[depth] = at + n;
                at += n; n = upn;
                __syncthreads();
            }
        }
        __syncthreads();
        if (tid < 32) {
            // First fit = the lowest cell whose remaining capacity takes the sample.
            const bool failed = K <= FFD_MAX_CELLS ? first_fit_rounds(dm, keys, tree, lev, depth, queue, cell_of, K, tid)
                                                   : first_fit_smem(dm, keys, fill, cell_of, K, (K + 31) / 32, tid);
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
    // sort keys (8 bytes each) and cell fills (4 bytes per cell, at most N cells) on chip when they fit
    size_t smem = (size_t)n_pow2 * sizeof(u64) + (size_t)dm.N * sizeof(int);
    u64 *keys_g = nullptr;
    int *fill_g = nullptr;
    if (smem > 160 * 1024) { keys_g = c->d_sort_keys; fill_g = (int *)(c->d_sort_keys + n_pow2); smem = 0; }
    if (smem > 32 * 1024)
        RP_CUDA(cudaFuncSetAttribute(k_pack_ffd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    // small windows: fewer warps make the block-wide barriers of the sort cheaper
    const int threads = n_pow2 >= PACK_THREADS ? PACK_THREADS : (n_pow2 < 256 ? 256 : n_pow2);
    k_pack_ffd<<<1, threads, smem, stream>>>(dm, c->d_t, c->cfg.min_rows, keys_g, n_pow2, fill_g,
                                                    c->d_seed_layout, (int *)(c->h_pin + 10), c->d_order);
    ++g_rp_launches;
    RP_CUDA(cudaGetLastError());
    return RP_OK;
}
