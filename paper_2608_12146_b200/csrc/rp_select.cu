// Canonicalize, CanonicalMap and QualityDiversitySelect (Section 4.1.1, Algorithm 2) over the
// population as the candidate set.
//
//   signature   a cell is named by its smallest sample; inside a row the cells of one EDP shard
//               are listed by name over the shard's slots (increasing slot), rows are listed by
//               their smallest sample.  Equal signatures = same plan up to row order and
//               exchangeable slots.  A 64-bit hash of the signature finds the candidates for an
//               exact comparison.
//   map         the representative of a class has the lowest score, then the lowest index.
//   distance    Q20 units: cell co-assignment + row co-assignment (1 - pairs together in both /
//               pairs together in either) + sketch distance
//               floor(16 * sum_k sum_r |phi_k(x)[r] - phi_k(y)[r]| / (n_proj * R * F)),
//               phi_k = sorted projection of the Q16 row features (tokens / (C*D), squared
//               lengths / (C*C*D), busiest rank of every (shard, layer) / (k*C*|D_g|)) onto the
//               +-1 vector whose f-th sign is the top bit of Philox(f, 0, k, 7).x.
//   selection   starts from the lowest score; then the representative maximising
//               (distance to the nearest selected one) - ((eta_q16 * gap) >> 16), gap =
//               floor((S0 - S0*) * 2^20 / S0*), ties by lower index.
#include "rp_common.cuh"
#include <algorithm>

#define SEL_THREADS 256
#define SEL_WARPS (SEL_THREADS / 32)

struct SelBuf {                 // per-member arrays in global memory
    int *lay;                   // [P][N] layouts
    int *canon;                 // [P][N] signatures
    u64 *hash;                  // [P]
    u32 *lab;                   // [P][N] cell | row << 16
    int *big;                   // [P][2] samples of the largest cell, of the largest row
    int *clist, *cstart;        // [P][N], [P][K+1] samples grouped by cell
    int *rlist, *rstart;        // [P][N], [P][R+1] samples grouped by row
    i64 *pc, *pr;               // [P] pairs together in a cell / in a row
    i64 *phi;                   // [P][n_proj][R] sorted projections
};

__device__ __forceinline__ u64 sel_mix(u64 x)
{
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}

// ---- signs of the projections: sgn[k][f] = 1 where the entry is -1 -----------------------------
__global__ void k_sel_signs(int F, int n_proj, u32 key0, u32 key1, unsigned char *__restrict__ sgn)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= F * n_proj) return;
    const int k = x / F, f = x % F;
    sgn[x] = (unsigned char)(rp_philox((u32)f, 0u, (u32)k, 7u, key0, key1).x >> 31);
}

// ---- per member: signature, hash, groupings, sketch ---------------------------------------------
__global__ void __launch_bounds__(SEL_THREADS)
k_sel_prepare(RpDims dm, RpBlob bl, const char *__restrict__ blobs, const int *__restrict__ anc,
              const int *__restrict__ W_all, const int *__restrict__ wloc, const unsigned short *__restrict__ g_of_cell,
              const unsigned char *__restrict__ sgn, int n_proj, SelBuf B)
{
    extern __shared__ __align__(16) unsigned char sel_smem[];
    const int N = dm.N, K = dm.K, R = dm.R, D = dm.D, G = dm.G, L = dm.L, P = dm.P;
    const int F = 2 + G * L;
    i64 *ph = (i64 *)sel_smem;                     // [n_proj][R] projections
    int *name = (int *)(ph + (size_t)n_proj * R);  // [K] smallest sample of the cell
    int *new_d = name + K;                         // [K] slot inside the row
    int *rname = new_d + K;                        // [R]
    int *new_r = rname + R;                        // [R]
    int *ccount = new_r + R;                       // [K + 1]
    int *rcount = ccount + K + 1;                  // [R + 1]
    int *ng = rcount + R + 1;                      // [G] slots per shard
    __shared__ u64 hsum;
    __shared__ i64 pcs, prs;
    __shared__ int big_s[2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int j = blockIdx.x;
    const int *lay = B.lay + (size_t)j * N;
    const char *blob = blobs + (size_t)anc[j] * bl.bytes;
    const int *T = (const int *)(blob + bl.off_T);
    const u64 *Q = (const u64 *)(blob + bl.off_Q);
    const int *W = W_all + (size_t)wloc[j] * dm.RG * dm.LP;

    for (int c = tid; c < K; c += SEL_THREADS) name[c] = N;
    for (int c = tid; c <= K; c += SEL_THREADS) ccount[c] = 0;
    for (int r = tid; r <= R; r += SEL_THREADS) rcount[r] = 0;
    for (int r = tid; r < R; r += SEL_THREADS) rname[r] = N;
    for (int g = tid; g < G; g += SEL_THREADS) ng[g] = 0;
    if (tid == 0) { hsum = 0; pcs = 0; prs = 0; big_s[0] = 0; big_s[1] = 0; }
    __syncthreads();
    for (int i = tid; i < N; i += SEL_THREADS) {
        const int c = lay[i], r = c / D;
        B.lab[(size_t)j * N + i] = (u32)c | ((u32)r << 16);
        atomicMin(&name[c], i);
        atomicAdd(&ccount[c + 1], 1);
        atomicAdd(&rcount[r + 1], 1);
    }
    for (int d = tid; d < D; d += SEL_THREADS) atomicAdd(&ng[g_of_cell[d]], 1);
    __syncthreads();
    for (int c = tid; c < K; c += SEL_THREADS) atomicMin(&rname[c / D], name[c]);
    {   // pairs together, from the group sizes
        i64 a = 0, b = 0;
        int ma = 0, mb = 0;
        for (int c = tid; c < K; c += SEL_THREADS) { const int n = ccount[c + 1]; a += (i64)n * (n - 1) / 2; ma = max(ma, n); }
        for (int r = tid; r < R; r += SEL_THREADS) { const int n = rcount[r + 1]; b += (i64)n * (n - 1) / 2; mb = max(mb, n); }
        ma = __reduce_max_sync(0xffffffffu, ma); mb = __reduce_max_sync(0xffffffffu, mb);
        if (lane == 0) { atomicMax(&big_s[0], ma); atomicMax(&big_s[1], mb); }
        if (a) atomicAdd((u64 *)&pcs, (u64)a);
        if (b) atomicAdd((u64 *)&prs, (u64)b);
    }
    __syncthreads();
    // position of every cell among the cells of its shard in its row, and of every row
    for (int c = tid; c < K; c += SEL_THREADS) {
        const int r = c / D, g = g_of_cell[c];
        int pos = 0;
        for (int d2 = 0; d2 < D; ++d2) pos += (g_of_cell[r * D + d2] == g && name[r * D + d2] < name[c]);
        int seen = 0, target = -1;
        for (int d2 = 0; d2 < D && target < 0; ++d2)
            if (g_of_cell[d2] == g) { if (seen == pos) target = d2; ++seen; }
        new_d[c] = target;
    }
    for (int r = tid; r < R; r += SEL_THREADS) {
        int pos = 0;
        for (int r2 = 0; r2 < R; ++r2) pos += (rname[r2] < rname[r]);
        new_r[r] = pos;
    }
    if (warp < 2) {              // starts of the groups: prefix sums of the sizes (one place on), a warp for cells, one for rows
        int *count = warp ? rcount : ccount;
        const int n = warp ? R : K;
        int run = 0;
        for (int x0 = 0; x0 <= n; x0 += 32) {
            const int x = x0 + lane;
            int v = x <= n ? count[x] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(0xffffffffu, v, o); if (lane >= o) v += y; }
            if (x <= n) count[x] = run + v;
            run += __shfl_sync(0xffffffffu, v, 31);
        }
    }
    __syncthreads();
    for (int c = tid; c <= K; c += SEL_THREADS) B.cstart[(size_t)j * (K + 1) + c] = ccount[c];
    for (int r = tid; r <= R; r += SEL_THREADS) B.rstart[(size_t)j * (R + 1) + r] = rcount[r];
    {
        u64 h = 0;
        for (int i = tid; i < N; i += SEL_THREADS) {
            const int c = lay[i];
            const int cn = new_r[c / D] * D + new_d[c];
            B.canon[(size_t)j * N + i] = cn;
            h += sel_mix((u64)i * (u64)K + (u64)cn);
        }
        atomicAdd((unsigned long long *)&hsum, (unsigned long long)h);
    }
    __syncthreads();
    // group lists (order inside a group does not matter to the pair counts)
    for (int i = tid; i < N; i += SEL_THREADS) {
        const int c = lay[i];
        B.clist[(size_t)j * N + atomicAdd(&ccount[c], 1)] = i;
        B.rlist[(size_t)j * N + atomicAdd(&rcount[c / D], 1)] = i;
    }
    // row features -> projections: one warp per row, lanes over the features, eight projections summed in registers at a time
    // (64-bit shared-memory atomics of all lanes on one row's sums took most of this kernel: 256 members of 2048 samples and 24
    // layers 500 us, now 84)
    const i64 CD = (i64)dm.C * D;
    for (int r = warp; r < R; r += SEL_WARPS) {
        for (int k0 = 0; k0 < n_proj; k0 += 8) {
            i64 acc[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) acc[k] = 0;
            for (int f = lane; f < F; f += 32) {
                i64 h;
                if (f < 2) {
                    if (f == 0) { i64 s = 0; for (int d = 0; d < D; ++d) s += T[r * D + d]; h = (s << 16) / CD; }
                    else { u64 s = 0; for (int d = 0; d < D; ++d) s += Q[r * D + d]; h = (i64)((s << 16) / ((u64)CD * (u64)dm.C)); }
                } else {
                    const int g = (f - 2) / L, l = (f - 2) % L;
                    const int *wr = W + ((size_t)r * G + g) * dm.LP + (size_t)l * P;
                    int m = 0;
                    if (P % 4 == 0) {
                        for (int p = 0; p < P; p += 4) { const int4 w = *(const int4 *)(wr + p); m = max(max(m, max(w.x, w.y)), max(w.z, w.w)); }
                    } else {
                        for (int p = 0; p < P; ++p) m = max(m, wr[p]);
                    }
                    h = ((i64)m << 16) / ((i64)dm.k * dm.C * ng[g]);
                }
#pragma unroll
                for (int k = 0; k < 8; ++k) if (k0 + k < n_proj) acc[k] += sgn[(size_t)(k0 + k) * F + f] ? -h : h;
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                for (int o = 16; o; o >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
                if (lane == 0 && k0 + k < n_proj) ph[(k0 + k) * R + r] = acc[k];
            }
        }
    }
    __syncthreads();
    for (int x = tid; x < n_proj * R; x += SEL_THREADS) {        // sort each projection by counting
        const int k = x / R, r = x % R;
        const i64 v = ph[x];
        int pos = 0;
        for (int r2 = 0; r2 < R; ++r2) { const i64 o = ph[k * R + r2]; pos += (o < v) || (o == v && r2 < r); }
        B.phi[((size_t)j * n_proj + k) * R + pos] = v;
    }
    if (tid == 0) { B.hash[j] = hsum; B.pc[j] = pcs; B.pr[j] = prs; B.big[2 * j] = big_s[0]; B.big[2 * j + 1] = big_s[1]; }
}

// ---- CanonicalMap: is member j the representative of its class? ---------------------------------
__global__ void __launch_bounds__(SEL_THREADS)
k_sel_map(int N, int Ppop, const int *__restrict__ canon, const u64 *__restrict__ hash,
          const i64 *__restrict__ score, int *__restrict__ rep)
{
    __shared__ int beaten;
    const int j = blockIdx.x;
    if (threadIdx.x == 0) beaten = 0;
    __syncthreads();
    const u64 hj = hash[j];
    const i64 a0 = score[3 * (size_t)j], a1 = score[3 * (size_t)j + 1], a2 = score[3 * (size_t)j + 2];
    const int lane = threadIdx.x & 31;
    for (int o0 = threadIdx.x - lane; o0 < Ppop; o0 += SEL_THREADS) {
        const int mine = o0 + lane;
        for (unsigned todo = __ballot_sync(0xffffffffu, mine < Ppop && mine != j && hash[min(mine, Ppop - 1)] == hj); todo; todo &= todo - 1) {
            const int o = o0 + __ffs(todo) - 1;        // the whole warp compares the two signatures
            bool same = true;
            for (int i = lane; i < N && same; i += 32) same = canon[(size_t)j * N + i] == canon[(size_t)o * N + i];
            if (!__all_sync(0xffffffffu, same)) continue;
            const i64 b0 = score[3 * (size_t)o], b1 = score[3 * (size_t)o + 1], b2 = score[3 * (size_t)o + 2];
            if (rp_lex_less(b0, b1, b2, a0, a1, a2) || (!rp_lex_less(a0, a1, a2, b0, b1, b2) && o < j)) beaten = 1;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) rep[j] = !beaten;
}

// ---- plan distances between representatives ------------------------------------------------------
// Pairs together in a group of both plans = sum over (group of a, group of b) of C(count, 2).  Every sample adds one to the
// count of its pair of groups in shared memory; what the atomic returns is the number of samples before it there, and these
// sum up to C(count, 2): no pass over the table.  Clearing stores a zero at the same places.  Bound by the shared-memory
// atomics, two a sample (cells and rows): 32640 pairs of plans of 2048 samples in 240 cells 0.23 ms (0.28 with eight warps' 64-bit
// additions to one address and groups fetched twice; the next plan's groups fetched ahead gave nothing); looking every pair of a
// cell's samples up in the other plan took 4.15 ms.
//
// Counts are as narrow as the largest group of a allows when the whole table fits only so (8 bits up to 255 samples); where
// no width fits, the groups of a are taken in blocks, whose samples are contiguous in a's grouped list.
#define SEL_CHUNK 8             // plans b per work item
#define SEL_HELD 8              // samples a thread keeps in registers
struct SelTab { u32 *tab; int n, lbits, block; };      // n groups; counts of 2^lbits bits; groups of a per pass

__device__ __forceinline__ SelTab sel_table(u32 *tab, size_t bytes, int n, int big)
{
    SelTab t = { tab, n, 5, n };
    const size_t bits = bytes * 8, all = (size_t)n * n;
    if (all * 32 > bits && big <= 65535) t.lbits = 4;
    if (t.lbits == 4 && all * 16 > bits && big <= 255) t.lbits = 3;
    if ((all << t.lbits) > bits) t.block = (int)((bits >> t.lbits) / n);
    return t;
}

__device__ __forceinline__ u32 sel_add(const SelTab &t, int x)
{
    const int per = 5 - t.lbits, sh = (x & ((1 << per) - 1)) << t.lbits;
    const u32 old = atomicAdd(&t.tab[x >> per], 1u << sh);
    return (old >> sh) & (0xffffffffu >> (32 - (1 << t.lbits)));
}

__device__ __forceinline__ void sel_clear(const SelTab &t, int x) { t.tab[x >> (5 - t.lbits)] = 0; }

// The same in blocks of a's groups; SH = 0 for cells, 16 for rows.
template <typename SUM, int SH>
__device__ __forceinline__ SUM sel_blocks(const SelTab &t, const int *list, const int *start, const u32 *la, const u32 *lb, int tid)
{
    SUM sum = 0;
    for (int g0 = 0; g0 < t.n; g0 += t.block) {
        const int x0 = start[g0], x1 = start[min(t.n, g0 + t.block)];
        for (int pass = 0; pass < 2; ++pass) {
            for (int x = x0 + tid; x < x1; x += SEL_THREADS) {
                const int i = list[x];
                const int at = ((int)((la[i] >> SH) & 0xffffu) - g0) * t.n + (int)((lb[i] >> SH) & 0xffffu);
                if (pass == 0) sum += sel_add(t, at); else sel_clear(t, at);
            }
            __syncthreads();
        }
    }
    return sum;
}

// SUM: 32 bits hold the pairs of up to 65535 samples.
template <typename SUM>
__global__ void __launch_bounds__(SEL_THREADS, 3)
k_sel_dist(RpDims dm, int Ppop, int n_proj, const int *__restrict__ rep, SelBuf B, i64 *__restrict__ dist, int ctab_bytes, int rtab_bytes)
{
    extern __shared__ __align__(16) u32 sel_tabs[];
    __shared__ u64 acc[SEL_CHUNK][3][SEL_WARPS];         // (a place a warp: 64-bit additions of eight warps to one address queue up)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int N = dm.N, K = dm.K, R = dm.R, F = 2 + dm.G * dm.L;
    const bool held = N <= SEL_HELD * SEL_THREADS;       // a thread's samples fit its registers
    for (int x = tid; x < (ctab_bytes + rtab_bytes) / 4; x += SEL_THREADS) sel_tabs[x] = 0;
    const int chunks = (Ppop + SEL_CHUNK - 1) / SEL_CHUNK;
    for (size_t item = blockIdx.x; item < (size_t)chunks * Ppop; item += gridDim.x) {
        const int a = (int)(item % Ppop), b0 = (int)(item / Ppop) * SEL_CHUNK;
        if (b0 + SEL_CHUNK - 1 <= a || !rep[a]) continue;
        __syncthreads();
        const SelTab ct = sel_table(sel_tabs, ctab_bytes, K, B.big[2 * a]), rt = sel_table(sel_tabs + ctab_bytes / 4, rtab_bytes, R, B.big[2 * a + 1]);
        const bool whole = ct.block == K && rt.block == R;
        const u32 *la = B.lab + (size_t)a * N;
        const i64 *pa = B.phi + (size_t)a * n_proj * R;
        int ca[SEL_HELD], ra[SEL_HELD];                          // where the samples' groups of a start in the tables
        if (held)
#pragma unroll
            for (int x = 0; x < SEL_HELD; ++x) {
                const int i = tid + x * SEL_THREADS;
                const u32 ga = i < N ? la[i] : 0;
                ca[x] = (int)(ga & 0xffffu) * K; ra[x] = (int)(ga >> 16) * R;
            }
        for (int u = 0; u < SEL_CHUNK; ++u) {
            const int b = b0 + u;
            if (b <= a || b >= Ppop || !rep[b]) continue;
            const u32 *lb = B.lab + (size_t)b * N;
            SUM bc = 0, br = 0;
            if (whole && held) {
                u32 gb[SEL_HELD];
#pragma unroll
                for (int x = 0; x < SEL_HELD; ++x) gb[x] = tid + x * SEL_THREADS < N ? __ldg(lb + tid + x * SEL_THREADS) : 0;
#pragma unroll
                for (int x = 0; x < SEL_HELD; ++x)
                    if (tid + x * SEL_THREADS < N) {
                        bc += sel_add(ct, ca[x] + (int)(gb[x] & 0xffffu));
                        br += sel_add(rt, ra[x] + (int)(gb[x] >> 16));
                    }
                __syncthreads();
#pragma unroll
                for (int x = 0; x < SEL_HELD; ++x)
                    if (tid + x * SEL_THREADS < N) { sel_clear(ct, ca[x] + (int)(gb[x] & 0xffffu)); sel_clear(rt, ra[x] + (int)(gb[x] >> 16)); }
            } else if (whole) {
#pragma unroll 4
                for (int i = tid; i < N; i += SEL_THREADS) {
                    const u32 ga = la[i], gb = lb[i];
                    bc += sel_add(ct, (int)(ga & 0xffffu) * K + (int)(gb & 0xffffu));
                    br += sel_add(rt, (int)(ga >> 16) * R + (int)(gb >> 16));
                }
                __syncthreads();
#pragma unroll 4
                for (int i = tid; i < N; i += SEL_THREADS) {
                    const u32 ga = la[i], gb = lb[i];
                    sel_clear(ct, (int)(ga & 0xffffu) * K + (int)(gb & 0xffffu));
                    sel_clear(rt, (int)(ga >> 16) * R + (int)(gb >> 16));
                }
            } else {
                bc = sel_blocks<SUM, 0>(ct, B.clist + (size_t)a * N, B.cstart + (size_t)a * (K + 1), la, lb, tid);
                br = sel_blocks<SUM, 16>(rt, B.rlist + (size_t)a * N, B.rstart + (size_t)a * (R + 1), la, lb, tid);
            }
            const i64 *pb = B.phi + (size_t)b * n_proj * R;
            i64 sw = 0;                                          // sketch
            for (int x = tid; x < n_proj * R; x += SEL_THREADS) { const i64 d = pa[x] - pb[x]; sw += d < 0 ? -d : d; }
            if (tid - lane < n_proj * R) for (int o = 16; o; o >>= 1) sw += __shfl_xor_sync(0xffffffffu, sw, o);
            if (sizeof(SUM) == 4) {
                const u32 sc = __reduce_add_sync(0xffffffffu, (u32)bc), sr = __reduce_add_sync(0xffffffffu, (u32)br);
                bc = sc; br = sr;
            } else {
                for (int o = 16; o; o >>= 1) { bc += __shfl_xor_sync(0xffffffffu, bc, o); br += __shfl_xor_sync(0xffffffffu, br, o); }
            }
            if (lane == 0) { acc[u][0][warp] = (u64)bc; acc[u][1][warp] = (u64)br; acc[u][2][warp] = (u64)sw; }
            __syncthreads();                                     // tables are clear again
        }
        const int b = b0 + tid;
        if (tid < SEL_CHUNK && b > a && b < Ppop && rep[b]) {
            i64 bc = 0, br = 0, sw = 0;
#pragma unroll
            for (int w = 0; w < SEL_WARPS; ++w) { bc += (i64)acc[tid][0][w]; br += (i64)acc[tid][1][w]; sw += (i64)acc[tid][2][w]; }
            const i64 uc = B.pc[a] + B.pc[b] - bc, ur = B.pr[a] + B.pr[b] - br;
            i64 d = 0;
            if (uc) d += ((i64)1 << 20) - (bc << 20) / uc;
            if (ur) d += ((i64)1 << 20) - (br << 20) / ur;
            d += (sw * 16) / ((i64)n_proj * R * F);
            dist[(size_t)a * Ppop + b] = d;
            dist[(size_t)b * Ppop + a] = d;
        }
        __syncthreads();
    }
}

// ---- greedy selection (one CTA) -------------------------------------------------------------------
// One selection after the other: a step is the load of one row of distances, three warp-wide minima, one barrier and the
// same minima over the warps' results, which every warp works out for itself (256 candidates, distances in L2, 220 us; a shuffle tree
// over triples, a serial pass of one thread and two barriers over 32 warps took 920); by a single warp where the distances are on chip.
#define GREEDY_THREADS 1024
#define GREEDY_SMEM (160 * 1024)        // nearest distances and penalties of the candidates on chip up to this
// The distances themselves on chip, each pair once, where they fit (up to 307 candidates): a step then does not wait for L2 (256
// candidates 220 -> 196 us).  In 32 bits: the two co-assignments are at most 2^20 each, and the sketch at most 2^21, since every row
// feature of a plan within the cap is at most 2^16.
#define GREEDY_DIST_MAX (184 * 1024)
static inline size_t greedy_tri(size_t P) { return P * (P - 1) / 2; }
struct SelPick { i64 v0, v1, v2; int j; };

// The steps by one warp, E candidates a lane: distances to the nearest selected one and penalties in registers, pairs in `near`; penalties
// below 2^30.  A step is a load, a minimum and a compare a candidate and two warp-wide minima, and no barrier (256 candidates 196 -> 70 us; 253
// where a branch around each load made one wait for the other).
template <int E>
__device__ __forceinline__ void greedy_by_warp(int Ppop, int nd, int last, const u32 *near, const i64 *mind, const i64 *pen, int *__restrict__ order, int lane)
{
    u32 m[E], p[E], left = 0;                                    // left: candidates not selected yet
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int j = lane + 32 * e;
        const bool on = j < Ppop && mind[min(j, Ppop - 1)] >= 0;
        m[e] = 0xffffffffu; p[e] = on ? (u32)pen[j] : 0;
        left |= on ? 1u << e : 0;
    }
    for (int n = 0; n < nd; ++n) {
        if (lane == 0) order[n] = last;
        if (lane == (last & 31)) left &= ~(1u << (last >> 5));
        const int row = last * (last - 1) / 2;
        u32 best = 0xffffffffu, who = 0xffffffffu, d[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {                            // (all at once: an entry that is not used is read, at 0)
            const int j = lane + 32 * e, at = j > last ? j * (j - 1) / 2 + last : row + j;
            d[e] = near[(left >> e) & 1u ? at : 0];
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
            m[e] = min(m[e], d[e]);
            const u32 key = (left >> e) & 1u ? p[e] - m[e] + 0x80000000u : 0xffffffffu;
            who = key < best ? (u32)(lane + 32 * e) : who;       // (ties: the lower index)
            best = min(best, key);
        }
        const u32 top = __reduce_min_sync(0xffffffffu, best);
        last = (int)__reduce_min_sync(0xffffffffu, best == top ? who : 0xffffffffu);
    }
}

__global__ void __launch_bounds__(GREEDY_THREADS)
k_sel_greedy(int Ppop, const int *__restrict__ rep, const i64 *__restrict__ score, const i64 *__restrict__ dist,
             i64 eta_q16, i64 *mind, i64 *pen, int *__restrict__ order, int *__restrict__ n_distinct, int tri)
{
    __shared__ SelPick red[GREEDY_THREADS / 32];
    __shared__ SelPick pick_s;
    __shared__ int nd_s;
    __shared__ u64 red_v[2][GREEDY_THREADS / 32];
    __shared__ int red_j[2][GREEDY_THREADS / 32];
    extern __shared__ __align__(16) i64 greedy_smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = (int)blockDim.x, nw = nt / 32;
    if (!mind) { mind = greedy_smem; pen = mind + Ppop; }
    if (tid == 0) nd_s = 0;
    __syncthreads();
    // winner by score (lowest triple, lowest index) and the number of representatives
    SelPick best = { 0x7fffffffffffffffll, 0x7fffffffffffffffll, 0x7fffffffffffffffll, 0x7fffffff };
    int cnt = 0;
    for (int j = tid; j < Ppop; j += nt) {
        if (!rep[j]) continue;
        ++cnt;
        const i64 s0 = score[3 * (size_t)j], s1 = score[3 * (size_t)j + 1], s2 = score[3 * (size_t)j + 2];
        if (rp_lex_less(s0, s1, s2, best.v0, best.v1, best.v2)) { best.v0 = s0; best.v1 = s1; best.v2 = s2; best.j = j; }
    }
    if (cnt) atomicAdd(&nd_s, cnt);
    auto reduce_min = [&](SelPick b) {
        for (int o = 16; o; o >>= 1) {
            SelPick ot;
            ot.v0 = __shfl_xor_sync(0xffffffffu, b.v0, o); ot.v1 = __shfl_xor_sync(0xffffffffu, b.v1, o);
            ot.v2 = __shfl_xor_sync(0xffffffffu, b.v2, o); ot.j = __shfl_xor_sync(0xffffffffu, b.j, o);
            if (rp_lex_less(ot.v0, ot.v1, ot.v2, b.v0, b.v1, b.v2) ||
                (ot.v0 == b.v0 && ot.v1 == b.v1 && ot.v2 == b.v2 && ot.j < b.j)) b = ot;
        }
        if (lane == 0) red[warp] = b;
        __syncthreads();
        if (tid == 0) {
            for (int w = 1; w < nw; ++w) {
                const SelPick ot = red[w];
                if (rp_lex_less(ot.v0, ot.v1, ot.v2, b.v0, b.v1, b.v2) ||
                    (ot.v0 == b.v0 && ot.v1 == b.v1 && ot.v2 == b.v2 && ot.j < b.j)) b = ot;
            }
            pick_s = b;
        }
        __syncthreads();
    };
    reduce_min(best);
    const int nd = nd_s;
    const i64 s0 = pick_s.v0;
    int last = pick_s.j;
    bool large = false;                                    // a penalty that 30 bits do not hold
    for (int j = tid; j < Ppop; j += nt) {
        i64 p = 0;
        if (rep[j] && s0 > 0) {
            const unsigned __int128 gap = ((unsigned __int128)(u64)(score[3 * (size_t)j] - s0) << 20) / (u64)s0;
            p = (i64)((gap * (unsigned __int128)(u64)eta_q16) >> 16);
        }
        pen[j] = p;
        large |= (u64)p >> 30;
        mind[j] = rep[j] ? 0x7fffffffffffffffll : -1;      // -1 = not a candidate (or already selected)
    }
    __syncthreads();
    // pair (i, j), i > j, at i (i - 1) / 2 + j
    u32 *near = (u32 *)(greedy_smem + 2 * (size_t)Ppop);
    if (tri) {
        for (int i = warp; i < Ppop; i += nw)                        // (no distance is used to a plan that stands for no class)
#pragma unroll 8
            for (int j = lane; j < i; j += 32) near[i * (i - 1) / 2 + j] = (u32)__ldg(dist + (size_t)i * Ppop + j);
    }
    large = __syncthreads_or(large);
    if (tri && !large) {
        if (warp == 0) {
            if (Ppop <= 64) greedy_by_warp<2>(Ppop, nd, last, near, mind, pen, order, lane);
            else if (Ppop <= 128) greedy_by_warp<4>(Ppop, nd, last, near, mind, pen, order, lane);
            else if (Ppop <= 256) greedy_by_warp<8>(Ppop, nd, last, near, mind, pen, order, lane);
            else greedy_by_warp<10>(Ppop, nd, last, near, mind, pen, order, lane);
        }
        __syncthreads();
    } else
    for (int n = 0; n < nd; ++n) {
        if (tid == 0) order[n] = last;
        // negated objective, as an unsigned number, so that the minimum applies: maximise distance - penalty, lowest index
        u64 bv = ~0ull;
        u32 bj = 0xffffffffu;
        for (int j = tid; j < Ppop; j += nt) {
            i64 m = mind[j];
            if (j == last) { mind[j] = -1; m = -1; }
            if (m < 0) continue;
            const int hi = max(last, j);
            const i64 d = tri ? (i64)near[hi * (hi - 1) / 2 + (last + j - hi)] : dist[(size_t)last * Ppop + j];
            if (d < m) { m = d; mind[j] = m; }
            const u64 neg = (u64)(pen[j] - m) ^ 0x8000000000000000ull;
            if (neg < bv) { bv = neg; bj = (u32)j; }
        }
        for (int pass = 0; pass < 2; ++pass) {
            const u32 hi = __reduce_min_sync(0xffffffffu, (u32)(bv >> 32));
            const bool in = (u32)(bv >> 32) == hi;
            const u32 lo = __reduce_min_sync(0xffffffffu, in ? (u32)bv : 0xffffffffu);
            bj = __reduce_min_sync(0xffffffffu, in && (u32)bv == lo ? bj : 0xffffffffu);
            bv = ((u64)hi << 32) | lo;
            if (pass) break;
            if (lane == 0) { red_v[n & 1][warp] = bv; red_j[n & 1][warp] = (int)bj; }
            __syncthreads();
            bv = lane < nw ? red_v[n & 1][lane] : ~0ull;
            bj = lane < nw ? (u32)red_j[n & 1][lane] : 0xffffffffu;
        }
        last = (int)bj;
    }
    for (int m = nd + tid; m < Ppop; m += nt) order[m] = order[m % nd];
    if (tid == 0) *n_distinct = nd;
}

__global__ void k_sel_fill(int N, const int *__restrict__ order, const int *__restrict__ lay, int *__restrict__ out)
{
    const int m = blockIdx.x;
    const int *src = lay + (size_t)order[m] * N;
    for (int i = threadIdx.x; i < N; i += blockDim.x) out[(size_t)m * N + i] = src[i];
}

// lay [P][N]: the population's layouts (input); out [P][N]: the selected population.
// score [P][3]: exact scores of the members.  order [P], n_distinct [1], dist [P][P] device outputs.
int rp_launch_select(rp_ctx *c, int *lay, int *out, const i64 *score, int n_proj, i64 eta_q16, int *order,
                     int *n_distinct, i64 *dist)
{
    const RpDims &dm = c->dm;
    const size_t P = (size_t)c->Ppop;
    const int F = 2 + dm.G * dm.L;
    SelBuf B;
    B.lay = lay;
    unsigned char *sgn = nullptr;
    int *rep = nullptr;
    i64 *mind = nullptr, *pen = nullptr;
    B.canon = nullptr; B.hash = nullptr; B.clist = nullptr; B.cstart = nullptr; B.rlist = nullptr; B.rstart = nullptr;
    B.pc = nullptr; B.pr = nullptr; B.phi = nullptr; B.lab = nullptr; B.big = nullptr;
    int st = dev_alloc(c, &B.canon, P * dm.N);
    if (st == RP_OK) st = dev_alloc(c, &B.hash, P);
    if (st == RP_OK) st = dev_alloc(c, &B.lab, P * dm.N);
    if (st == RP_OK) st = dev_alloc(c, &B.big, 2 * P);
    if (st == RP_OK) st = dev_alloc(c, &B.clist, P * dm.N);
    if (st == RP_OK) st = dev_alloc(c, &B.cstart, P * (dm.K + 1));
    if (st == RP_OK) st = dev_alloc(c, &B.rlist, P * dm.N);
    if (st == RP_OK) st = dev_alloc(c, &B.rstart, P * (dm.R + 1));
    if (st == RP_OK) st = dev_alloc(c, &B.pc, P);
    if (st == RP_OK) st = dev_alloc(c, &B.pr, P);
    if (st == RP_OK) st = dev_alloc(c, &B.phi, P * n_proj * dm.R);
    if (st == RP_OK) st = dev_alloc(c, &sgn, (size_t)F * n_proj);
    if (st == RP_OK) st = dev_alloc(c, &rep, P);
    const bool greedy_smem = 2 * sizeof(i64) * P <= GREEDY_SMEM;
    if (st == RP_OK && !greedy_smem) st = dev_alloc(c, &mind, P);
    if (st == RP_OK && !greedy_smem) st = dev_alloc(c, &pen, P);
    const size_t smem = sizeof(i64) * (size_t)n_proj * dm.R + sizeof(int) * ((size_t)3 * dm.K + 3 * dm.R + dm.G + 2) + 16;
    if (st == RP_OK && smem > 200 * 1024) st = RP_ERR_RANGE;
    cudaError_t e = cudaSuccess;
    if (st == RP_OK) {
        if (smem > 32 * 1024) e = cudaFuncSetAttribute(k_sel_prepare, cudaFuncAttributeMaxDynamicSharedMemorySize, RP_SMEM_LIMIT);
        if (e == cudaSuccess) {
            k_sel_signs<<<(F * n_proj + 255) / 256, 256, 0, c->stream>>>(F, n_proj, (u32)c->cfg.seed, (u32)(c->cfg.seed >> 32), sgn);
            k_sel_prepare<<<(int)P, SEL_THREADS, smem, c->stream>>>(dm, c->bl, c->buf[c->cur].blob, c->d_anc, c->d_W, c->d_wloc,
                                                                    (const unsigned short *)(c->d_static + c->sl.off_g), sgn, n_proj, B);
            k_sel_map<<<(int)P, SEL_THREADS, 0, c->stream>>>(dm.N, (int)P, B.canon, B.hash, score, rep);
            e = cudaMemsetAsync(dist, 0, sizeof(i64) * P * P, c->stream);
        }
        if (e == cudaSuccess) {
            // Tables of three CTAs per SM; larger ones are worked through in blocks.  (Prepare's limit keeps K below 18 k, so
            // that a block has at least one group.)
            const size_t rtab = std::min<size_t>(sizeof(int) * (size_t)dm.R * dm.R, std::max<size_t>(8 * 1024, sizeof(int) * (size_t)dm.R));
            const size_t ctab = std::min<size_t>(sizeof(int) * (size_t)dm.K * dm.K, std::max<size_t>((72 * 1024 - rtab) / 4 * 4, sizeof(int) * (size_t)dm.K));
            const void *fn = dm.N <= 65535 ? (const void *)k_sel_dist<u32> : (const void *)k_sel_dist<u64>;
            if (ctab + rtab > 32 * 1024) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, RP_SMEM_LIMIT);
            if (e == cudaSuccess) {
                const size_t items = P * ((P + SEL_CHUNK - 1) / SEL_CHUNK);
                const int grid = (int)std::min<size_t>(items, (size_t)148 * 3);
                if (dm.N <= 65535) k_sel_dist<u32><<<grid, SEL_THREADS, ctab + rtab, c->stream>>>(dm, (int)P, n_proj, rep, B, dist, (int)ctab, (int)rtab);
                else k_sel_dist<u64><<<grid, SEL_THREADS, ctab + rtab, c->stream>>>(dm, (int)P, n_proj, rep, B, dist, (int)ctab, (int)rtab);
            }
            const int tri = greedy_smem && sizeof(u32) * greedy_tri(P) <= GREEDY_DIST_MAX;
            const int gt = tri ? GREEDY_THREADS : (int)std::min<size_t>(GREEDY_THREADS, (P + 31) / 32 * 32);
            const size_t gm = greedy_smem ? 2 * sizeof(i64) * P + (tri ? sizeof(u32) * greedy_tri(P) + 16 : 0) : 0;        // (one pair at least)
            if (e == cudaSuccess && gm > 32 * 1024) e = cudaFuncSetAttribute(k_sel_greedy, cudaFuncAttributeMaxDynamicSharedMemorySize, RP_SMEM_LIMIT);
            if (e == cudaSuccess)
                k_sel_greedy<<<1, gt, gm, c->stream>>>((int)P, rep, score, dist, eta_q16, mind, pen, order, n_distinct, tri);
            k_sel_fill<<<(int)P, 256, 0, c->stream>>>(dm.N, order, lay, out);
            g_rp_launches += 6;
            e = cudaGetLastError();
        }
    }
    dev_free(c, B.canon); dev_free(c, B.hash); dev_free(c, B.clist); dev_free(c, B.cstart); dev_free(c, B.rlist);
    dev_free(c, B.rstart); dev_free(c, B.pc); dev_free(c, B.pr); dev_free(c, B.phi); dev_free(c, sgn); dev_free(c, rep);
    dev_free(c, mind); dev_free(c, pen); dev_free(c, B.lab); dev_free(c, B.big);
    if (e != cudaSuccess) return rp_fail(e);
    return st;
}
