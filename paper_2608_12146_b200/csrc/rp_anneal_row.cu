// Chain kernel of the population annealing for windows whose rank-load rows are short enough to be
// scored from registers: a warp per chain (or half a warp), one layer per lane.
//
// A chain of Algorithm 3 is a sequence of dependent rounds; what bounds a level is the latency of a
// round times the rounds of a chain, over the chains an SM keeps in flight.  The kernel shortens and
// removes rounds:
//  * Rejections without rank loads.  For any rank p of a layer, max_p (W + d) >= W[p] + d[p].  With one
//    fixed rank per layer (the busiest of the window as a whole) and f_i = sum_l q[i][l][p_l], the new
//    expert cost of the row-shard that gives sample i and takes i2 is at least F - f_i + f_i2, F the sum of
//    f over its samples (kept as the slack Esum - F).  Score and energy are monotone in it, so the lane that proposes a step can
//    reject it by itself from cell statistics, F and two scalars: 32 steps at a time (16 where two chains share a warp), no rank load read.
//    Windows whose samples follow one routing mix have the same busiest rank nearly everywhere, and
//    then every rejection is decided this way and what is scored is accepted (large, wide, heavy, medium of
//    the named windows: all but 1e-4 of the rejections); with four routing mixes an eighth to a third
//    is.  A candidate that is not rejected by its bound is scored exactly.  The bound is worked out in single precision with an
//    allowance for its roundings: in 64-bit integers it was a third of a round's instructions (with the decision shared by two
//    lanes, heavy 1.10 times as fast, wide 1.02, medium 1.04).
//  * Rows in registers.  A lane holds whole layers (layer = lane, lane + 32, ...) of the two slices and the two
//    demand rows, or, one launch per level with rows of two or four chunks a layer, the chunks are dealt out to the lanes in turn and
//    a layer's maximum meets in shuffles: 16-byte loads, one trip, no staging; the new slices are stored from the
//    same registers.
//  * Compressed rows (COMP: rank counts of 8 and more whose full rows do not fit the registers).  A row keeps, per
//    layer, the loads of the three ranks that are busiest in the window and an upper bound of every
//    other rank's load: the sum over the samples of each one's largest count among those ranks.
//    While the bound does not exceed the three, their maximum is the layer's maximum; where it
//    does, the layer's loads are added up from the samples of the row-shard.  Used when the seed's
//    row-shards nearly all satisfy it (checked on the device, see k_member_rows): 16 bytes per layer
//    instead of 4*P: an eighth of the traffic at 32 ranks.
//  * Two chains to a warp (sixteen lanes each, see row_pairs) where there are more members than a warp each keeps resident.
//  * No staging area, so 12 or 16 warps per SM instead of 5 to 10.
// What bounds it now: the latency of a round, about 2200 cycles alone on an SM (medium), 3300 with 7 warps (large), 3800 with 11 (wide)
// and 5900 for two chains with 16 (heavy), where the warps' instructions share the issue slots; launched once for all levels the
// slowest chain of a level takes twice the mean, three quarters of the level's time.  A level's time with the warp-per-chain kernel
// (medium: warp per candidate) and now: heavy 15.0 -> 2.7 ms, wide 1.2 -> 0.40 ms, large 0.21 -> 0.10 ms, medium 50 -> 29 us.
// Step for step this is the sequential chain: proposals are evaluated against the current state,
// feasible ones are decided in step order, and the speculation is redone after an acceptance.
//
// Two forms.  CHIP: the rank loads of a chain live in shared memory, every chain is resident at once
// and one launch runs all levels; a CTA holds several chains and works out the level barrier
// for itself.  Otherwise one launch per level, rank loads as slices of a pool shared copy-on-write (see AnnealArgs).
#include <algorithm>
#include <string.h>

#include "rp_anneal_row.cuh"

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

// Member m = blockIdx.x, row-shard rg = blockIdx.y: the slack (sum of the busiest loads less the samples' f), and the row-shard's
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
        if (__ldg(rg_of + cells[i]) == rg) { f += __ldg(&tf[i].y); list[atomicAdd(&n_s, 1)] = i; }
    if (f) atomicAdd(&f_s, (u64)f);
    __syncthreads();
    if (tid == 0) {
        const i64 es = ((const i64 *)(blob + bl.off_Esum))[rg], slack = es - (i64)f_s;
        Fo[(size_t)m * dm.RG + rg] = slack;
        if (loose && slack * 16 > es) atomicAdd(undecided, 1);
    }
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

// The slacks alone, one CTA per member: one scan of the assignment (a CTA per row-shard scans it once for each: 256 members of 2048
// samples in 240 row-shards 134 us, 5.4 here).  Sums in shared memory by the lower and upper 16 bits of each f apart (below 65536
// samples neither passes 32 bits): a 64-bit addition there is a loop, and where many samples of a row-shard meet it took 180 us for 8192
// samples in four row-shards, 10 here, and 24 in a CTA per row-shard.
__global__ void __launch_bounds__(256)
k_member_slack(RpDims dm, RpBlob bl, const char *__restrict__ blobs, const char *__restrict__ static_blk, RpStatic sl, const int2 *__restrict__ tf,
               i64 *__restrict__ Fo, int *__restrict__ undecided, int loose)
{
    extern __shared__ uint2 sum[];                      // [RG]
    const int m = blockIdx.x, tid = threadIdx.x;
    const char *blob = blobs + (size_t)m * bl.bytes;
    const unsigned short *cells = (const unsigned short *)(blob + bl.off_cell);
    const unsigned short *rg_of = (const unsigned short *)(static_blk + sl.off_rg);
    for (int rg = tid; rg < dm.RG; rg += 256) sum[rg] = make_uint2(0, 0);
    __syncthreads();
#pragma unroll 8
    for (int i = tid; i < dm.N; i += 256) {
        uint2 *s = sum + __ldg(rg_of + cells[i]);
        const u32 f = (u32)__ldg(&tf[i].y);
        atomicAdd(&s->x, f & 0xffffu);
        if (f >> 16) atomicAdd(&s->y, f >> 16);
    }
    __syncthreads();
    int n = 0;
    for (int rg = tid; rg < dm.RG; rg += 256) {
        const uint2 s = sum[rg];
        const i64 es = ((const i64 *)(blob + bl.off_Esum))[rg], slack = es - ((i64)s.x + ((i64)s.y << 16));
        Fo[(size_t)m * dm.RG + rg] = slack;
        n += loose && slack * 16 > es;
    }
    if (n) atomicAdd(undecided, n);
}

// ---------------------------------------------------------------------------------------------
// Which windows, which form.
// ---------------------------------------------------------------------------------------------
static int chunks_of(int cpl) { return cpl <= 1 ? 1 : (cpl <= 2 ? 2 : (cpl <= 4 ? 4 : (cpl <= 8 ? 8 : 0))); }

// Chunks a lane that takes whole layers would hold per row, rounded up to powers of two; 0 = too many.
static int row_chunks(const RpDims &dm, int cpl)
{
    const int l = rp_row_layers(dm), c = chunks_of(cpl);
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
    // records that members hand on: as many bytes as the blob's arrays before the assignment
    X.off_E = 16 * dm.RG; X.off_Q = X.off_E + 8 * dm.RG; X.off_TC = X.off_Q + 8 * dm.K; X.off_U = X.off_TC + 8 * dm.K;
    X.off_S = X.off_U + 8 * dm.G; X.cs_bytes = X.off_S + 8 * 4;
    size_t c = ((size_t)X.cs_bytes + 15) & ~(size_t)15;
    X.off_top = (int)c;   c += dm.own_shard ? 0 : (size_t)8 * dm.K + (size_t)18 * dm.RG * dm.S;
    c = (c + 7) & ~(size_t)7;
    X.off_F = (int)c;     c += (size_t)8 * dm.RG;
    X.off_mbar = (int)c;  c += 8;
    X.off_ws = (int)c;    c += chip ? 0 : (size_t)8 * dm.RG;
    c = (c + 15) & ~(size_t)15;
    const size_t lay = (2 * (size_t)dm.N + 15) & ~(size_t)15;
    X.off_cell = (int)c;  c += chip ? lay : 0;
    X.off_snap = (int)c;  c += chip ? lay : 0;
    // (records of 256 steps at most, twice)
    X.recs = chip && cw < ROW_THREADS / 32 ? std::min(steps, 256) : (!chip && cw == 2 ? 16 : 0);       // (two chains a warp: 32 steps, once)
    X.off_recs = (int)c;  c += (size_t)2 * X.recs * sizeof(StepRec);
    c = (c + 15) & ~(size_t)15;
    X.off_list = (int)c;  c += X.comp ? (size_t)4 * (ROW_LIST + 1) : 0;
    X.off_W = (int)c;     c += chip ? (size_t)4 * dm.RG * X.rlp : 0;
    X.chain_bytes = (int)((c + 15) & ~(size_t)15);
    X.smem_bytes = X.off_chain + X.chain_bytes * cw;
    X.cw = cw;
    X.off_tf = 0;
}

// Full rows (padded to whole chunks).
static void full_rows(const RpDims &dm, RowArgs &X)
{
    X.cpl = (dm.P + 3) / 4; X.rlp = dm.L * X.cpl * 4; X.comp = 0;
}

// One launch for all levels, the chains' rank loads on chip: at most eight chunks per lane, every chain resident at once.
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
    if (dm.P >= 8 && dm.P <= 128 && rp_row_layers(dm)) return 2;      // (128: ranks the placement kernel orders)
    return 0;
}

// Whether the form that launches once per level is taken by the shared memory of a chain (a warp to itself).  Where DP slot d is
// shard d, as far as it fits: it is the fastest kernel even with one chain per SM (L = 24, P = 16, 1024 members, three levels of
// 200 steps: 63 KB 3.4 ms and 4.2 for the next best kernel, 93 KB 4.0 and 5.4, 118 KB 8.4 and 23).  Else the attention of a shard's slots
// is looked up (8*K + 18*R*G*S bytes more, S stages a move) and a chain's rounds are longer: with up to two stages where an SM holds two
// chains, with more where it holds three.  The same search with shards of two slots, below the line and beyond it: two stages 61 KB
// 4.0 and 4.9, 109 KB 5.9 and 19, beyond 130 KB 11.8 and 24; four stages 43 KB 1.3 and 2.2, 66 KB 3.0 and 3.4, beyond 86 KB 6.6 and 5.8,
// 107 KB 6.7 and 7.8; eight stages 54 KB 1.5 and 2.8, beyond 79 KB 2.64 and 2.68, 108 KB 7.7 and 7.2.  (The line was drawn by an
// earlier form of the kernel, which fell behind there; today's is about even for some way beyond.)
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
    if (!c->undecided_clear) RP_CUDA(cudaMemsetAsync(c->d_undecided, 0, sizeof(int), c->stream));
    c->undecided_clear = 0;
    i64 *Fo = c->d_rowF + (size_t)c->cur * c->Ppop * dm.RG;
    if (!sep)                       // (a chain keeps 40 bytes of a row-shard in shared memory: no more than 5632)
        k_member_slack<<<n, 256, sizeof(uint2) * (size_t)dm.RG, c->stream>>>(dm, c->bl, c->buf[c->cur].blob, c->d_static, c->sl, (const int2 *)c->d_tf, Fo,
                                                                          c->d_undecided, c->row_check);
    else
        k_member_rows<<<dim3(n, dm.RG), 256, smem, c->stream>>>(dm, c->bl, c->buf[c->cur].blob, c->d_static, c->sl, (const int2 *)c->d_tf, X.qr, X.rlp,
                                                                X.comp, Fo, c->d_Wr, c->d_wloc, c->d_undecided, c->row_check);
    ++g_rp_launches;
    RP_CUDA(cudaGetLastError());
    c->row_counted = n;
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
    // lengths and fixed-rank demands of the samples too, if there is room (an L2 trip for every 32 steps)
    if (X.smem_bytes + 8 * c->dm.N <= ROW_SMEM_MAX) { X.off_tf = X.smem_bytes; X.smem_bytes += 8 * c->dm.N; }
    A.w_on_chip = 1;
    A.slices = c->dm.slices;
    A.smem_bytes = (unsigned)X.smem_bytes;
    A.lo.cand_layout = c->d_cand_layout;
    RP_TRY(rp_launch_row_chip(c, A, X, (c->Ppop + cw - 1) / cw, done));
    if (*done) c->row_form = 1;
    return RP_OK;
}

// Whether two chains share a warp: compressed rows of up to 32 layers where slot d is shard d, if there are more members than chains
// resident with a warp each, and an SM keeps at least half as many again when they share.  A round takes longer then (heavy
// 5900 cycles for two, 4300 for one) and half the warps do it.  How many warps are resident is asked for: 16 by the registers of
// today's instances (128 a thread), fewer by the shared memory of windows with many row-shards.  20 levels of 100 steps, one chain to
// a warp and two, in ms, with 2368 (16 on each of 148 SMs), 2400 and 3000 members: 16 layers of 32 ranks, 4000 samples 2.77 and 2.82,
// 3.18 and 2.87, 3.60 and 2.97; 32 layers, 1000 samples 1.90 and 2.16, 2.04 and 2.18, 2.35 and 2.27; heavy 4.23 and 4.47, 5.31 and
// 4.66, (3500) 6.46 and 5.21.  (14 were counted before, so that 2073 to 2368 members shared warps: 2200 members of the second 1.87
// ms, 2.15.)  Of 48 layers a lane would have three, and wide's 288 row-shards leave shared memory for six warps: 8.5 and 12.7 ms.
static int row_pairs(const rp_ctx *c, const RowArgs &X0, bool *pair)
{
    *pair = false;
    if (!X0.comp || !c->dm.own_shard || c->dm.L > 32) return RP_OK;
    RowArgs X = X0;
    int one = 0, two = 0;
    chain_layout(c->dm, c->bl, c->sl, X, false, 1, c->Ppop, 0);
    RP_TRY(rp_row_level_resident(c, X, &one));
    if (c->Ppop <= one * rp_sms(c)) return RP_OK;
    chain_layout(c->dm, c->bl, c->sl, X, false, 2, c->Ppop, 0);
    if (X.smem_bytes > ROW_SMEM_MAX) return RP_OK;         // (what a launch may ask for is a little less than an SM has)
    RP_TRY(rp_row_pair_resident(c, X, &two));
    *pair = 2 * 2 * two >= 3 * one;
    return RP_OK;
}

int rp_launch_level_end(rp_ctx *c, const AnnealArgs &A);
int rp_launch_level_turn(rp_ctx *c, const AnnealArgs &A);

int rp_launch_anneal_row(rp_ctx *c, AnnealArgs &A)
{
    RowArgs X;
    row_args(c, X);
    if (A.level == 0) RP_TRY(row_pairs(c, X, &c->row_pair));
    const bool pair = c->row_pair;
    chain_layout(c->dm, c->bl, c->sl, X, false, pair ? 2 : 1, c->Ppop, 0);
    if (X.smem_bytes > ROW_SMEM_MAX) return RP_ERR_RANGE;
    A.smem_bytes = (unsigned)X.smem_bytes;
    A.slices = 1;
    A.lo.cand_layout = nullptr;
    RP_TRY(pair ? rp_launch_row_pair(c, A, X) : rp_launch_row_level(c, A, X));
    c->row_form = pair ? 5 : X.comp ? 4 : rp_row_split(X.cpl) ? 3 : 2;
    if (!A.last && rp_row_turns(c)) return rp_launch_level_turn(c, A);
    return rp_launch_level_end(c, A);
}
