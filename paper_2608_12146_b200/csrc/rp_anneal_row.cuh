// What the one-layer-per-lane chain kernel is given beside AnnealArgs (rp_anneal_row.cu).
#pragma once
#include "rp_anneal.cuh"

#define ROW_MAX_WARPS 8          // chains of a CTA in the launch that runs all levels, at most
#define ROW_THREADS 256          // its threads
#define ROW_SMEM_MAX (220 * 1024)
#define ROW_LIST 256             // samples of a row-shard collected at a time where its loads are added up anew

struct RowArgs {
    const int *qr;               // [N][rlp] demand rows: cpl 16-byte chunks per layer
    const int2 *tf;              // [N] length, and the demand on the layers' fixed ranks summed over the layers
    int *Wr;                     // rank-load slices in the same form
    const i64 *F_src;            // [P_pop][RG] slack of a row-shard: sum of its busiest loads less sum of its samples' tf.y; the level's start, its end, both buffers
    i64 *F_dst, *F_buf;
    int rlp, cpl, comp;
    int off_tab, off_leF, off_chain, off_tf;                                       // shared memory of the CTA
    int off_E, off_Q, off_TC, off_U, off_S, cs_bytes;                      // of one chain: records handed on from level to level,
    int off_F, off_mbar, off_ws, off_top, off_cell, off_snap, off_recs, off_list, off_W;   // the rest
    int chain_bytes, smem_bytes, cw, recs;
};

__device__ __forceinline__ int4 sub4(const int4 &a, const int4 &b) { return make_int4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w); }
__device__ __forceinline__ int4 add4(const int4 &a, const int4 &b) { return make_int4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }

// The chains of a level may be launched before the launch between two levels (rp_level_turn.cu) has ended: once each of its CTAs has called
// rp_let_next_launch_start or has ended.  What it leaves behind, or reads still, they touch behind rp_wait_for_launch_before, which
// waits for its end.

// Bounded wait of one thread until a counter that the other CTAs of the launch add to has reached
// `target`; false when the time allowed ran out or another chain has raised the time-out word.
__device__ __forceinline__ bool rp_wait_count(const int *ctr, int target, const AnnealArgs &A)
{
    u64 t0;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    for (unsigned it = 0;; ++it) {
        int v;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
        if (v >= target) return true;
        if ((it & 15u) == 15u) {
            if (__ldcg(&A.status[RP_SW_TIMEOUT])) return false;
            u64 t1;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
            if (t1 - t0 > A.bar_timeout_ns) return false;
        }
    }
}

// Layers per lane where a lane takes whole layers (0: too many layers); whether a row's chunks are dealt out to the lanes instead.
static inline int rp_row_layers(const RpDims &dm) { return dm.L <= 32 ? 1 : (dm.L <= 64 ? 2 : (dm.L <= 128 ? 4 : 0)); }
static inline bool rp_row_split(int cpl) { return cpl == 2 || cpl == 4; }
// Whether they may start right away, up to four to an SM: their first step records and tables are then ready when the launch before ends
// (300 members of 17 layers 1469 us at its end, 1401 right away; 512 of 24 2730 and 2715).  With more, the SM is full and what its
// rows have left of the L1 cache counts (1024 members 2377 and 2390).  Only where there is a launch between two levels to start beside.
static inline bool rp_row_starts_early(const rp_ctx *c) { return rp_row_turns(c) && c->Ppop <= 4 * rp_sms(c); }
int rp_launch_row_chip(rp_ctx *c, const AnnealArgs &A, const RowArgs &X, int grid, int *done);
int rp_launch_row_level(rp_ctx *c, const AnnealArgs &A, const RowArgs &X);
int rp_launch_row_pair(rp_ctx *c, const AnnealArgs &A, const RowArgs &X);
// Warps of the instance that the launch would take which an SM keeps resident.
int rp_row_level_resident(const rp_ctx *c, const RowArgs &X, int *warps);
int rp_row_pair_resident(const rp_ctx *c, const RowArgs &X, int *warps);
