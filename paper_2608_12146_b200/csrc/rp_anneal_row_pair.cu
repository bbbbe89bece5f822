// One launch per level (compressed rows as slices), two chains to a warp, sixteen lanes each: the instructions of a round are issued
// once for both.
#include "rp_anneal_row_chain.cuh"

int rp_launch_row_pair(rp_ctx *c, const AnnealArgs &A, const RowArgs &X)
{
    const int grid = (c->Ppop + 1) / 2;
    int done;
    if (c->dm.L <= 16) return launch_row_t<16, 1, 1, false, false, true, true>(c, A, X, grid, &done);
    if (c->dm.L <= 32) return launch_row_t<16, 2, 1, false, false, true, true>(c, A, X, grid, &done);
    return RP_ERR_STATE;
}

int rp_row_pair_resident(const rp_ctx *c, const RowArgs &X, int *warps)
{
    return c->dm.L <= 16 ? row_resident_t<16, 1, 1, false, true, true>(X, warps) : row_resident_t<16, 2, 1, false, true, true>(X, warps);
}
