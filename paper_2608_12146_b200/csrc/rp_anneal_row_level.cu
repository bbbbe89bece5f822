// One launch per level (rank loads as slices), a warp a chain.
#include "rp_anneal_row_chain.cuh"

template <bool IDENT>
static int launch(rp_ctx *c, const AnnealArgs &A, const RowArgs &X, int l, int k, int grid)
{
    int done;
#define ROW_CASE(L_, K_, C_) if (l == L_ && k == K_ && X.comp == C_) return launch_row_t<32, L_, K_, false, C_, IDENT>(c, A, X, grid, &done)
    ROW_CASE(1, 1, 1); ROW_CASE(2, 1, 1); ROW_CASE(4, 1, 1);
    ROW_CASE(1, 1, 0); ROW_CASE(1, 2, 0); ROW_CASE(1, 4, 0); ROW_CASE(2, 1, 0); ROW_CASE(2, 2, 0); ROW_CASE(4, 1, 0);
#undef ROW_CASE
    return RP_ERR_STATE;
}

int rp_launch_row_level(rp_ctx *c, const AnnealArgs &A, const RowArgs &X, int l, int k, int grid)
{
    return c->dm.own_shard ? launch<true>(c, A, X, l, k, grid) : launch<false>(c, A, X, l, k, grid);
}
