// One launch for all levels (rank loads on chip).
#include "rp_anneal_row_chain.cuh"

template <bool IDENT>
static int launch(rp_ctx *c, const AnnealArgs &A, const RowArgs &X, int grid, int *done)
{
    const int l = rp_row_layers(c->dm), k = X.cpl <= 4 ? X.cpl : 8;
#define ROW_CASE(L_, K_) if (l == L_ && k == K_) return launch_row_t<32, L_, K_, false, true, false, IDENT>(c, A, X, grid, done)
    ROW_CASE(1, 1); ROW_CASE(1, 2); ROW_CASE(1, 3); ROW_CASE(1, 4); ROW_CASE(1, 8);
    ROW_CASE(2, 1); ROW_CASE(2, 2); ROW_CASE(2, 3); ROW_CASE(2, 4);
    ROW_CASE(4, 1); ROW_CASE(4, 2);
#undef ROW_CASE
    return RP_ERR_STATE;
}

int rp_launch_row_chip(rp_ctx *c, const AnnealArgs &A, const RowArgs &X, int grid, int *done)
{
    return c->dm.own_shard ? launch<true>(c, A, X, grid, done) : launch<false>(c, A, X, grid, done);
}
