// One launch per level (rank loads as slices), a warp a chain.
#include "rp_anneal_row_chain.cuh"

template <bool IDENT>
static int launch(rp_ctx *c, const AnnealArgs &A, const RowArgs &X)
{
    const int l = rp_row_layers(c->dm), n = (c->dm.L * X.cpl + 31) / 32;
    int done;
#define ROW_CASE(WHEN, L_, K_, SPLIT_, COMP_) if (WHEN) return launch_row_t<32, L_, K_, SPLIT_, false, COMP_, IDENT>(c, A, X, c->Ppop, &done)
    if (X.comp) { ROW_CASE(l == 1, 1, 1, false, true); ROW_CASE(l == 2, 2, 1, false, true); ROW_CASE(l == 4, 4, 1, false, true); }
    else if (rp_row_split(X.cpl)) {
        ROW_CASE(n <= 1, 1, 1, true, false); ROW_CASE(n <= 2, 1, 2, true, false); ROW_CASE(n <= 3, 1, 3, true, false); ROW_CASE(n <= 4, 1, 4, true, false);
    } else {
        ROW_CASE(l == 1 && X.cpl == 1, 1, 1, false, false); ROW_CASE(l == 2 && X.cpl == 1, 2, 1, false, false);
        ROW_CASE(l == 4 && X.cpl == 1, 4, 1, false, false); ROW_CASE(l == 1 && X.cpl == 3, 1, 3, false, false);
    }
#undef ROW_CASE
    return RP_ERR_STATE;
}

int rp_launch_row_level(rp_ctx *c, const AnnealArgs &A, const RowArgs &X)
{
    return c->dm.own_shard ? launch<true>(c, A, X) : launch<false>(c, A, X);
}

// (asked for compressed rows of up to 32 layers where slot d is shard d)
int rp_row_level_resident(const rp_ctx *, const RowArgs &X, int *warps)
{
    return row_resident_t<32, 1, 1, false, true, true>(X, warps);
}
