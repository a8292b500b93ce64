// a5-a6 in float64 for tuples of 2-6 orbitals: the launches of the sector solver for the
// tuples that the mixed launch flagged.
#include "casci_sector64.cuh"

namespace mbe {

template <int N, int K>
static int launch_class(mbe_ctx *ctx, const BatchArgs &a, int b)
{
    using C = Cls<N, K>;
    const size_t smem = al16((int)sizeof(SectorTables<C>)) + sizeof(Sector64<C>) * a.warps;
    MBE_CU(allow_smem(k_sector64<C, true>, ctx->smem_optin));
    int per_sm = 0;
    MBE_CU(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sector64<C, true>, a.warps * 32, smem));
    if (per_sm < 1) per_sm = 1;
    k_sector64<C, true><<<sector_grid(ctx, a, per_sm), a.warps * 32, smem, ctx->stream>>>(a, b);
    MBE_CU(cudaGetLastError());
    ++ctx->launches;
    return MBE_OK;
}

// The classes of three orbitals: they last about as long, and one after the other cost small batches
// the latency of a solve (4 tuples of both 129 us, 107 by the list-driven kernel that took both).
static int launch_pair(mbe_ctx *ctx, const BatchArgs &a, int b)
{
    using C0 = Cls<3, 1>;
    using C1 = Cls<3, 2>;
    auto *kernel = k_sector64_pair<C0, C1, true>;
    const size_t smem = std::max(al16((int)sizeof(SectorTables<C0>)) + sizeof(Sector64<C0>) * a.warps,
                                 al16((int)sizeof(SectorTables<C1>)) + sizeof(Sector64<C1>) * a.warps);
    MBE_CU(allow_smem(kernel, ctx->smem_optin));
    int per_sm = 0;
    MBE_CU(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, a.warps * 32, smem));
    if (per_sm < 1) per_sm = 1;
    const int grid = std::min(2 * sector_grid(ctx, a, per_sm), ctx->sm_count * per_sm);
    kernel<<<grid, a.warps * 32, smem, ctx->stream>>>(a, b);
    MBE_CU(cudaGetLastError());
    ++ctx->launches;
    return MBE_OK;
}

int launch_sector64_redo(mbe_ctx *ctx, const BatchArgs &a, int b, int k)
{
    switch (a.n * 8 + k) {
    case 2 * 8 + 1: return launch_class<2, 1>(ctx, a, b);
    case 3 * 8 + 1: return launch_pair(ctx, a, b);  // (and k = 2)
    case 4 * 8 + 1: return launch_class<4, 1>(ctx, a, b);
    case 4 * 8 + 2: return launch_class<4, 2>(ctx, a, b);
    case 4 * 8 + 3: return launch_class<4, 3>(ctx, a, b);
    case 5 * 8 + 1: return launch_class<5, 1>(ctx, a, b);
    case 5 * 8 + 2: return launch_class<5, 2>(ctx, a, b);
    case 5 * 8 + 3: return launch_class<5, 3>(ctx, a, b);
    case 5 * 8 + 4: return launch_class<5, 4>(ctx, a, b);
    case 6 * 8 + 1: return launch_class<6, 1>(ctx, a, b);
    case 6 * 8 + 2: return launch_class<6, 2>(ctx, a, b);
    case 6 * 8 + 3: return launch_class<6, 3>(ctx, a, b);
    case 6 * 8 + 4: return launch_class<6, 4>(ctx, a, b);
    case 6 * 8 + 5: return launch_class<6, 5>(ctx, a, b);
    }
    set_error("casci_batch: no sector solver for the class (%d, %d)", a.n, k);
    return MBE_EUNSUPPORTED;
}

}  // namespace mbe
