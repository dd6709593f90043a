// Launches of the product kernel (gemm_tc_kernel.cuh) by tile-width code.
#include <algorithm>
#include <cstring>

#include "svt_internal.h"

namespace svt {

namespace {

cudaError_t launch_width(const TcLaunch &l, bool chain, int bn, int total_tiles, int num_sms,
                         cudaStream_t s)
{
    if (bn == kBn64)
        return tc_launch_64(l, chain, total_tiles, num_sms, s);
    if (bn == 256)
        return tc_launch_256(l, chain, total_tiles, num_sms, s);
    if (bn == 128)
        return tc_launch_128(l, chain, total_tiles, num_sms, s);
    if (bn == kBnPair)
        return tc_launch_pair(l, chain, false, total_tiles, num_sms, s);
    if (bn == kBnPair128)
        return tc_launch_pair128(l, chain, total_tiles, num_sms, s);
    return cudaErrorInvalidValue;
}

} // namespace

cudaError_t tc_gemm_launch_fused(const TcLaunch &l, int bn, int total_tiles, int num_sms,
                                 cudaStream_t s, bool strips)
{
    TcLaunch g = l;
    g.nprob = 0;
    if (strips)  // per-strip dependencies
        return bn == kBnPair ? tc_launch_pair(g, true, true, total_tiles, num_sms, s)
                             : cudaErrorInvalidValue;
    return launch_width(g, true, bn, total_tiles, num_sms, s);
}

cudaError_t tc_gemm_load_fused(int bn, int num_sms)
{
    TcLaunch none;
    std::memset(&none, 0, sizeof(none));
    return launch_width(none, true, bn, 0, num_sms, nullptr);
}

int tc_num_tiles(const TcProblem &p, int bn)
{
    return p.sym ? sym_tiles(bn, p.tiles_n) : p.tiles_m * p.tiles_n;
}

int tc_valid_ctas(const TcProblem &p, int bn)
{
    int n = 0;
    if (!p.sym)
        n = p.tiles_m * p.tiles_n;
    else
        for (int tn = 0; tn < p.tiles_n; ++tn)
            n += std::min(sym_rows(bn, tn), p.tiles_m);
    return n * ctas_per_tile(bn);
}

cudaError_t tc_gemm_launch(const TcLaunch &l, int bn, int num_sms, cudaStream_t s)
{
    if (l.gtab)
        return cudaErrorInvalidValue;
    return launch_width(l, false, bn, l.tile_start[l.nprob], num_sms, s);
}

} // namespace svt
