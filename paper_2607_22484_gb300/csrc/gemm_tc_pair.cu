// The product kernel on 256 x 256 tiles, a pair of CTAs each: 5 stages of 32 KiB per CTA.
#include "gemm_tc_kernel.cuh"

namespace svt {

cudaError_t tc_launch_pair(const TcLaunch &l, bool chain, bool strips, int total_tiles, int num_sms,
                           cudaStream_t s)
{
    if (strips)
        return launch_kernel<256, 5, true, true, true>(l, total_tiles, num_sms, s);
    return chain ? launch_kernel<256, 5, true, true>(l, total_tiles, num_sms, s)
                 : launch_kernel<256, 5, false, true>(l, total_tiles, num_sms, s);
}

} // namespace svt
