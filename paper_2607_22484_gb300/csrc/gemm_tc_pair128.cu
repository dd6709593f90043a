// The product kernel on 256 x 128 tiles, a pair of CTAs each: 6 stages of 24 KiB per CTA.
#include "gemm_tc_kernel.cuh"

namespace svt {

cudaError_t tc_launch_pair128(const TcLaunch &l, bool chain, int total_tiles, int num_sms, cudaStream_t s)
{
    return chain ? launch_kernel<128, 6, true, true>(l, total_tiles, num_sms, s)
                 : launch_kernel<128, 6, false, true>(l, total_tiles, num_sms, s);
}

} // namespace svt
