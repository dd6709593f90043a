// The product kernel on 128 x 128 tiles, one CTA each: 5 stages of 32 KiB.
#include "gemm_tc_kernel.cuh"

namespace svt {

cudaError_t tc_launch_128(const TcLaunch &l, bool chain, int total_tiles, int num_sms, cudaStream_t s)
{
    return chain ? launch_kernel<128, 5, true, false>(l, total_tiles, num_sms, s)
                 : launch_kernel<128, 5, false, false>(l, total_tiles, num_sms, s);
}

} // namespace svt
