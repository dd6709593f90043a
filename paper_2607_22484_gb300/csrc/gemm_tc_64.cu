// The product kernel on 128 x 64 tiles, one CTA each: 6 stages of 24 KiB.
#include "gemm_tc_kernel.cuh"

namespace svt {

cudaError_t tc_launch_64(const TcLaunch &l, bool chain, int total_tiles, int num_sms, cudaStream_t s)
{
    return chain ? launch_kernel<64, 6, true, false>(l, total_tiles, num_sms, s)
                 : launch_kernel<64, 6, false, false>(l, total_tiles, num_sms, s);
}

} // namespace svt
