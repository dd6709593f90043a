// The product kernel on 128 x 256 tiles, one CTA each: 3 stages of 48 KiB.
#include "gemm_tc_kernel.cuh"

namespace svt {

cudaError_t tc_launch_256(const TcLaunch &l, bool chain, int total_tiles, int num_sms, cudaStream_t s)
{
    return chain ? launch_kernel<256, 3, true, false>(l, total_tiles, num_sms, s)
                 : launch_kernel<256, 3, false, false>(l, total_tiles, num_sms, s);
}

} // namespace svt
