// whg_kernels_few8.cu -- the step kernel for few warps per SM, 8-term Stumpff series.
#include "whg_device.cuh"

cudaError_t whg_launch_step_few_nt8(const WhgState& st, const WhgBuckets& bk, long long n, int gr_mode,
                                    const WhgLaunch& l)
{
    if (gr_mode == 0)
        whg::k_step<8, 0, 1><<<l.grid, l.block, 0, l.stream>>>(st, bk, n);
    else if (gr_mode == 1)
        whg::k_step<8, 1, 1><<<l.grid, l.block, 0, l.stream>>>(st, bk, n);
    else
        whg::k_step<8, 2, 1><<<l.grid, l.block, 0, l.stream>>>(st, bk, n);
    return cudaGetLastError();
}
