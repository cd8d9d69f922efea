// whg_kernels_wide6.cu -- the step kernel for small ensembles, 6-term Stumpff series.
#include "whg_wide.cuh"

cudaError_t whg_launch_step_wide_nt6(const WhgState& st, const WhgBuckets& bk, long long n, int gr_mode,
                                     const WhgLaunch& l)
{
    const long long threads = (long long)whg_wide_warps(bk) * 32;
    const int grid = (int)((threads + l.block - 1) / l.block);
    if (gr_mode == 0)
        whg::k_step_wide<6, 0><<<grid, l.block, 0, l.stream>>>(st, bk, n);
    else if (gr_mode == 1)
        whg::k_step_wide<6, 1><<<grid, l.block, 0, l.stream>>>(st, bk, n);
    else
        whg::k_step_wide<6, 2><<<grid, l.block, 0, l.stream>>>(st, bk, n);
    return cudaGetLastError();
}
