// sn_selftest.cu — the bounded-wait rule exercised on purpose, so that failure
// detection can be tested on a GPU without a fault.
//
// sn_selftest_wait_timeout:
// One CTA of two warps sets up like the pipeline kernels (an mbarrier, an abort
// flag, 32 columns of tensor memory), then both warps wait for a phase of the
// barrier that no thread and no copy ever completes, with the same bounded wait
// (tc::warp_wait).  The first to pass the wait limit raises the CTA's abort
// flag and records SN_EBIT_TIMEOUT in the basis' error word; the other stops on
// the flag.  The CTA then frees its tensor memory and returns, leaving the
// context usable.
//
// sn_selftest_barrier_timeout: one CTA waits in the grid barrier of the cooperative kernels
// for twice the arrivals that its grid makes, and gives up at the limit; its next wait
// ends at once on the flag that the first one left.
#include "sn_tc.cuh"

namespace {

__global__ void __launch_bounds__(64, 1) k_wait_timeout(unsigned int *err)
{
    using namespace sn::tc;
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    const int warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bar), 1);     // one arrival expected, none is ever made
        abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 0)
        tmem_alloc(smem_u32(&tmem_slot), 32);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    warp_wait(smem_u32(&bar), 0, &abort_flag, err);    // phase 0 never completes

    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, 32);
    }
}

__global__ void __launch_bounds__(64, 1) k_barrier_timeout(unsigned int *err)
{
    __shared__ unsigned int bar[2];       // the arrivals and the flag of one CTA alone
    if (threadIdx.x < 2)
        bar[threadIdx.x] = 0;
    sn::tc::grid_barrier(bar, 2, err);    // one arrival is made
    sn::tc::grid_barrier(bar, 3, err);
}

sn_status selftest(sn_basis_t b, void (*kernel)(unsigned int *), cudaStream_t stream)
{
    if (!b)
        return SN_ERR_INVALID_ARG;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev != b->device)
        return SN_ERR_INVALID_ARG;
    kernel<<<1, 64, 0, stream>>>(b->err);
    sn::count_launch();
    return cudaGetLastError() == cudaSuccess ? SN_OK : SN_ERR_CUDA;
}

}  // namespace

extern "C" sn_status sn_selftest_wait_timeout(sn_basis_t b, sn_stream_t stream)
{
    return selftest(b, k_wait_timeout, (cudaStream_t)stream);
}

extern "C" sn_status sn_selftest_barrier_timeout(sn_basis_t b, sn_stream_t stream)
{
    return selftest(b, k_barrier_timeout, (cudaStream_t)stream);
}
