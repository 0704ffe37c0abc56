// What a plan's host side does when a bounded device-side wait ran out.
#pragma once

#include <cuda_runtime.h>

#include <stddef.h>

namespace epic {

// The CUDA runtime's calls on the default stream; tests use stand-ins.
struct CudaRt {
    cudaError_t read(int* host, const int* dev) { return cudaMemcpy(host, dev, sizeof(int), cudaMemcpyDeviceToHost); }
    cudaError_t zero(int* dev, size_t n) { return cudaMemset(dev, 0, n * sizeof(int)); }
    cudaError_t wait() { return cudaStreamSynchronize(nullptr); }
};

// Reads the bounded-wait flag of finished calls.  Set: clears it, and the counts of the parts of split work items,
// which only the block that stores an item's last part brings back to zero -- left standing by blocks whose
// partner gave up, they would make the next launch add parts that are not stored yet.  All of it is in
// before the return: later calls' streams need not wait for the default one.
template <class Rt>
cudaError_t take_wait_flag(Rt&& rt, int* status, int* counters, size_t n_counters, int* flag)
{
    *flag = 0;
    if (!status) return cudaSuccess;
    cudaError_t e = rt.read(flag, status);
    if (e != cudaSuccess || !*flag) return e;
    e = rt.zero(status, 1);
    if (e == cudaSuccess && counters) e = rt.zero(counters, n_counters);
    if (e == cudaSuccess) e = rt.wait();
    return e;
}

}  // namespace epic
