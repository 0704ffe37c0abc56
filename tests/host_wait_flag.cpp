// Test driver for what follows a bounded wait that ran out (wait_flag.h), with a stand-in for the CUDA runtime,
// built by test_wait_flag.py with the host compiler.  One line of output per case: result, flag, status and
// counters afterwards, whether the zeros were waited for.
#include <cstdio>
#include <cstring>

#include "wait_flag.h"

struct Fake {
    bool waited = false;
    cudaError_t read(int* h, const int* d)
    {
        *h = *d;
        return cudaSuccess;
    }
    cudaError_t zero(int* d, size_t n)
    {
        std::memset(d, 0, n * sizeof(int));
        waited = false;
        return cudaSuccess;
    }
    cudaError_t wait()
    {
        waited = true;
        return cudaSuccess;
    }
};

int main()
{
    for (int set = 0; set < 2; ++set)
        for (int have = 0; have < 2; ++have) {
            int status = set, counters[3] = {2, 0, 5}, flag = 7;
            Fake f;
            const cudaError_t e = epic::take_wait_flag(f, &status, have ? counters : nullptr, 3, &flag);
            std::printf("%d %d %d %d %d %d %d\n", e == cudaSuccess, flag, status, counters[0], counters[1], counters[2], f.waited);
        }
    int flag = 7;
    Fake f;
    const cudaError_t e = epic::take_wait_flag(f, nullptr, nullptr, 0, &flag);
    std::printf("%d %d\n", e == cudaSuccess, flag);
    return 0;
}
