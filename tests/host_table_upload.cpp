// Test driver for the upload of a set of device tables (table_upload.h) with a stand-in for the CUDA runtime,
// built by test_table_upload.py with the host compiler.  The k-th call of the stand-in's malloc and copy fails,
// for every k and for none; one line of output each: calls, tables held afterwards, allocations not given back,
// whether the held tables have the right contents.
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "table_upload.h"

struct Fake {
    int fail_at, calls = 0, live = 0;
    cudaError_t malloc(void** p, size_t n)
    {
        if (calls++ == fail_at) return cudaErrorMemoryAllocation;
        *p = std::malloc(n);
        ++live;
        return cudaSuccess;
    }
    cudaError_t copy(void* d, const void* s, size_t n)
    {
        if (calls++ == fail_at) return cudaErrorInvalidValue;
        std::memcpy(d, s, n);
        return cudaSuccess;
    }
    void free(void* p)
    {
        std::free(p);
        --live;
    }
};

int main()
{
    const std::vector<int> a = {1, 2, 3}, none;
    const std::vector<float2> b = {make_float2(4.f, 5.f)};
    for (int k = 0; k <= 5; ++k) {
        int *da = nullptr, *dn = nullptr;
        void* db = nullptr;
        epic::TableUpload t;
        t.add(&da, a);
        t.add(&dn, none);
        t.add(&db, b);
        Fake f{k};
        const cudaError_t e = t.upload_with(f);
        const int held = (da != nullptr) + (dn != nullptr) + (db != nullptr);
        const bool same = da && db && !std::memcmp(da, a.data(), 12) && !std::memcmp(db, b.data(), 8);
        std::printf("%d %d %d %d %d\n", e == cudaSuccess, held, f.live, same, (int)t.bytes());
    }
    return 0;
}
