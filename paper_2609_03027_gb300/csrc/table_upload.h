// Uploads of a set of tables of which a plan needs all or none.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

namespace epic {

class TableUpload {
public:
    // v goes to device memory that *dst points to after upload(); v stays alive until then
    template <class T, class U>
    void add(T** dst, const std::vector<U>& v)
    {
        items_.push_back(Item{reinterpret_cast<void**>(dst), v.data(), v.size() * sizeof(U)});
    }
    size_t bytes() const
    {
        size_t b = 0;
        for (const Item& i : items_) b += i.bytes;
        return b;
    }
    // All tables, or an error with every *dst as it was and nothing left allocated.  Rt: cudaMalloc, cudaMemcpy and
    // cudaFree, or stand-ins for them.
    template <class Rt>
    cudaError_t upload_with(Rt&& rt)
    {
        std::vector<void*> got(items_.size(), nullptr);
        cudaError_t e = cudaSuccess;
        for (size_t i = 0; i < items_.size() && e == cudaSuccess; ++i) {
            e = rt.malloc(&got[i], std::max<size_t>(1, items_[i].bytes));
            if (e != cudaSuccess) got[i] = nullptr;
            else if (items_[i].bytes) e = rt.copy(got[i], items_[i].src, items_[i].bytes);
        }
        for (size_t i = 0; i < items_.size(); ++i) {
            if (e == cudaSuccess) *items_[i].dst = got[i];
            else if (got[i]) rt.free(got[i]);
        }
        return e;
    }
    cudaError_t upload()
    {
        struct {
            cudaError_t malloc(void** p, size_t n) { return cudaMalloc(p, n); }
            cudaError_t copy(void* d, const void* s, size_t n) { return cudaMemcpy(d, s, n, cudaMemcpyHostToDevice); }
            void free(void* p) { cudaFree(p); }
        } rt;
        const cudaError_t e = upload_with(rt);
        if (e == cudaErrorMemoryAllocation) cudaGetLastError();  // reported here: not by the next launch's check
        return e;
    }

private:
    struct Item {
        void** dst;
        const void* src;
        size_t bytes;
    };
    std::vector<Item> items_;
};

}  // namespace epic
