// cbg_context.h -- host state that belongs to a CUDA context: a memory pool, opted-in kernel
// attributes.  A device reset destroys all of it and the next call works in a new context, so it is
// kept per context id (unique over the process's lifetime), not once per process.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include <mutex>
#include <utility>
#include <vector>

namespace cbg {

// Id of the current context, which is created if need be; 0 when the driver does not tell.
inline unsigned long long context_id()
{
    using GetId = CUresult (*)(CUcontext, unsigned long long*);
    static const GetId get = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &p, 12000, cudaEnableDefault, &q) != cudaSuccess) {
            cudaGetLastError();
            return (GetId) nullptr;
        }
        return (GetId)p;
    }();
    unsigned long long id = 0;
    if (!get) return 0;
    if (get(nullptr, &id) == CUDA_SUCCESS) return id;
    cudaFree(nullptr);                       // no context yet (or none since a reset): the runtime makes one
    return get(nullptr, &id) == CUDA_SUCCESS ? id : 0;
}

// One T per context: the first call in it has make(T&) fill it in; kept if that returns true.
template <class T> class PerContext {
public:
    template <class Make> T get(Make make)
    {
        const unsigned long long id = context_id();
        std::lock_guard<std::mutex> lk(mu_);
        for (const auto& e : all_)
            if (e.first == id) return e.second;
        T t{};
        if (make(t)) {
            try {
                all_.emplace_back(id, t);
            } catch (...) {                  // (out of host memory: not kept)
            }
        }
        return t;
    }

private:
    std::mutex mu_;
    std::vector<std::pair<unsigned long long, T>> all_;
};

}  // namespace cbg
