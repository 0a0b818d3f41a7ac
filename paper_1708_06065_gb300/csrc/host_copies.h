// host_copies.h -- copies from pageable host memory to the device.
#pragma once

#include <cuda_runtime_api.h>

#include <memory>
#include <vector>

namespace lair {

// A copy from pageable memory may return before its source has been read: the runtime promises a staged source only
// where it has to stage at all, and on a host whose memory the GPU reads by itself it does not have to. So a source
// belongs to the handle until the stream has been synchronised.
class HostSources {
   public:
    // dst[0 .. size) = v, ordered on stream s
    template <class T>
    cudaError_t upload(T *dst, const std::shared_ptr<std::vector<T>> &v, cudaStream_t s) {
        if (v->empty()) return cudaSuccess;
        held.push_back(v);
        return cudaMemcpyAsync(dst, v->data(), sizeof(T) * v->size(), cudaMemcpyHostToDevice, s);
    }
    // after a synchronisation of the stream
    void release() { held.clear(); }

   private:
    std::vector<std::shared_ptr<void>> held;
};

}  // namespace lair
