// side_stream.h -- streams that a call runs on beside its ensemble's own.
#pragma once
#include <vector>

#include <cuda_runtime_api.h>

namespace fpk {

struct SideStream {   // joined to the ensemble's stream before its call goes on
    cudaStream_t st = nullptr;
    cudaEvent_t ev = nullptr;
};

// One more, with its event; after a failure `side` is as it was, so that a later call can try again.
inline cudaError_t add_side_stream(std::vector<SideStream> &side) {
    side.emplace_back();
    SideStream &x = side.back();
    cudaError_t e = cudaStreamCreateWithFlags(&x.st, cudaStreamNonBlocking);
    if (e == cudaSuccess) {
        e = cudaEventCreateWithFlags(&x.ev, cudaEventDisableTiming);
        if (e != cudaSuccess) cudaStreamDestroy(x.st);
    }
    if (e != cudaSuccess) side.pop_back();
    return e;
}

}  // namespace fpk
