// add_side_stream against a fake CUDA runtime: one failed call leaves nothing behind that a later
// call would take for a stream with its event.
#include <cstdint>
#include <cstdio>

#include "side_stream.h"

static int fail_stream = 0, fail_event = 0, streams = 0, events = 0;
static uintptr_t next_handle = 16;

extern "C" {
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
    if (fail_stream) return cudaErrorMemoryAllocation;
    ++streams;
    *s = (cudaStream_t)(next_handle += 16);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) {
    if (fail_event) return cudaErrorMemoryAllocation;
    ++events;
    *e = (cudaEvent_t)(next_handle += 16);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) {
    --streams;
    return cudaSuccess;
}
}

#define EXPECT(c)                                   \
    do {                                            \
        if (!(c)) {                                 \
            std::printf("failed: %s\n", #c);        \
            return 1;                               \
        }                                           \
    } while (0)

int main() {
    std::vector<fpk::SideStream> side;
    EXPECT(fpk::add_side_stream(side) == cudaSuccess && side.size() == 1);
    fail_event = 1;
    EXPECT(fpk::add_side_stream(side) == cudaErrorMemoryAllocation && side.size() == 1);
    fail_event = 0;
    fail_stream = 1;
    EXPECT(fpk::add_side_stream(side) == cudaErrorMemoryAllocation && side.size() == 1);
    fail_stream = 0;
    EXPECT(fpk::add_side_stream(side) == cudaSuccess && side.size() == 2);
    for (const fpk::SideStream &x : side) EXPECT(x.st && x.ev);
    EXPECT(streams == 2 && events == 2);
    std::puts("ok");
    return 0;
}
