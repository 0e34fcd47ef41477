// fake_cuda.h -- a CUDA runtime for tests of host code without a GPU: device
// memory is host memory, streams run at once, kernels do nothing but what the
// test says, and calls fail where the test wants it.
#pragma once

#include <atomic>
#include <cstddef>
#include <map>
#include <mutex>

namespace fake {

extern std::atomic<bool> busy;             // events are not ready, streams wait
extern std::atomic<void*> busy_stream;     // this one alone waits
extern std::atomic<size_t> largest_malloc; // larger ones fail (device memory)
extern std::atomic<bool> event_fault;      // events report a device fault
extern std::mutex mu;
extern std::map<const void*, int> max_shared;   // cudaFuncAttributeMaxDynamicSharedMemorySize by function

}  // namespace fake

#define CHECK(c)                                                       \
    do {                                                               \
        if (!(c)) {                                                    \
            std::printf("%s:%d: %s\n", __FILE__, __LINE__, #c);        \
            std::exit(1);                                              \
        }                                                              \
    } while (0)
