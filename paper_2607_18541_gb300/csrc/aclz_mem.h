// Device memory of the library: handles' arrays and the temporaries of
// uploads, encodes and hashes.
#pragma once

#include <cstddef>
#include <cuda_runtime.h>

namespace aclz {

// Bytes on the current device, usable in stream order on st (on any stream
// once st has been synchronized).
cudaError_t dev_alloc(void **p, size_t bytes, cudaStream_t st);

// Give p back in stream order on st (null: nothing).
void dev_free(void *p, cudaStream_t st);

// A temporary of one call, given back in stream order on the stream it was
// allocated on.
struct Scratch {
    void *p = nullptr;
    cudaStream_t st = nullptr;
    Scratch() = default;
    Scratch(const Scratch &) = delete;
    Scratch &operator=(const Scratch &) = delete;
    ~Scratch() { dev_free(p, st); }
    cudaError_t alloc(size_t bytes, cudaStream_t s) {
        st = s;
        return dev_alloc(&p, bytes, s);
    }
    template <class T>
    T *as() const {
        return (T *)p;
    }
};

}  // namespace aclz
