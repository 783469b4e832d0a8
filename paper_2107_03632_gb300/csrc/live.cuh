// Vectors that the kernels of a chain hand on to one another (launch_chained
// in common.cuh).
//
// A chained kernel is resident while the one before it still writes, so what
// that one writes is not constant for the kernel's lifetime.  It must not be
// read through the non-coherent path (__ldg, or a `const ... __restrict__`
// parameter, which the compiler turns into the same load), and no parameter
// that points to it may be __restrict__: nothing then keeps its loads behind
// pdl_wait().  A Live<T> parameter has no address to pass to __ldg and no
// qualifier; its elements are ordinary loads, which the wait's memory clobber
// holds back.  Vectors that a chained kernel writes are plain pointers.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace rbffd {

template <class T>
struct Live {
    const T* p;
    Live() = default;
    __host__ __device__ Live(const T* q) : p(q) {}
    __device__ __forceinline__ T operator[](int64_t i) const { return p[i]; }
    __device__ __forceinline__ explicit operator bool() const { return p != nullptr; }
};

}  // namespace rbffd
