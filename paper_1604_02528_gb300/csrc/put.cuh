// Descriptors of a call, from the host's stack to the device in stream order.
#pragma once

#include <cuda_runtime.h>

#include "launch.h"

namespace selinv {

template <typename T> __global__ void k_put(T v, T *dst) { *dst = v; }

// dst[0 .. n - 1] = v[0 .. n - 1].  A copy node of a graph that the caller is
// capturing would read v when the graph is launched, after the call's stack is
// gone; there the values travel as kernel arguments, which the graph holds.
template <typename T> inline cudaError_t put(T *dst, const T *v, int n, cudaStream_t st) {
    static_assert(sizeof(T) <= 4000, "fits the parameters of a kernel");
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    const bool capturing = st != nullptr && st != cudaStreamLegacy && cudaStreamIsCapturing(st, &cs) == cudaSuccess &&
                           cs != cudaStreamCaptureStatusNone;
    if (!capturing) return cudaMemcpyAsync(dst, v, n * sizeof(T), cudaMemcpyHostToDevice, st);
    for (int i = 0; i < n; i++) k_put<T><<<1, 1, 0, st>>>(v[i], dst + i);
    note_launch(n);
    return cudaGetLastError();
}

}  // namespace selinv
