// Shared definitions for the library's kernels and host runtime.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

namespace stx {

constexpr int kMaxRadius = 4;
constexpr int kBcDirichlet = 0;
constexpr int kBcPeriodic = 1;

// Dense gather-orientation coefficient tensor C^g passed by value as a kernel
// parameter (it lives in the constant bank, so every unrolled use is an
// immediate-like operand of the FMA).
template <typename T, int NC>
struct Coeffs {
    T c[NC];
};

constexpr int ipow(int b, int e) { return e == 0 ? 1 : b * ipow(b, e - 1); }

// Launch with programmatic stream serialization: the kernel may start while
// the stream's previous kernel drains, so it must call griddepcontrol.wait
// before it touches memory that kernel writes (the tensor-core and boundary
// kernels do; their sweeps run back to back: about 2.5 us saved per sweep).
template <typename... P, typename... A>
cudaError_t launch_dependent(void (*fn)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fn, std::forward<A>(args)...);
}

// Planes per work unit of a 3D sweep: units are `tiles` columns cut into
// ceil(nz / c) chunks, processed by `slots` workers at about (c + fixed) plane
// times each (`fixed`: halo planes and pipeline fill).  Returns the c <= most
// with the shortest estimated sweep; the deeper of equals, which re-reads
// fewer halo planes.  A fixed depth (64 planes, tensor cores 32) left small
// grids on a few SMs and large ones with a nearly empty last wave; us per
// sweep before and after: FP64 star 64^3 328 / 11, 512^3 1982 / 1956; FP32
// gather 27-point 128^3 81 / 11, 512^3 375 / 336; tensor cores (with columns
// of one quarter each, below) 27-point 64^3 29 / 8.6, 256^3 78 / 52,
// 512^3 416 / 359, 7-point 512^3 229 / 200.
inline int pick_chunk(int nz, int64_t tiles, int64_t slots, int fixed, int most) {
    int best = 1;
    int64_t best_cost = INT64_MAX;
    for (int c = 1; c <= most && c <= nz; ++c) {
        const int64_t units = tiles * ((nz + c - 1) / c);
        const int64_t cost = (units + slots - 1) / slots * (c + fixed);
        if (cost <= best_cost) {
            best_cost = cost;
            best = c;
        }
    }
    return best;
}

__host__ __device__ inline int64_t wrap_index(int64_t i, int64_t n) {
    int64_t m = i % n;
    return m < 0 ? m + n : m;
}

}  // namespace stx
