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
// times each (`fixed`: halo planes and pipeline fill).  Waves of units count in
// steps of 1/`parts`: workers that share an SM run faster when some of them
// have nothing left.  Returns the deepest c <= most within 1/`slack` of the
// shortest estimated sweep (deeper units re-read fewer halo planes).
// A fixed depth (64 planes, tensor cores 32) left small grids on a few SMs and
// large ones with a nearly empty last wave; us per sweep before and after:
// FP64 star 64^3 328 / 8.2, 512^3 1982 / 1863; FP32 gather 27-point 128^3
// 81 / 9.3, 512^3 375 / 337; tensor cores (with columns of one quarter each,
// mx3d.cu) 27-point 64^3 29 / 7.1, 256^3 78 / 52, 512^3 416 / 360, 7-point 512^3
// 229 / 197.
inline int pick_chunk(int nz, int64_t tiles, int64_t slots, int parts, int fixed, int most, int slack) {
    auto cost = [&](int c) { return (tiles * ((nz + c - 1) / c) * parts + slots - 1) / slots * (c + fixed); };
    int64_t least = cost(1);
    for (int c = 2; c <= most && c <= nz; ++c) least = cost(c) < least ? cost(c) : least;
    int c = most < nz ? most : nz;
    while (c > 1 && cost(c) > least + least / slack) --c;
    return c;
}

__host__ __device__ inline int64_t wrap_index(int64_t i, int64_t n) {
    int64_t m = i % n;
    return m < 0 ? m + n : m;
}

}  // namespace stx
