// CUDA-core gather kernels: the baseline form of the stencil,
//   B[x] = sum_o C^g[o] * A[x + o - r]                       (Eq. (stencil-2d9p))
// evaluated point by point with FMAs.  One launch advances the field by `tb`
// time steps (temporal blocking): a block stages its output tile plus a halo
// of width r*tb in shared memory, performs tb sub-steps there (the valid
// region shrinks by r per sub-step; with a zero Dirichlet boundary, points
// outside the domain are reset to 0 after every sub-step), and writes the
// tile once.  Each thread computes blocks of 4 x 4 outputs (2D FP32) or strips
// of outputs along the slowest axis, reusing every loaded shared-memory row
// for all outputs it feeds.
//
// Single grids run persistent kernels that stage their tiles with TMA:
//  * 2D: each CTA walks its tiles through a ring of NST shared-memory stages
//    (two or three), the next tiles' halo blocks loading (one
//    cp.async.bulk.tensor each, zero fill outside the grid = the Dirichlet
//    halo) while the current one computes.
//  * 3D (one step per launch): a work unit is a column of output planes; the
//    CTA streams its input planes through a ring of 2r+2 plane buffers, each
//    loaded by TMA while the planes before it are used, so every input plane
//    is read from global memory once per unit instead of once per 3D tile.
// With a periodic boundary, tiles (3D: planes of units) whose halo crosses
// the grid's edge are staged by TMA like the others; then only their cells
// outside the grid are overwritten with wrapped values (`wrap_halo_block`).
// Waits are bounded; a timeout sets the plan's host-visible error word.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <type_traits>

#include "common.cuh"
#include "kernels.h"
#include "mxutil.cuh"
#include "ptx.cuh"

namespace stx {

namespace {

constexpr int kBX = 32;   // threads along the contiguous axis (one warp)
constexpr int kRS = 8;    // outputs per thread along the strip axis

// Asynchronous global->shared copy of one element (Ampere-style cp.async):
// many copies stay in flight per thread, so the tile load runs at HBM rate.
template <typename T>
__device__ __forceinline__ void cp_async_elem(T* dst, const T* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if constexpr (sizeof(T) == 4)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
}

__device__ __forceinline__ void cp_async_16(float* dst, const float* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Address of a tile element after the boundary rule, or nullptr for a zero.
template <typename T>
__device__ __forceinline__ const T* src2(const T* __restrict__ a, int64_t y, int64_t x, int64_t ny,
                                         int64_t nx, int64_t ldx, int bc) {
    if (y < 0 || y >= ny || x < 0 || x >= nx) {
        if (bc == kBcDirichlet) return nullptr;
        y = wrap_index(y, ny);
        x = wrap_index(x, nx);
    }
    return a + y * ldx + x;
}

template <typename T>
__device__ __forceinline__ const T* src3(const T* __restrict__ a, int64_t z, int64_t y, int64_t x,
                                         int64_t nz, int64_t ny, int64_t nx, int64_t ldx, int bc) {
    if (z < 0 || z >= nz || y < 0 || y >= ny || x < 0 || x >= nx) {
        if (bc == kBcDirichlet) return nullptr;
        z = wrap_index(z, nz);
        y = wrap_index(y, ny);
        x = wrap_index(x, nx);
    }
    return a + (z * ny + y) * ldx + x;
}

// ---------------------------------------------------------------------------
// 2D FP32 sub-steps, register-blocked: a thread computes kVR rows x 4 adjacent
// columns.  Each input row it needs is read as three 16-byte shared-memory
// loads (columns x-4 .. x+7, enough for r <= 4) and every weight is applied to
// four columns at once, so an update costs its P FMAs and about one
// shared-memory load (the scalar strips spend about 7.5 loads and the index
// arithmetic around them).  The sum of an output runs over the rows, then the
// columns of C^g in order, as everywhere in this file: results do not depend
// on tiles, depth or blocking.
// ---------------------------------------------------------------------------
constexpr int kVR = 4;         // rows per thread
constexpr int kSlackRows = 4;  // rows after a buffer that ragged blocks read (and, before the last sub-step, write)

// base = element (row of the first output - R, column of the first output - 4).
template <int R, bool STAR>
__device__ __forceinline__ void block_f32(const float* base, int SX, const Coeffs<float, ipow(2 * R + 1, 2)>& cf,
                                          float (&acc)[kVR][4]) {
    static_assert(R <= 4, "three 16-byte loads cover x-4 .. x+7");
    constexpr int W = 2 * R + 1;
#pragma unroll
    for (int j = 0; j < kVR; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[j][q] = 0.0f;
#pragma unroll
    for (int yi = 0; yi < kVR + 2 * R; ++yi) {
        float v[12];   // v[k] = column x - 4 + k of input row yi
#pragma unroll
        for (int k4 = 0; k4 < 3; ++k4) {
            const float4 u = *reinterpret_cast<const float4*>(base + yi * SX + 4 * k4);
            v[4 * k4] = u.x;
            v[4 * k4 + 1] = u.y;
            v[4 * k4 + 2] = u.z;
            v[4 * k4 + 3] = u.w;
        }
#pragma unroll
        for (int j = 0; j < kVR; ++j) {
            const int a = yi - j;
            if (a >= 0 && a < W) {
#pragma unroll
                for (int b = 0; b < W; ++b)
                    if (!STAR || a == R || b == R) {
                        const float w = cf.c[a * W + b];
#pragma unroll
                        for (int q = 0; q < 4; ++q) acc[j][q] = fmaf(w, v[4 + q + b - R], acc[j][q]);
                    }
            }
        }
    }
}

// Geometry of a tile of TY x TX outputs in shared memory for depth tb: H halo
// rows, HX halo columns (a multiple of 4), SY x SX elements.  Element (sy, sx)
// is grid point (y0 - H + sy, x0 - HX + sx).
struct TileGeom {
    int H, HX, SY, SX;
    __host__ __device__ TileGeom(int r, int tb, int ty, int tx)
        : H(r * tb), HX((r * tb + 3) / 4 * 4), SY(ty + 2 * r * tb), SX(tx + 2 * ((r * tb + 3) / 4 * 4)) {}
    // One buffer: the tile, then the slack rows (which also end the last row's ragged reads).
    __host__ __device__ int elems() const { return (SY + kSlackRows) * SX; }
};
constexpr int kLeadElems = 32;   // before the first buffer: ragged reads left of row 0

// Sub-step t < tb of a tile: src -> dst, both in shared memory.  Rows R t ..
// SY - R t and the columns that the later sub-steps still need are computed,
// rounded out to whole blocks: the extra cells read cells outside the tile
// (neighbouring rows' ends, slack), hold garbage and are never used.  `zero`
// (tiles across the grid's edge, zero boundary): cells outside the grid are
// zero again after the sub-step.
template <int R, bool STAR, int TX>
__device__ __forceinline__ void substep_f32(const float* src, float* dst, const TileGeom& g, int t, int tb, bool zero,
                                            int ny, int nx, int gy0, int gx0, int tid, int nthreads,
                                            const Coeffs<float, ipow(2 * R + 1, 2)>& cf) {
    const int lo = R * t;
    const int c0 = (g.HX - R * (tb - t)) & ~3;
    const int ncg = (g.HX + TX + R * (tb - t) - c0 + 3) >> 2;
    const int nstrips = (g.SY - 2 * lo + kVR - 1) / kVR;
    const unsigned magic = ((1u << 20) + ncg - 1) / ncg;   // item / ncg = item * magic >> 20 for items below 2^20 / ncg
    for (int item = tid; item < nstrips * ncg; item += nthreads) {
        const int strip = (int)((item * magic) >> 20), cgi = item - strip * ncg;
        const int sy = lo + strip * kVR, sx = c0 + 4 * cgi;
        float acc[kVR][4];
        block_f32<R, STAR>(src + (sy - R) * g.SX + (sx - 4), g.SX, cf, acc);
        if (zero) {
#pragma unroll
            for (int j = 0; j < kVR; ++j) {
                const int gy = gy0 + sy + j;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int gx = gx0 + sx + q;
                    if (gy < 0 || gy >= ny || gx < 0 || gx >= nx) acc[j][q] = 0.0f;
                }
            }
        }
#pragma unroll
        for (int j = 0; j < kVR; ++j)
            *reinterpret_cast<float4*>(dst + (sy + j) * g.SX + sx) = make_float4(acc[j][0], acc[j][1], acc[j][2], acc[j][3]);
    }
}

// Last sub-step of a tile, to the grid: the valid region starts at the aligned
// column HX, so rows of four outputs go out as 16-byte stores when the grid's
// rows are 16-byte aligned (`vec`).
template <int R, bool STAR, int TY, int TX>
__device__ __forceinline__ void last_substep_f32(const float* src, float* __restrict__ out, const TileGeom& g, bool vec,
                                                 int ny, int nx, int64_t ldx, int y0, int x0, int tid, int nthreads,
                                                 const Coeffs<float, ipow(2 * R + 1, 2)>& cf) {
    static_assert(TY % kVR == 0 && TX % 4 == 0, "whole blocks");
    constexpr int ncg = TX / 4;
    for (int item = tid; item < TY / kVR * ncg; item += nthreads) {
        const int strip = item / ncg, cgi = item - strip * ncg;   // a warp: consecutive column groups
        float acc[kVR][4];
        block_f32<R, STAR>(src + (g.H + strip * kVR - R) * g.SX + (g.HX + 4 * cgi - 4), g.SX, cf, acc);
        const int gx = x0 + 4 * cgi;
#pragma unroll
        for (int j = 0; j < kVR; ++j) {
            const int gy = y0 + strip * kVR + j;
            if (gy < ny) {
                float* o = out + (int64_t)gy * ldx + gx;
                if (vec && gx + 3 < nx) {
                    *reinterpret_cast<float4*>(o) = make_float4(acc[j][0], acc[j][1], acc[j][2], acc[j][3]);
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (gx + q < nx) o[q] = acc[j][q];
                }
            }
        }
    }
}

// One FP32 tile (origin y0, x0) loaded element by element (any row alignment,
// either boundary) and advanced by tb steps; buffers a and b ping-pong.  A
// grid without 16-byte rows gets its outputs through shared memory: written
// as blocks, four 4-byte stores 16 bytes apart per lane would touch every
// sector four times.  WIDE: the last tiles of a row reach past column 2^31 (a
// template parameter: 64-bit columns in every tile cost up to 5%, 1021 x 1533).
template <int R, bool STAR, int TY, int TX, bool WIDE = false>
__device__ __forceinline__ void tile2_f32(const float* __restrict__ in, float* __restrict__ out, int ny, int nx,
                                          int64_t ldx, int bc, int tb, const Coeffs<float, ipow(2 * R + 1, 2)>& cf,
                                          int y0, int x0, float* a, float* b, int tid, int nthreads) {
    const TileGeom g(R, tb, TY, TX);
    const int gy0 = y0 - g.H, gx0 = x0 - g.HX;
    const int lane = tid & 31, warp = tid >> 5, nwarps = nthreads >> 5;
    const auto gxl = (std::conditional_t<WIDE, int64_t, int>)gx0;
    const bool inside = gy0 >= 0 && gy0 + g.SY <= ny && gx0 >= 0 && gxl + g.SX <= nx;
    const bool vec = ldx % 4 == 0 && ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 15u) == 0;
    for (int sy = warp; sy < g.SY; sy += nwarps) {
        float* d = a + sy * g.SX;
        if (inside && vec) {
            const float* s = in + (int64_t)(gy0 + sy) * ldx + gx0;
            for (int sx = 4 * lane; sx < g.SX; sx += 128) cp_async_16(d + sx, s + sx);
        } else if (inside) {
            const float* s = in + (int64_t)(gy0 + sy) * ldx + gx0;
            for (int sx = lane; sx < g.SX; sx += 32) cp_async_elem(d + sx, s + sx);
        } else {
            for (int sx = lane; sx < g.SX; sx += 32) {
                const float* s = src2(in, gy0 + sy, gxl + sx, ny, nx, ldx, bc);
                if (s) cp_async_elem(d + sx, s);
                else d[sx] = 0.0f;
            }
        }
    }
    cp_async_wait_all();
    __syncthreads();
    const bool zero = !inside && bc == kBcDirichlet;
    for (int t = 1; t < tb; ++t) {
        substep_f32<R, STAR, TX>(a, b, g, t, tb, zero, ny, nx, gy0, gx0, tid, nthreads, cf);
        float* const other = a;
        a = b;
        b = other;
        __syncthreads();
    }
    if (vec) {
        last_substep_f32<R, STAR, TY, TX>(a, out, g, true, ny, nx, ldx, y0, x0, tid, nthreads, cf);
    } else {
        substep_f32<R, STAR, TX>(a, b, g, tb, tb, false, ny, nx, gy0, gx0, tid, nthreads, cf);
        __syncthreads();
        const int cols = min(TX, nx - x0);
        for (int y = warp; y < TY && y0 + y < ny; y += nwarps) {
            const float* s = b + (g.H + y) * g.SX + g.HX;
            float* o = out + (int64_t)(y0 + y) * ldx + x0;
            for (int x = lane; x < cols; x += 32) o[x] = s[x];
        }
    }
    __syncthreads();   // both buffers are free
}

// ---------------------------------------------------------------------------
// 2D.  Block = (32, BY) threads; output tile TY x TX.  Strips run along y.
// ---------------------------------------------------------------------------
// One output tile (origin y0, x0) advanced by tb steps; shared by the
// single-problem and the batched kernels.
template <typename T, int R, bool STAR, int BY, int TX, int TY>
__device__ __forceinline__ void gather2d_tile(const T* __restrict__ in, T* __restrict__ out, int64_t ny,
                                              int64_t nx, int64_t ldx, int bc, int tb, const Coeffs<T, ipow(2 * R + 1, 2)>& cf,
                                              int64_t y0, int64_t x0, T* smem) {
    constexpr int W = 2 * R + 1;
    const int H = R * tb;
    const int SX = TX + 2 * H;
    const int SY = TY + 2 * H;
    // buf[0] | buf[1] (tb > 1 only) | kRS slack rows read (never used) by ragged strips
    T* buf[2] = {smem, smem + SY * SX};
    const int rows_alloc = (tb > 1 ? 2 * SY : SY) + kRS;
    const int tx = threadIdx.x, ty = threadIdx.y;

    const bool interior = (y0 - H >= 0) && (y0 + TY + H <= ny) && (x0 - H >= 0) && (x0 + TX + H <= nx);
    for (int sy = ty; sy < rows_alloc; sy += BY) {
        const int64_t gy = y0 - H + sy;
        for (int sx = tx; sx < SX; sx += kBX) {
            const int64_t gx = x0 - H + sx;
            T* d = smem + sy * SX + sx;
            const T* g = nullptr;
            if (sy < SY) g = interior ? in + gy * ldx + gx : src2(in, gy, gx, ny, nx, ldx, bc);
            if (g) cp_async_elem(d, g);
            else *d = T(0);
        }
    }
    cp_async_wait_all();
    __syncthreads();

    for (int t = 1; t <= tb; ++t) {
        const T* src = buf[(t - 1) & 1];
        T* dst = buf[t & 1];
        const bool last = (t == tb);
        const int lo = R * t;
        const int Ht = SY - 2 * lo, Wt = SX - 2 * lo;
        const int nstrips = (Ht + kRS - 1) / kRS;
        for (int strip = ty; strip < nstrips; strip += BY) {
            const int sy0 = lo + strip * kRS;
            for (int c = tx; c < Wt; c += kBX) {
                const int sx = lo + c;
                T acc[kRS];
#pragma unroll
                for (int j = 0; j < kRS; ++j) acc[j] = T(0);
                const T* base = src + (sy0 - R) * SX + (sx - R);
#pragma unroll
                for (int yi = 0; yi < kRS + 2 * R; ++yi) {
                    T v[W];
#pragma unroll
                    for (int b = 0; b < W; ++b) v[b] = base[yi * SX + b];
#pragma unroll
                    for (int j = 0; j < kRS; ++j) {
                        const int a = yi - j;
                        if (a >= 0 && a < W) {
#pragma unroll
                            for (int b = 0; b < W; ++b) {
                                if (!STAR || a == R || b == R) acc[j] = fma(cf.c[a * W + b], v[b], acc[j]);
                            }
                        }
                    }
                }
                const int64_t gx = x0 - H + sx;
#pragma unroll
                for (int j = 0; j < kRS; ++j) {
                    const int sy = sy0 + j;
                    if (sy < SY - lo) {
                        const int64_t gy = y0 - H + sy;
                        if (last) {
                            if (gy < ny && gx < nx) out[gy * ldx + gx] = acc[j];
                        } else {
                            const bool outside = (bc == kBcDirichlet) && (gy < 0 || gy >= ny || gx < 0 || gx >= nx);
                            dst[sy * SX + sx] = outside ? T(0) : acc[j];
                        }
                    }
                }
            }
        }
        __syncthreads();
    }
}

template <typename T, int R, bool STAR, int BY, int TX, int TY, bool WIDE>
__global__ void __launch_bounds__(kBX * BY)
gather2d_kernel(const T* __restrict__ in, T* __restrict__ out, int64_t ny, int64_t nx, int64_t ldx, int bc,
                int tb, Coeffs<T, ipow(2 * R + 1, 2)> cf) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if constexpr (sizeof(T) == 4) {
        float* a = reinterpret_cast<float*>(smem_raw) + kLeadElems;
        tile2_f32<R, STAR, TY, TX, WIDE>(in, out, (int)ny, (int)nx, ldx, bc, tb, cf, (int)blockIdx.y * TY,
                                         (int)blockIdx.x * TX, a, a + TileGeom(R, tb, TY, TX).elems(),
                                         threadIdx.y * kBX + threadIdx.x, kBX * BY);
    } else {
        gather2d_tile<T, R, STAR, BY, TX, TY>(in, out, ny, nx, ldx, bc, tb, cf, (int64_t)blockIdx.y * TY,
                                              (int64_t)blockIdx.x * TX, reinterpret_cast<T*>(smem_raw));
    }
}

// Persistent batched sweep: the tiles of many independent problems, each
// advanced by its own depth, processed by one grid-stride launch.  Problem
// p owns tiles [tile0[p], tile0[p+1]); its coefficients sit at coef + p*NC.
// Registers: FP64 two CTAs' worth per SM (with one, the compiler takes up to 254
// and a lone CTA's barriers leave the FP64 pipe idle: 48 problems of up to 1500^2,
// 24 steps, r = 1 star 3.89 ms, with two 3.22; r = 3 star 7.20 and 6.30), but for
// the 49 weights of r = 3 boxes in the large tile (22.6 ms, with two 25.3).
template <typename T, int R, bool STAR, int BY, int TX, int TY>
__global__ void __launch_bounds__(kBX * BY, sizeof(T) == 8 ? (R == 3 && !STAR && TY == 64 ? 1 : 2) : R == 1 ? 16 / BY + 1 : 1)
gather2d_batch_kernel(const BatchProblem* __restrict__ probs, int nprob, int total_tiles,
                      const T* __restrict__ coef) {
    constexpr int NC = ipow(2 * R + 1, 2);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int lo = 0;   // problem of tile t: the last one whose first tile <= t
    for (int t = blockIdx.x; t < total_tiles; t += gridDim.x) {
        // a CTA's tiles ascend: search on from the previous tile's problem, a
        // warp's width at a time (each lane one candidate)
        for (;;) {
            const int k = lo + 1 + (int)threadIdx.x;
            const unsigned past = __ballot_sync(0xffffffffu, k >= nprob || probs[k].tile0 > t);
            if (past) {
                lo += __ffs(past) - 1;
                break;
            }
            lo += 32;
        }
        const BatchProblem P = probs[lo];
        const int local = t - P.tile0;
        const int y0 = local / P.tiles_x * TY, x0 = local % P.tiles_x * TX;
        Coeffs<T, NC> cf;
#pragma unroll
        for (int i = 0; i < NC; ++i) cf.c[i] = coef[(size_t)P.coef_index * NC + i];
        if constexpr (sizeof(T) == 4) {
            float* a = reinterpret_cast<float*>(smem_raw) + kLeadElems;
            tile2_f32<R, STAR, TY, TX>((const float*)P.src, (float*)P.dst, P.ny, P.nx, P.nx, P.bc, P.depth, cf, y0, x0, a,
                                       a + TileGeom(R, P.depth, TY, TX).elems(), threadIdx.y * kBX + threadIdx.x, kBX * BY);
        } else {
            gather2d_tile<T, R, STAR, BY, TX, TY>((const T*)P.src, (T*)P.dst, P.ny, P.nx, P.nx, P.bc, P.depth, cf, y0, x0,
                                                  reinterpret_cast<T*>(smem_raw));
        }
    }
}

// ---------------------------------------------------------------------------
// 3D.  Block = (32, BY) threads covering (y, x); strips run along z.
// Output tile TZ x TY x TX.
// ---------------------------------------------------------------------------
template <typename T, int R, bool STAR, int BY, int TX, int TY, int TZ>
__global__ void __launch_bounds__(kBX * BY)
gather3d_kernel(const T* __restrict__ in, T* __restrict__ out, int64_t nz, int64_t ny, int64_t nx,
                int64_t ldx, int bc, int tb, Coeffs<T, ipow(2 * R + 1, 3)> cf) {
    constexpr int W = 2 * R + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* smem = reinterpret_cast<T*>(smem_raw);
    const int H = R * tb;
    const int SX = TX + 2 * H, SY = TY + 2 * H, SZ = TZ + 2 * H;
    const int plane = SY * SX;
    // buf[0] | buf[1] (tb > 1 only) | kRS slack planes read (never used) by ragged strips
    const int planes_alloc = (tb > 1 ? 2 * SZ : SZ) + kRS;
    T* buf[2] = {smem, smem + SZ * plane};
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int64_t z0 = (int64_t)blockIdx.z * TZ, y0 = (int64_t)blockIdx.y * TY,
                  x0 = (int64_t)blockIdx.x * TX;
    const bool interior = (z0 - H >= 0) && (z0 + TZ + H <= nz) && (y0 - H >= 0) &&
                          (y0 + TY + H <= ny) && (x0 - H >= 0) && (x0 + TX + H <= nx);
    for (int sz = 0; sz < planes_alloc; ++sz) {
        const int64_t gz = z0 - H + sz;
        for (int sy = ty; sy < SY; sy += BY) {
            const int64_t gy = y0 - H + sy;
            for (int sx = tx; sx < SX; sx += kBX) {
                const int64_t gx = x0 - H + sx;
                T* d = smem + sz * plane + sy * SX + sx;
                const T* g = nullptr;
                if (sz < SZ) g = interior ? in + (gz * ny + gy) * ldx + gx : src3(in, gz, gy, gx, nz, ny, nx, ldx, bc);
                if (g) cp_async_elem(d, g);
                else *d = T(0);
            }
        }
    }
    cp_async_wait_all();
    __syncthreads();

    for (int t = 1; t <= tb; ++t) {
        const T* src = buf[(t - 1) & 1];
        T* dst = buf[t & 1];
        const bool last = (t == tb);
        const int lo = R * t;
        const int Dt = SZ - 2 * lo, Ht = SY - 2 * lo, Wt = SX - 2 * lo;
        const int nstrips = (Dt + kRS - 1) / kRS;
        for (int strip = 0; strip < nstrips; ++strip) {
            const int sz0 = lo + strip * kRS;
            for (int cy = ty; cy < Ht; cy += BY) {
                const int sy = lo + cy;
                for (int cx = tx; cx < Wt; cx += kBX) {
                    const int sx = lo + cx;
                    T acc[kRS];
#pragma unroll
                    for (int j = 0; j < kRS; ++j) acc[j] = T(0);
                    const T* base = src + (sz0 - R) * plane + (sy - R) * SX + (sx - R);
#pragma unroll
                    for (int zi = 0; zi < kRS + 2 * R; ++zi) {
#pragma unroll
                        for (int a1 = 0; a1 < W; ++a1) {
                            T v[W];
#pragma unroll
                            for (int b = 0; b < W; ++b) v[b] = base[zi * plane + a1 * SX + b];
#pragma unroll
                            for (int j = 0; j < kRS; ++j) {
                                const int a0 = zi - j;
                                if (a0 >= 0 && a0 < W) {
#pragma unroll
                                    for (int b = 0; b < W; ++b) {
                                        const bool on_axis = (a1 == R && b == R) || (a0 == R && b == R) ||
                                                             (a0 == R && a1 == R);
                                        if (!STAR || on_axis)
                                            acc[j] = fma(cf.c[(a0 * W + a1) * W + b], v[b], acc[j]);
                                    }
                                }
                            }
                        }
                    }
                    const int64_t gy = y0 - H + sy, gx = x0 - H + sx;
#pragma unroll
                    for (int j = 0; j < kRS; ++j) {
                        const int sz = sz0 + j;
                        if (sz < SZ - lo) {
                            const int64_t gz = z0 - H + sz;
                            if (last) {
                                if (gz < nz && gy < ny && gx < nx) out[(gz * ny + gy) * ldx + gx] = acc[j];
                            } else {
                                const bool outside = (bc == kBcDirichlet) &&
                                                     (gz < 0 || gz >= nz || gy < 0 || gy >= ny || gx < 0 || gx >= nx);
                                dst[sz * plane + sy * SX + sx] = outside ? T(0) : acc[j];
                            }
                        }
                    }
                }
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// TMA-staged persistent kernels (single grids).
// ---------------------------------------------------------------------------
constexpr long long kGatherWait = 4000000000LL;   // ~2 s of SM clock per wait

__host__ __device__ constexpr int round_up(int v, int a) { return (v + a - 1) / a * a; }

// Bounded wait on an mbarrier phase; false when the limit ran out.
__device__ __forceinline__ bool gwait(uint64_t* bar, uint32_t parity) {
    return ptx::mbar_wait(bar, parity, kGatherWait);
}

// 2D tile: TY x TX outputs per tile, threads (32, BY), a ring of TMA stages
// (one less in flight ahead of the tile being computed).  FP32: 32 x 128
// outputs (256 blocks of the last sub-step, one per thread); one step per
// launch takes three stages (three CTAs of 62 KB per SM, six tiles in flight),
// several steps two and a work buffer (72-78 KB: three CTAs per SM for depths
// up to r tb = 4, so that one CTA's barriers and loads hide behind the
// others' sub-steps).  FP64: 32 x 32 outputs, one strip of 8 rows per thread,
// two stages, four CTAs of four warps per SM: the FP64 pipe (2 FMAs per clock
// and SM) is the limit, and with two CTAs of eight warps it sat idle a quarter
// of the time around their barriers.  Grids with fewer such tiles than SMs
// take 16 x 32 tiles (strips of 4 rows).  us per sweep before / after, star
// r = 1: 256^2 8.3 / 2.8, 4096^2 187 / 175; box r = 2 4096^2 840 / 815: 515 G FMAs per
// second, where bare FP64 FMAs on all SMs reach 525.
// Several FP64 steps per sweep compute a halo of r (tb - t) points around the
// tile at sub-step t, so grids with many tiles take 64 x 32 outputs by CTAs of
// eight warps, two per SM (stars and r = 4 only while two fit the shared memory):
// 4096^2, us per step with 32 / 64 rows, r = 3 star tb = 2 811 / 725, tb = 3
// 994 / 868, r = 3 box tb = 3 3499 / 3204, tb = 4 (one CTA) 4081 / 3815, r = 2 box
// tb = 4 1847 / 1709, r = 1 box tb = 4 628 / 615; one CTA: r = 4 star tb = 3
// 1261 / 1357, box 100 x 30000 1370 / 1424.
template <typename T>
struct Tile2 {
    static constexpr int TY = 32;
    static constexpr int TYS = sizeof(T) == 4 ? 32 : 16;   // small grids
    static constexpr int TYD = sizeof(T) == 4 ? 32 : 64;   // several steps per sweep, many tiles
    static constexpr int TX = sizeof(T) == 4 ? 128 : 32;
    static constexpr int by(int ty) { return sizeof(T) == 4 || ty == 64 ? 8 : 4; }   // warps per CTA
    static constexpr int AL = 16 / (int)sizeof(T);   // TMA x granule (16 bytes)
};
__host__ __device__ constexpr int stages2(size_t elem, bool multi) { return elem == 4 && !multi ? 3 : 2; }

struct G2Args {
    const void* in;
    void* out;
    unsigned int* err;   // host-mapped error word (may be null)
    int64_t ldx;         // row stride of the grids (elements)
    int ny, nx, bc, tb;
    int tiles_x, tiles_total;
    int* sched;          // tile counter pair (0 between launches): [0] tiles claimed, [1] CTAs done; null: fixed shares
};

// Shared-memory layout of the 2D kernel for depth tb: the TMA ring's stages
// and, for tb > 1, a work buffer for the sub-step ping-pong; slack rows after
// each buffer are read by ragged strips or blocks (FP32 blocks also write
// them), never used.
template <typename T, int TY>
struct Layout2 {
    int H, HX, SY, SX, buf;   // halo rows, halo columns, rows, columns, elements per buffer
    __host__ __device__ Layout2(int r, int tb) {
        H = r * tb;
        HX = round_up(H, Tile2<T>::AL);
        SY = TY + 2 * H;
        SX = Tile2<T>::TX + 2 * HX;
        buf = round_up((SY + (sizeof(T) == 4 ? kSlackRows : kRS)) * SX, 128 / (int)sizeof(T));
    }
    __host__ __device__ int buffers(int tb) const { return stages2(sizeof(T), tb > 1) + (tb > 1 ? 1 : 0); }
    // alignment slack, lead elements, buffers, barriers
    __host__ __device__ size_t bytes(int tb) const { return 128 + 128 + (size_t)buffers(tb) * buf * sizeof(T) + 64; }
};

// One sub-step of depth t of the 2D tile: src -> dst (or -> the output grid
// on the last sub-step).  The buffer's element (sy, sx) is grid point
// (y0 - H + sy, x0 - HX + sx).
template <typename T, int R, bool STAR, int TY>
__device__ __forceinline__ void substep2(const T* src, T* dst, T* __restrict__ out, const Layout2<T, TY>& L, int t,
                                         bool last, int64_t ny, int64_t nx, int64_t ldx, int bc, int64_t y0, int64_t x0,
                                         const Coeffs<T, ipow(2 * R + 1, 2)>& cf) {
    constexpr int W = 2 * R + 1;
    constexpr int RS = TY / Tile2<T>::by(TY);   // rows per strip
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int lo = R * t;                  // rows of the valid region skipped at the top
    const int lox = L.HX - L.H + R * t;    // columns skipped at the left
    const int Ht = L.SY - 2 * lo, Wt = L.SX - 2 * lox;
    const int nstrips = (Ht + RS - 1) / RS;
    for (int strip = ty; strip < nstrips; strip += Tile2<T>::by(TY)) {
        const int sy0 = lo + strip * RS;
        for (int c = tx; c < Wt; c += kBX) {
            const int sx = lox + c;
            T acc[RS];
#pragma unroll
            for (int j = 0; j < RS; ++j) acc[j] = T(0);
            const T* base = src + (sy0 - R) * L.SX + (sx - R);
#pragma unroll
            for (int yi = 0; yi < RS + 2 * R; ++yi) {
                T v[W];
#pragma unroll
                for (int b = 0; b < W; ++b) v[b] = base[yi * L.SX + b];
#pragma unroll
                for (int j = 0; j < RS; ++j) {
                    const int a = yi - j;
                    if (a >= 0 && a < W) {
#pragma unroll
                        for (int b = 0; b < W; ++b)
                            if (!STAR || a == R || b == R) acc[j] = fma(cf.c[a * W + b], v[b], acc[j]);
                    }
                }
            }
            const int64_t gx = x0 - L.HX + sx;
#pragma unroll
            for (int j = 0; j < RS; ++j) {
                const int sy = sy0 + j;
                if (sy < L.SY - lo) {
                    const int64_t gy = y0 - L.H + sy;
                    if (last) {
                        if (gy < ny && gx < nx) out[gy * ldx + gx] = acc[j];
                    } else {
                        const bool outside = (bc == kBcDirichlet) && (gy < 0 || gy >= ny || gx < 0 || gx >= nx);
                        dst[sy * L.SX + sx] = outside ? T(0) : acc[j];
                    }
                }
            }
        }
    }
}

// i mod n; one add or subtract for the usual halo offsets (|i| < 2n).
__device__ __forceinline__ int wrap_fast(int i, int n) {
    if (i >= 0 && i < n) return i;
    if (i < 0 && i >= -n) return i + n;
    if (i >= n && i < 2 * n) return i - n;
    const int m = i % n;
    return m < 0 ? m + n : m;
}

// Periodic boundary, a staged block (SY rows x SX columns, cell (0, 0) =
// grid point (gy0, gx0) of the plane `in`) that crosses the grid's edge: TMA
// filled the cells outside the grid with zeros; the CTA overwrites exactly
// those cells with their wrapped values: the rows outside the grid in full,
// then the columns outside it in the other rows.  Four loads per thread are
// in flight at a time.  The 2D kernel calls it out of line (inlined, it
// raised the register pressure of the whole kernel); in the 3D kernel, whose
// budget is 64 registers, a call cost more spills than the inlined copy.
template <typename T>
__device__ __forceinline__ void wrap_halo_block_inl(T* buf, int SY, int SX, const T* __restrict__ in, int64_t ldx,
                                                    int ny, int nx, int gy0, int gx0) {
    const int top = min(SY, max(0, -gy0));          // rows [0, top) lie above the grid
    const int bot = max(top, min(SY, ny - gy0));     // rows [bot, SY) lie below it
    const int cl = min(SX, max(0, -gx0));           // columns [0, cl) left of it
    const int cr = max(cl, min(SX, nx - gx0));      // columns [cr, SX) right of it
    const int ncx = cl + (SX - cr);                 // outside columns per inside row
    const int n_rows = (top + (SY - bot)) * SX;     // cells of the outside rows
    const int n_all = n_rows + (bot - top) * ncx;
    const int nthr = blockDim.x * blockDim.y;
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    for (int i0 = tid; i0 < n_all; i0 += 4 * nthr) {
        T v[4];
        int off[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * nthr;
            off[u] = -1;
            v[u] = T(0);
            if (i < n_all) {
                int sy, sx;
                if (i < n_rows) {
                    const int rr = i / SX;
                    sy = rr < top ? rr : bot + (rr - top);
                    sx = i - rr * SX;
                } else {
                    const int j = i - n_rows, rr = j / ncx, c = j - rr * ncx;
                    sy = top + rr;
                    sx = c < cl ? c : cr + (c - cl);
                }
                off[u] = sy * SX + sx;
                v[u] = __ldcg(in + (int64_t)wrap_fast(gy0 + sy, ny) * ldx + wrap_fast(gx0 + sx, nx));
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (off[u] >= 0) buf[off[u]] = v[u];
    }
}

template <typename T>
__device__ __noinline__ void wrap_halo_block(T* buf, int SY, int SX, const T* __restrict__ in, int64_t ldx, int ny,
                                             int nx, int gy0, int gx0) {
    wrap_halo_block_inl<T>(buf, SY, SX, in, ldx, ny, nx, gy0, gx0);
}

// Register budgets of the persistent kernels: left alone, the compiler keeps
// the coefficients and unrolled sums in registers and one CTA fills an SM.
template <typename T, int R, bool STAR, bool MULTI, int TY>
constexpr int ctas2() {
    if (sizeof(T) == 8) return TY == 64 || (STAR && R >= 3) ? 2 : 4;   // (strips of wide stars hold 2r+1 rows in registers)
    return MULTI ? (R == 1 ? 3 : R == 2 ? 2 : 1) : (STAR && R >= 4) ? 2 : 3;
}

template <typename T, int R, bool STAR, bool MULTI, int TY>
__global__ void __launch_bounds__(kBX * Tile2<T>::by(TY), (ctas2<T, R, STAR, MULTI, TY>()))
gather2d_tma_kernel(const __grid_constant__ CUtensorMap tin, const G2Args a, const Coeffs<T, ipow(2 * R + 1, 2)> cf) {
    constexpr int TX = Tile2<T>::TX;
    constexpr int kThr = kBX * Tile2<T>::by(TY);
    extern __shared__ __align__(128) unsigned char smem_dyn[];
    unsigned char* smem_raw = (unsigned char*)(((uintptr_t)smem_dyn + 127) & ~(uintptr_t)127);
    const Layout2<T, TY> L(R, a.tb);
    constexpr int NST = stages2(sizeof(T), MULTI);
    T* const stage0 = reinterpret_cast<T*>(smem_raw + kLeadElems * 4);
    T* work = stage0 + NST * L.buf;
    uint64_t* full = reinterpret_cast<uint64_t*>(stage0 + (size_t)L.buffers(a.tb) * L.buf);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(full + NST);
    volatile int* stage_tile = abort_flag + 1;   // [NST] tile of each stage (-1: no more)
    const int tid = threadIdx.y * kBX + threadIdx.x;
    const T* in = (const T*)a.in;
    T* out = (T*)a.out;
    const uint32_t box_bytes = (uint32_t)(L.SY * L.SX * sizeof(T));
    if (tid == 0) {
        for (int i = 0; i < NST; ++i) ptx::mbar_init(&full[i], 1);
        *abort_flag = 0;
        ptx::fence_mbar_init();
        ptx::prefetch_tensormap(&tin);
    }
    // programmatic dependent launch (common.cuh): a grid with a CTA per tile lets
    // the next sweep set itself up beside it (not FP64: the CTAs that wait crowd
    // on to the free SMs and then share their FP64 pipes: 256^2 r = 1 star 4.8 us
    // per sweep against 2.8); the grids are touched from here on
    if (sizeof(T) == 4 && (int)gridDim.x == a.tiles_total) ptx::launch_dependents();
    ptx::grid_dependency_wait();
    __syncthreads();
    // Every tile is staged by TMA; with a periodic boundary, a tile whose
    // staged block crosses the grid's edge then gets its outside cells wrapped.
    auto edge = [&](int t) {
        if (a.bc != kBcPeriodic) return false;
        const int y0 = (t / a.tiles_x) * TY, x0 = (t % a.tiles_x) * TX;
        return !(y0 - L.H >= 0 && y0 + TY + L.H <= a.ny && x0 - L.HX >= 0 && x0 + TX + L.HX <= a.nx);
    };
    // Thread 0 tracks the ring: bit s of `inflight` = a load into stage s not
    // yet waited for, bit s of `phase` = parity of stage s's next completion.
    // The first NST - 1 tiles of a CTA are fixed; on grids of more tiles the
    // others are claimed one ahead of the stage that comes free, so that the
    // atomic's round trip is never waited for.  SMs do not run equally fast: with
    // fixed shares the CTAs' positions, and so the rows in flight, drift apart
    // (8192^2 r = 1 box 91 us, with claims 79: the copy bandwidth).
    uint32_t inflight = 0, phase = 0;
    int issued = 0, claimed = 0;
    bool more = true;
    auto issue = [&]() {
        if (!more) return;
        const int s = issued % NST;
        const int t = a.sched && issued >= NST - 1 ? (NST - 1) * (int)gridDim.x + claimed
                                                   : (int)blockIdx.x + issued * (int)gridDim.x;
        if (a.sched && issued >= NST - 2 && t < a.tiles_total) claimed = atomicAdd(&a.sched[0], 1);
        ++issued;
        more = t < a.tiles_total;
        stage_tile[s] = more ? t : -1;
        if (!more) {
            ptx::mbar_arrive(&full[s]);
            return;
        }
        const int y0 = (t / a.tiles_x) * TY, x0 = (t % a.tiles_x) * TX;
        ptx::mbar_arrive_expect_tx(&full[s], box_bytes);
        ptx::tma_load_2d(stage0 + s * L.buf, &tin, x0 - L.HX, y0 - L.H, &full[s]);
        inflight |= 1u << s;
    };
    if (tid == 0)
        for (int i = 0; i < NST - 1; ++i) issue();
    for (int k = 0;; ++k) {
        const int s = k % NST;
        T* st_buf = stage0 + s * L.buf;
        // the stage computed at iteration k - 1 is free (barrier at its end);
        // its generic-proxy writes (halo wrap, sub-steps) are ordered
        // before the TMA write that refills it
        if (tid == 0) {
            ptx::fence_proxy_async_smem();
            issue();
        }
        {
            const uint32_t par = (phase >> s) & 1u;   // every thread tracks the parities
            if (!gwait(&full[s], par)) *abort_flag = 1;
            phase ^= 1u << s;
            if (tid == 0) inflight &= ~(1u << s);
        }
        const int t = stage_tile[s];
        if (t < 0) break;
        const int64_t y0 = (int64_t)(t / a.tiles_x) * TY, x0 = (int64_t)(t % a.tiles_x) * TX;
        if (edge(t)) {
            __syncthreads();   // every thread has seen the load land (or the abort)
            if (!*abort_flag)
                wrap_halo_block<T>(st_buf, L.SY, L.SX, in, a.ldx, a.ny, a.nx, (int)y0 - L.H, (int)x0 - L.HX);
        }
        __syncthreads();
        if (*abort_flag) break;
        // sub-steps alternate between the work buffer and the stage
        if constexpr (sizeof(T) == 4) {
            const float* src = st_buf;
            const TileGeom g(R, MULTI ? a.tb : 1, TY, TX);
            if constexpr (MULTI) {
                const int gy0 = (int)y0 - g.H, gx0 = (int)x0 - g.HX;
                const bool zero = a.bc == kBcDirichlet &&
                                  !(gy0 >= 0 && gy0 + g.SY <= a.ny && gx0 >= 0 && gx0 + g.SX <= a.nx);
                for (int st = 1; st < a.tb; ++st) {
                    float* dst = (st & 1) ? work : st_buf;
                    substep_f32<R, STAR, TX>(src, dst, g, st, a.tb, zero, a.ny, a.nx, gy0, gx0, tid, kThr, cf);
                    src = dst;
                    __syncthreads();
                }
            }
            const bool vec = (reinterpret_cast<uintptr_t>(out) & 15u) == 0;   // rows are (TMA)
            last_substep_f32<R, STAR, TY, TX>(src, out, g, vec, a.ny, a.nx, a.ldx, (int)y0, (int)x0, tid, kThr, cf);
            __syncthreads();   // the stage is free
        } else {
            T* src = st_buf;
            for (int st = 1; st <= a.tb; ++st) {
                T* dst = (st & 1) ? work : st_buf;
                substep2<T, R, STAR, TY>(src, dst, out, L, st, st == a.tb, a.ny, a.nx, a.ldx, a.bc, y0, x0, cf);
                src = dst;
                __syncthreads();   // sub-step st is complete (and, after the last, the stage is free)
            }
        }
    }
    if (*abort_flag) {
        // let the loads still in flight land before the CTA gives up its shared memory
        if (tid == 0) {
            for (int s2 = 0; s2 < NST; ++s2)
                if ((inflight >> s2) & 1u) ptx::mbar_wait(&full[s2], (phase >> s2) & 1u, kGatherWait / 8);
            if (a.err) atomicOr(a.err, 2u);
        }
    }
    if (a.sched && tid == 0) {   // this CTA has made its last claim: the last CTA resets the counter
        __threadfence();
        if (atomicAdd(&a.sched[1], 1) == (int)gridDim.x - 1) {
            atomicExch(&a.sched[0], 0);
            atomicExch(&a.sched[1], 0);
        }
    }
}

// 3D streaming kernel: a work unit is a.tzc output planes of a TY x TX column
// (chosen per grid by pick_chunk); its tzc + 2R input planes stream through
// NPL = 2R + 2 plane buffers.
template <typename T>
struct Tile3 {
    static constexpr int TY = 32;
    static constexpr int TX = sizeof(T) == 4 ? 64 : 32;   // FP64: CTAs of half the size, four per SM (as in 2D)
    static constexpr int THREADS = TX * (TY / kRS);       // one strip of kRS rows of one column each
    static constexpr int AL = 16 / (int)sizeof(T);
};

struct G3Args {
    const void* in;
    void* out;
    unsigned int* err;
    int64_t ldx;         // row stride of the grids (elements); planes are ny rows
    int nz, ny, nx, bc;
    int tiles_x, tiles_y, units;
    int tzc;             // output planes per work unit
};

template <typename T, int R>
struct Layout3 {
    static constexpr int NPL = 2 * R + 2;
    static constexpr int HX = round_up(R, Tile3<T>::AL);
    static constexpr int SY = Tile3<T>::TY + 2 * R;
    static constexpr int SX = Tile3<T>::TX + 2 * HX;
    static constexpr int PLANE = round_up(SY * SX, 128 / (int)sizeof(T));
    static constexpr size_t bytes() { return (size_t)NPL * PLANE * sizeof(T) + 8 * NPL + 16 + 128; }
};

template <typename T, int R, bool STAR>
__global__ void __launch_bounds__(Tile3<T>::THREADS, sizeof(T) == 4 ? 4 : (R >= 3 ? 1 : 4))
gather3d_stream_kernel(const __grid_constant__ CUtensorMap tin, const G3Args a, const Coeffs<T, ipow(2 * R + 1, 3)> cf) {
    using L = Layout3<T, R>;
    constexpr int W = 2 * R + 1, TY = Tile3<T>::TY, TX = Tile3<T>::TX, NPL = L::NPL;
    extern __shared__ __align__(128) unsigned char smem_dyn[];
    unsigned char* smem_raw = (unsigned char*)(((uintptr_t)smem_dyn + 127) & ~(uintptr_t)127);
    T* planes = reinterpret_cast<T*>(smem_raw);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem_raw + (size_t)NPL * L::PLANE * sizeof(T));
    volatile int* abort_flag = reinterpret_cast<volatile int*>(full + NPL);
    const int tid = threadIdx.x;
    const T* in = (const T*)a.in;
    T* out = (T*)a.out;
    constexpr uint32_t box_bytes = (uint32_t)(L::SY * L::SX * sizeof(T));
    if (tid == 0) {
        for (int b = 0; b < NPL; ++b) ptx::mbar_init(&full[b], 1);
        *abort_flag = 0;
        ptx::fence_mbar_init();
        ptx::prefetch_tensormap(&tin);
    }
    // No early trigger of the next sweep, as in 2D: its CTAs would crowd on to the
    // SMs with free slots and then share them while others idle (us per sweep
    // with / without, r = 3 box 256^3 568 / 357, r = 1 box 256^3 76 / 54, 64^3 4.3 / 3.9).
    ptx::grid_dependency_wait();
    __syncthreads();
    int uses[NPL];   // TMA loads into each plane buffer so far (mbarrier phases)
#pragma unroll
    for (int b = 0; b < NPL; ++b) uses[b] = 0;
    const int col = tid % TX;            // output column of this thread
    const int sy0 = (tid / TX) * kRS;    // first output row of its strip
    unsigned int in_flight = 0;          // buffers with a TMA load nobody waited for yet (bit mask)
    for (int u = blockIdx.x; u < a.units && !*abort_flag; u += gridDim.x) {
        const int tx_ = u % a.tiles_x, ty_ = (u / a.tiles_x) % a.tiles_y, tz_ = u / (a.tiles_x * a.tiles_y);
        const int x0 = tx_ * TX, y0 = ty_ * TY, z0 = tz_ * a.tzc;
        const int nout = min(a.tzc, a.nz - z0);
        // with a periodic boundary, an edge unit's planes (staged by TMA like
        // the others, from the wrapped plane index) get their cells outside
        // the grid in y and x wrapped once they have landed
        const bool edge = a.bc == kBcPeriodic &&
                          !(y0 - R >= 0 && y0 + TY + R <= a.ny && x0 - L::HX >= 0 && x0 + TX + L::HX <= a.nx);
        // input plane i of the unit is grid plane z0 - R + i, held in buffer i % NPL
        auto load = [&](int i) {
            const int b = i % NPL;
            int gz = z0 - R + i;
            if (a.bc == kBcPeriodic) gz = (int)wrap_index(gz, a.nz);
            if (tid == 0) {
                ptx::fence_proxy_async_smem();   // after the fix-ups of the plane it replaces
                ptx::mbar_arrive_expect_tx(&full[b], box_bytes);
                ptx::tma_load_3d(planes + b * L::PLANE, &tin, x0 - L::HX, y0 - R, gz, &full[b]);
            }
            in_flight |= 1u << b;
        };
        auto ready = [&](int i) {   // input plane i is in its buffer
            const int b = i % NPL;
            if (!gwait(&full[b], (uint32_t)(uses[b] & 1))) *abort_flag = 1;
            ++uses[b];
            in_flight &= ~(1u << b);
        };
        auto wrap_plane = [&](int i) {
            int gz = z0 - R + i;
            gz = (int)wrap_index(gz, a.nz);
            wrap_halo_block_inl<T>(planes + (i % NPL) * L::PLANE, L::SY, L::SX, in + (int64_t)gz * a.ny * a.ldx,
                                   a.ldx, a.ny, a.nx, y0 - R, x0 - L::HX);
        };
        const int nin = nout + 2 * R;
        for (int i = 0; i < NPL && i < nin; ++i) load(i);
        for (int o = 0; o < nout; ++o) {
            const int i_lo = o == 0 ? 0 : o + 2 * R;   // planes that land now
            for (int i = i_lo; i <= o + 2 * R; ++i) ready(i);
            if (edge) {
                __syncthreads();   // every thread has seen the planes land (or the abort)
                if (*abort_flag) break;
                for (int i = i_lo; i <= o + 2 * R; ++i) wrap_plane(i);
            }
            __syncthreads();
            if (*abort_flag) break;
            // output plane z0 + o from input planes o .. o + 2R
            T acc[kRS];
#pragma unroll
            for (int j = 0; j < kRS; ++j) acc[j] = T(0);
            const int sx = L::HX + col;
#pragma unroll
            for (int dz = 0; dz < W; ++dz) {
                const T* pl = planes + ((o + dz) % NPL) * L::PLANE;
                if (STAR && dz != R) {
                    const T w = cf.c[(dz * W + R) * W + R];
#pragma unroll
                    for (int j = 0; j < kRS; ++j) acc[j] = fma(w, pl[(sy0 + R + j) * L::SX + sx], acc[j]);
                } else {
                    const T* base = pl + sy0 * L::SX + (sx - R);
#pragma unroll
                    for (int yi = 0; yi < kRS + 2 * R; ++yi) {
                        T v[W];
#pragma unroll
                        for (int b = 0; b < W; ++b) v[b] = base[yi * L::SX + b];
#pragma unroll
                        for (int j = 0; j < kRS; ++j) {
                            const int a1 = yi - j;
                            if (a1 >= 0 && a1 < W) {
#pragma unroll
                                for (int b = 0; b < W; ++b)
                                    if (!STAR || a1 == R || b == R)
                                        acc[j] = fma(cf.c[(dz * W + a1) * W + b], v[b], acc[j]);
                            }
                        }
                    }
                }
            }
            const int64_t gz = z0 + o, gx = x0 + col;
            if (gx < a.nx) {
#pragma unroll
                for (int j = 0; j < kRS; ++j) {
                    const int64_t gy = y0 + sy0 + j;
                    if (gy < a.ny) out[(gz * a.ny + gy) * a.ldx + gx] = acc[j];
                }
            }
            __syncthreads();   // input plane o is no longer needed: its buffer takes plane o + NPL
            if (o + NPL < nin) load(o + NPL);
        }
        // planes loaded but not needed (short last chunk) are waited for before reuse
        for (int b = 0; b < NPL; ++b)
            if (in_flight & (1u << b)) {
                if (!gwait(&full[b], (uint32_t)(uses[b] & 1))) *abort_flag = 1;
                ++uses[b];
            }
        in_flight = 0;
        __syncthreads();
    }
    if (*abort_flag) {
        if (tid == 0) {
            for (int b = 0; b < NPL; ++b)
                if (in_flight & (1u << b)) ptx::mbar_wait(&full[b], (uint32_t)(uses[b] & 1), kGatherWait / 8);
            if (a.err) atomicOr(a.err, 2u);
        }
    }
}

// Tile shapes.
constexpr int k2BY = 8, k2TX = 128, k2TY = 64;
constexpr int k3BY = 8, k3TX = 32, k3TY = 16, k3TZ = 8;
// Tile shapes of the batched kernel (rows x columns), chosen per batch by the
// autotuner: the single-grid shape, and a smaller one that wastes less of the
// ragged edge tiles of small problems.
constexpr int kBatchShapes = 2;
constexpr int kBatchTY[kBatchShapes] = {64, 32};
constexpr int kBatchTX[kBatchShapes] = {128, 64};
constexpr int kBatchBY[kBatchShapes] = {8, 4};   // FP32: warps per CTA (two and one blocks per thread and sub-step)

// What the deepest tile of a plan may take (a plan is refused beyond it).
template <typename T>
size_t gather_smem_bytes_t(int ndim, int r, int tb) {
    const int H = r * tb;
    const int nb = tb > 1 ? 2 : 1;
    if (ndim == 2) return (size_t)(nb * (k2TY + 2 * H) + kRS) * (k2TX + 2 * H) * sizeof(T);
    return (size_t)(nb * (k3TZ + 2 * H) + kRS) * (k3TY + 2 * H) * (k3TX + 2 * H) * sizeof(T);
}

// Shared memory of an element-loaded 2D tile (FP32: two blocked buffers; FP64:
// the strips' layout).
template <typename T>
size_t tile2_smem_bytes(int r, int tb, int ty, int tx) {
    if (sizeof(T) == 4) return (size_t)(kLeadElems + 2 * TileGeom(r, tb, ty, tx).elems()) * 4;
    const int H = r * tb;
    return (size_t)((tb > 1 ? 2 : 1) * (ty + 2 * H) + kRS) * (tx + 2 * H) * sizeof(T);
}

int max_smem_optin() {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return v;
}

// Let a kernel take as much dynamic shared memory as the device allows.  The
// limit belongs to the kernel, and plans and launches of different depth share
// one: set to what one of them needs, it would fall below what another needs.
template <typename K>
cudaError_t allow_smem(K kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem_optin());
}

template <typename T, int R, bool STAR>
cudaError_t launch2d_tiles(const GatherProblem& p, const void* in, void* out, int tb, cudaStream_t s) {
    constexpr int NC = ipow(2 * R + 1, 2);
    Coeffs<T, NC> cf;
    for (int i = 0; i < NC; ++i) cf.c[i] = (T)p.cg[i];
    const size_t smem = tile2_smem_bytes<T>(R, tb, k2TY, k2TX);
    constexpr bool F32 = sizeof(T) == 4;   // (FP64 tiles compute all columns in 64 bits)
    auto kern = F32 && p.n[1] > INT32_MAX - 512 ? gather2d_kernel<T, R, STAR, k2BY, k2TX, k2TY, F32>
                                                : gather2d_kernel<T, R, STAR, k2BY, k2TX, k2TY, false>;
    cudaError_t e = allow_smem(kern);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)((p.n[1] + k2TX - 1) / k2TX), (unsigned)((p.n[0] + k2TY - 1) / k2TY));
    kern<<<grid, dim3(kBX, k2BY), smem, s>>>((const T*)in, (T*)out, p.n[0], p.n[1], p.ldx, p.bc, tb, cf);
    return cudaGetLastError();
}

template <typename T, int R, bool STAR>
cudaError_t launch3d_tiles(const GatherProblem& p, const void* in, void* out, int tb, cudaStream_t s) {
    constexpr int NC = ipow(2 * R + 1, 3);
    Coeffs<T, NC> cf;
    for (int i = 0; i < NC; ++i) cf.c[i] = (T)p.cg[i];
    const size_t smem = gather_smem_bytes_t<T>(3, R, tb);
    auto kern = gather3d_kernel<T, R, STAR, k3BY, k3TX, k3TY, k3TZ>;
    cudaError_t e = allow_smem(kern);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)((p.n[2] + k3TX - 1) / k3TX), (unsigned)((p.n[1] + k3TY - 1) / k3TY),
              (unsigned)((p.n[0] + k3TZ - 1) / k3TZ));
    kern<<<grid, dim3(kBX, k3BY), smem, s>>>((const T*)in, (T*)out, p.n[0], p.n[1], p.n[2], p.ldx, p.bc, tb, cf);
    return cudaGetLastError();
}

int sm_count() {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v;
}

// TMA tiled view of a C-order grid: dims (innermost first) and element type;
// false when the driver entry point is missing or the encoder rejects it.
template <typename T>
bool encode_grid_map(CUtensorMap* map, const void* base, int rank, const cuuint64_t* dims, int64_t ldx,
                     const cuuint32_t* box) {
    auto enc = mxu::get_encode();
    if (!enc) return false;
    cuuint64_t strides[2];   // rows of ldx elements; planes of dims[1] rows
    strides[0] = (cuuint64_t)ldx * sizeof(T);
    if (rank == 3) strides[1] = strides[0] * dims[1];
    cuuint32_t es[3] = {1, 1, 1};
    return enc(map, sizeof(T) == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT64, rank,
               const_cast<void*>(base), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int smem_limit(const GatherProblem& p) { return p.tuned ? p.tuned->max_smem : max_smem_optin(); }

// The TMA kernels need 16-byte aligned grid bases and rows.
template <typename T>
bool tma_layout_ok(const GatherProblem& p, const void* in) {
    return ((uintptr_t)in & 15u) == 0 && (p.ldx * (int64_t)sizeof(T)) % 16 == 0;
}

// How many CTAs of a TMA kernel fit: from the plan, which asks the runtime once
// (p.prepare, at its creation), or asked now.
template <typename K>
cudaError_t tuned_for(const GatherProblem& p, K kern, int threads, size_t smem, int tb, GatherTuned* t) {
    if (p.tuned && !p.prepare) {
        *t = *p.tuned;
        if (t->per_sm[tb] > 0) return cudaSuccess;
    }
    cudaError_t e = allow_smem(kern);
    if (e != cudaSuccess) return e;
    t->sms = sm_count();
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&t->per_sm[tb], kern, threads, smem);
    if (t->per_sm[tb] < 1) t->per_sm[tb] = 1;
    if (e == cudaSuccess && p.prepare) {
        p.prepare->sms = t->sms;
        p.prepare->per_sm[tb] = t->per_sm[tb];
    }
    return e;
}

template <typename T, int R, bool STAR, int TY>
cudaError_t launch2d_tma(const GatherProblem& p, const void* in, void* out, int tb, cudaStream_t s) {
    const Layout2<T, TY> L(R, tb);
    const size_t smem = L.bytes(tb);
    constexpr int NC = ipow(2 * R + 1, 2);
    Coeffs<T, NC> cf;
    for (int i = 0; i < NC; ++i) cf.c[i] = (T)p.cg[i];
    G2Args a;
    a.in = in;
    a.out = out;
    a.err = p.err;
    a.ldx = p.ldx;
    a.ny = (int)p.n[0];
    a.nx = (int)p.n[1];
    a.bc = p.bc;
    a.tb = tb;
    a.tiles_x = (a.nx + Tile2<T>::TX - 1) / Tile2<T>::TX;
    a.tiles_total = a.tiles_x * ((a.ny + TY - 1) / TY);
    alignas(64) CUtensorMap tin;
    const cuuint64_t dims[2] = {(cuuint64_t)a.nx, (cuuint64_t)a.ny};
    const cuuint32_t box[2] = {(cuuint32_t)L.SX, (cuuint32_t)L.SY};
    if (!encode_grid_map<T>(&tin, in, 2, dims, p.ldx, box)) return cudaErrorInvalidValue;
    constexpr bool F32 = sizeof(T) == 4;
    auto kern = F32 && tb > 1 ? gather2d_tma_kernel<T, R, STAR, F32, TY> : gather2d_tma_kernel<T, R, STAR, false, TY>;
    constexpr int threads = kBX * Tile2<T>::by(TY);
    GatherTuned t;
    cudaError_t e = tuned_for(p, kern, threads, smem, tb, &t);
    if (e != cudaSuccess || p.prepare) return e;
    int grid = t.sms * t.per_sm[tb];
    if (grid > a.tiles_total) grid = a.tiles_total;
    a.sched = sizeof(T) == 4 && grid < a.tiles_total ? p.sched : nullptr;   // FP64: compute-bound, fixed shares do
    return launch_dependent(kern, dim3(grid), dim3(kBX, Tile2<T>::by(TY)), smem, s, tin, a, cf);
}

template <typename T, int R, bool STAR>
cudaError_t launch2d(const GatherProblem& p, const void* in, void* out, int tb, cudaStream_t s) {
    constexpr int TY = Tile2<T>::TY, TYS = Tile2<T>::TYS, TYD = Tile2<T>::TYD, TX = Tile2<T>::TX;
    const Layout2<T, TY> L(R, tb);
    if (!tma_layout_ok<T>(p, in) || L.bytes(tb) > (size_t)smem_limit(p) || L.SX > 256 || L.SY > 256)
        return p.prepare ? cudaSuccess : launch2d_tiles<T, R, STAR>(p, in, out, tb, s);
    const int64_t tiles_x = (p.n[1] + TX - 1) / TX, tiles = ((p.n[0] + TY - 1) / TY) * tiles_x;
    const int sms = p.tuned ? p.tuned->sms : sm_count();
    if (TYD != TY && tb > 1 && (p.n[0] + TYD - 1) / TYD * tiles_x >= 8 * sms) {
        const Layout2<T, TYD> D(R, tb);
        if (D.bytes(tb) <= (size_t)smem_limit(p) / (STAR || R == 4 ? 2 : 1) && D.SY <= 256)
            return launch2d_tma<T, R, STAR, TYD>(p, in, out, tb, s);
    }
    if (TYS != TY && tiles < sms) return launch2d_tma<T, R, STAR, TYS>(p, in, out, tb, s);
    return launch2d_tma<T, R, STAR, TY>(p, in, out, tb, s);
}

template <typename T, int R, bool STAR>
cudaError_t launch3d(const GatherProblem& p, const void* in, void* out, int tb, cudaStream_t s) {
    using L = Layout3<T, R>;
    const size_t smem = L::bytes();
    if (tb != 1 || !tma_layout_ok<T>(p, in) || smem > (size_t)smem_limit(p) || L::SX > 256 || L::SY > 256)
        return p.prepare ? cudaSuccess : launch3d_tiles<T, R, STAR>(p, in, out, tb, s);
    constexpr int NC = ipow(2 * R + 1, 3);
    Coeffs<T, NC> cf;
    for (int i = 0; i < NC; ++i) cf.c[i] = (T)p.cg[i];
    G3Args a;
    a.in = in;
    a.out = out;
    a.err = p.err;
    a.ldx = p.ldx;
    a.nz = (int)p.n[0];
    a.ny = (int)p.n[1];
    a.nx = (int)p.n[2];
    a.bc = p.bc;
    a.tiles_x = (a.nx + Tile3<T>::TX - 1) / Tile3<T>::TX;
    a.tiles_y = (a.ny + Tile3<T>::TY - 1) / Tile3<T>::TY;
    alignas(64) CUtensorMap tin;
    const cuuint64_t dims[3] = {(cuuint64_t)a.nx, (cuuint64_t)a.ny, (cuuint64_t)a.nz};
    const cuuint32_t box[3] = {(cuuint32_t)L::SX, (cuuint32_t)L::SY, 1};
    if (!encode_grid_map<T>(&tin, in, 3, dims, p.ldx, box)) return cudaErrorInvalidValue;
    auto kern = gather3d_stream_kernel<T, R, STAR>;
    GatherTuned t;
    cudaError_t e = tuned_for(p, kern, Tile3<T>::THREADS, smem, 1, &t);
    if (e != cudaSuccess || p.prepare) return e;
    int grid = t.sms * t.per_sm[1];
    // A unit's fixed cost in planes: FP32 units re-read 2R halo planes and wait
    // for the first 2R + 1 to land; FP64 units compute far longer than that per
    // plane, so even shares matter most.  Four FP64 CTAs on an SM run faster when
    // two have nothing left; one alone of two (r >= 3) does not keep the FP64 pipe
    // busy, so there whole waves count (256^3 r = 3 in half waves / whole: star
    // 846 / 681 us per sweep, box 14637 / 11726).
    const int tiles = a.tiles_x * a.tiles_y;
    a.tzc = sizeof(T) == 8 ? pick_chunk(a.nz, tiles, grid, t.per_sm[1] >= 4 ? 2 : 1, 1, 64, 1 << 20)
                           : pick_chunk(a.nz, tiles, grid, 2, 2 * R + 2, 64, 32);
    a.units = tiles * ((a.nz + a.tzc - 1) / a.tzc);
    if (grid > a.units) grid = a.units;
    return launch_dependent(kern, dim3(grid), dim3(Tile3<T>::THREADS), smem, s, tin, a, cf);
}

template <typename T, bool STAR>
cudaError_t dispatch_r(const GatherProblem& p, const void* in, void* out, int tb, cudaStream_t s) {
    if (p.ndim == 2) {
        switch (p.r) {
            case 1: return launch2d<T, 1, STAR>(p, in, out, tb, s);
            case 2: return launch2d<T, 2, STAR>(p, in, out, tb, s);
            case 3: return launch2d<T, 3, STAR>(p, in, out, tb, s);
            case 4: return launch2d<T, 4, STAR>(p, in, out, tb, s);
        }
    } else {
        switch (p.r) {
            case 1: return launch3d<T, 1, STAR>(p, in, out, tb, s);
            case 2: return launch3d<T, 2, STAR>(p, in, out, tb, s);
            case 3: return launch3d<T, 3, STAR>(p, in, out, tb, s);
            case 4: return launch3d<T, 4, STAR>(p, in, out, tb, s);
        }
    }
    return cudaErrorInvalidValue;
}

template <typename T>
size_t batch_smem_bytes_t(int r, int tb, int shape) {
    return tile2_smem_bytes<T>(r, tb, kBatchTY[shape], kBatchTX[shape]);
}

template <typename T, int R, bool STAR, int S>
cudaError_t launch_batch(const BatchProblem* probs, int nprob, int total_tiles, const void* coef, int max_tb,
                         int grid, cudaStream_t s) {
    const size_t smem = batch_smem_bytes_t<T>(R, max_tb, S);
    constexpr int BY = sizeof(T) == 4 ? kBatchBY[S] : k2BY;
    auto kern = gather2d_batch_kernel<T, R, STAR, BY, kBatchTX[S], kBatchTY[S]>;
    cudaError_t e = allow_smem(kern);
    if (e != cudaSuccess) return e;
    if (grid <= 0) {
        int dev = 0, sms = 0, per = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, kBX * BY, smem);
        grid = sms * (per > 0 ? per : 1);
    }
    if (grid > total_tiles) grid = total_tiles;
    if (grid <= 0) return cudaSuccess;
    kern<<<grid, dim3(kBX, BY), smem, s>>>(probs, nprob, total_tiles, (const T*)coef);
    return cudaGetLastError();
}

template <typename T, bool STAR, int S>
cudaError_t dispatch_batch_r(int r, const BatchProblem* probs, int nprob, int total_tiles, const void* coef,
                             int max_tb, int grid, cudaStream_t s) {
    switch (r) {
        case 1: return launch_batch<T, 1, STAR, S>(probs, nprob, total_tiles, coef, max_tb, grid, s);
        case 2: return launch_batch<T, 2, STAR, S>(probs, nprob, total_tiles, coef, max_tb, grid, s);
        case 3: return launch_batch<T, 3, STAR, S>(probs, nprob, total_tiles, coef, max_tb, grid, s);
    }
    return cudaErrorInvalidValue;
}

template <typename T, bool STAR>
cudaError_t dispatch_batch(int r, const BatchProblem* probs, int nprob, int total_tiles, const void* coef,
                           int max_tb, int shape, cudaStream_t s) {
    if (shape == 1) return dispatch_batch_r<T, STAR, 1>(r, probs, nprob, total_tiles, coef, max_tb, 0, s);
    return dispatch_batch_r<T, STAR, 0>(r, probs, nprob, total_tiles, coef, max_tb, 0, s);
}

}  // namespace

cudaError_t gather_batch_sweep(bool f64, bool star, int r, const BatchProblem* d_probs, int nprob, int total_tiles,
                               const void* d_coef, int max_tb, int shape, cudaStream_t s) {
    if (shape < 0 || shape >= kBatchShapes) return cudaErrorInvalidValue;
    if (f64) return star ? dispatch_batch<double, true>(r, d_probs, nprob, total_tiles, d_coef, max_tb, shape, s)
                         : dispatch_batch<double, false>(r, d_probs, nprob, total_tiles, d_coef, max_tb, shape, s);
    return star ? dispatch_batch<float, true>(r, d_probs, nprob, total_tiles, d_coef, max_tb, shape, s)
                : dispatch_batch<float, false>(r, d_probs, nprob, total_tiles, d_coef, max_tb, shape, s);
}

int gather_batch_shapes() { return kBatchShapes; }

void gather_batch_tile_shape(int shape, int* ty, int* tx) {
    *ty = kBatchTY[shape];
    *tx = kBatchTX[shape];
}

size_t gather_batch_smem_bytes(bool f64, int r, int tb, int shape) {
    return f64 ? batch_smem_bytes_t<double>(r, tb, shape) : batch_smem_bytes_t<float>(r, tb, shape);
}

size_t gather_smem_bytes(const GatherProblem& p, int tb) {
    return p.f64 ? gather_smem_bytes_t<double>(p.ndim, p.r, tb) : gather_smem_bytes_t<float>(p.ndim, p.r, tb);
}

cudaError_t gather_prepare(const GatherProblem& p, const void* grid, int tb, GatherTuned* t) {
    t->sms = sm_count();
    t->max_smem = max_smem_optin();
    GatherProblem q = p;
    q.tuned = t;
    q.prepare = t;
    for (int d = 1; d <= tb && d <= kMaxTb; ++d) {
        const cudaError_t e = gather_sweep(q, grid, nullptr, d, nullptr);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t gather_sweep(const GatherProblem& p, const void* in, void* out, int tb, cudaStream_t s) {
    if (p.f64) return p.star ? dispatch_r<double, true>(p, in, out, tb, s) : dispatch_r<double, false>(p, in, out, tb, s);
    return p.star ? dispatch_r<float, true>(p, in, out, tb, s) : dispatch_r<float, false>(p, in, out, tb, s);
}

}  // namespace stx
