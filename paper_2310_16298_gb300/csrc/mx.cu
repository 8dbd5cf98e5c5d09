// Matrixized 2D stencil sweep on the 5th-generation tensor cores (tcgen05).
//
// Scatter-mode formulation (Sec. 3): every coefficient line contributes, to
// an output block, the sum over its input vectors of (input vector) x
// (coefficient vector) outer products -- Eq. (final).  The lines run along
// the contiguous axis x (the orientation of Eq. (to-outer-product-2-star)):
// line a holds row a of C^g, i.e. the weights of input row offset a - r.  For
// an output block of NB = 16 columns starting at X0, line a applied to input
// row y is the product of the row's K window (columns X0-4 .. X0-4+W-1) with
// the line's banded Toeplitz operand
//
//     H_a[k, q] = C^g[a, k - q - 4 + r],
//
// whose columns are the coefficient vectors (windows of a column of C^o,
// Eq. (co)).  One tcgen05.mma (M = 128, N, K = 8 or 16) sums K such outer
// products for 128 rows at once; the accumulators stay in tensor memory.
//
// Row pairs.  The line sum needs, for output row Y, the partials of line a
// at input row Y + a - r: a shift across the accumulator rows (TMEM lanes),
// which only warp shuffles can apply.  To halve those shuffles every TMEM
// lane m holds two input rows, 2m (even) and 2m+1 (odd), side by side along
// K (K = 2W), and the B operand is made of 2r+2 column blocks, block (p, d)
// stacking H_{a0} over H_{a0+1} with a0 = 2d - p + r (lines outside 0..2r
// are zero).  Lane m+d of block (p, d) then holds exactly the contribution
// of its two rows to output row 2m+p, so
//
//     B[2m + p, :] = sum_d D[m + d, block (p, d)],     |d| <= ceil(r/2),
//
// r shuffles per output instead of 2r, and fewer MACs per output than one
// lane per row.
//
// Tiles are handed out at run time (an atomic counter per plan, reset by the
// last CTA to finish), so SMs that run faster take more tiles.
//
// Boundaries: rows and columns outside the grid are TMA's out-of-bounds zero
// fill (the zero Dirichlet halo).  With a periodic boundary, or when a sweep
// advances several steps (R is then the order of the composed stencil), the
// points near the faces are boundary strips, computed beside the tiles; on
// small, short or narrow grids (sweep_kind) and in plain precisions the
// periodic boundary's wrapped terms are added afterwards by the edge kernel
// (edges.cu).
//
// Roles (one persistent CTA per SM, warp specialised):
//  * warp 0: TMA producer.  A tile is 4 lane quarters x 64 input rows; each
//    quarter is loaded as two 32-row boxes through row-parity tensor maps
//    (even rows, odd rows), so a warp reads consecutive rows (no bank
//    conflicts) and every lane's two rows sit in the same smem slot.
//  * warps 1 and 18: MMA issuers (one thread each), alternating items.  A
//    thread issuing tcgen05.mma is held at the tensor pipe's rate, so with
//    one issuer the pipe drains while that thread waits on the next item's
//    barriers; with two, one issuer's waits overlap the other's MMAs.
//  * warps 2..9: split warps, one per (quarter, row parity): input rows ->
//    TF32 hi/lo (or BF16 parts) -> tensor memory (tcgen05.st).
//  * warps 10..17: epilogue warps, one per (quarter, output parity): tensor
//    memory -> shuffles -> swizzled smem -> TMA store through the output
//    row-parity tensor map.
//  * warp 19: boundary strips, straight from and to global memory.
// Two or three accumulator sets and A stages (as many as tensor memory
// holds) overlap split, MMA and epilogue; every wait is bounded
// (a timeout sets a host-visible error word, drains copies in flight and
// frees tensor memory).  Every CTA loads the banded operands from one of
// several identical copies, so the CTAs starting together do not all read
// the same L2 lines.
//
// Precision: TF32, TF32x3, BF16, BF16x2, BF16x3 (operand parts products
// accumulated smallest first in FP32; the epilogue sums the blocks in FP32
// round-to-nearest).
#include <cuda.h>
#include <cudaTypedefs.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "mx.h"
#include "mxutil.cuh"
#include "plan.h"
#include "ptx.cuh"

namespace stx {

namespace {

using namespace mxu;

constexpr int kPad = 4;                 // input columns left of the output block
constexpr int kLanes = 32;              // TMEM lanes per warp (lane quarter)
constexpr int kQuarters = 4;
constexpr int kNb = 16;                 // output columns per MMA item
constexpr int kItems = 2;               // items (16-column blocks) per tile
constexpr int kTw = kItems * kNb;       // output columns per tile
constexpr int kSplitWarps = 2 * kQuarters;   // (quarter, input row parity)
constexpr int kEpiWarps = 2 * kQuarters;     // (quarter, output row parity)
constexpr int kMma2Warp = 2 + kSplitWarps + kEpiWarps;   // second MMA issuer
constexpr int kStripWarp = kMma2Warp + 1;                // boundary strips
constexpr int kThreads = 32 * (kStripWarp + 1);
constexpr int kMaxDepth = 4;            // time steps one sweep can advance
constexpr int kStripMin = 96;           // smallest extent of a grid whose sweeps may have boundary strips
constexpr int kStripCols = 4;           // columns of the left strip: one 16-byte group
constexpr int kStripRow = 12;           // floats per row of a strip weight table (2R+1 weights, 16-byte rows)
constexpr int kBopCopies = 16;          // most copies of the banded operands in global memory
constexpr int kCtasPerCopy = 10;        // CTAs that read one copy when a sweep starts
constexpr size_t kMostOperands = (size_t)1 << 20;   // bytes of a plan's operands (what a server charges for them)
constexpr int kMaxRawStages = 6;
constexpr int kTileRing = 8;            // tile ids handed from the producer to the epilogue
constexpr int kTmemCols = 512;
constexpr int kSmemBudget = 227 * 1024;

__host__ __device__ constexpr int cmin(int a, int b) { return a < b ? a : b; }

// Row-pair geometry of order R.
template <int R>
struct Pair {
    static constexpr int DM = (R + 1) / 2;              // lanes an output row reaches on either side
    static constexpr int LANES_OUT = kLanes - 2 * DM;   // lanes of a quarter that produce outputs
    static constexpr int ROWS_OUT = 2 * LANES_OUT;      // output rows per quarter
    static constexpr int NBP = R + 1;                   // blocks per output parity
    static constexpr int NBLK = 2 * NBP;
    // lane offset d of block (p, i) is dlo(p) + i
    __host__ __device__ static constexpr int dlo(int p) { return -((R + 1 - p) / 2); }
    // Place of block (p, i) along N.  Two blocks hold one line only (a line past
    // either end stands where their other one would): (e, R) uses even input
    // rows only, (1 - e, 0) odd rows only, e = R mod 2.  The first comes first
    // and the second last, so that each row parity's MMAs run on the NBLK - 1
    // adjacent blocks that use it (issue_pair_products).
    __host__ __device__ static constexpr int pos(int p, int i) {
        return p == R % 2 && i == R          ? 0
               : p != R % 2 && i == 0        ? NBLK - 1
               : R % 2 == 0 ? (p == 0 ? 1 + i : R + i)
                            : (p == 0 ? i : R + 1 + i);
    }
};

template <bool BF>
__host__ __device__ constexpr int window(int nb) { return BF ? OpFmt<true>::window(nb) : OpFmt<false>::window(nb); }

// Shared-memory row pitch of the raw tile: the window widened to an odd
// number of 16-byte chunks (eight consecutive rows = eight bank groups).
__host__ __device__ constexpr int raw_pitch(int w) { return ((w / 4) & 1) ? w : w + 4; }
// Raw tile row: the windows of all items of a tile (item j starts 16 j columns in).
template <bool BF>
__host__ __device__ constexpr int raw_row(int nb) { return nb * (kItems - 1) + window<BF>(nb); }
template <bool BF>
__host__ __device__ constexpr int raw_stage_bytes() { return 2 * kQuarters * kLanes * raw_pitch(raw_row<BF>(kNb)) * 4; }

// Output staging: one buffer per epilogue warp of (32 - 2 DM) rows x kTw floats
// (both items of a tile, written with one TMA store).
__host__ __device__ constexpr int out_warp_bytes() { return 32 * kTw * 4; }
__host__ __device__ constexpr int out_bytes() { return kEpiWarps * out_warp_bytes(); }

template <int R, bool BF>
__host__ __device__ constexpr int bop_bytes() {
    return (BF ? 3 * 2 : 2 * 4) * 2 * window<BF>(kNb) * Pair<R>::NBLK * kNb;
}
template <int R, bool BF>
__host__ __device__ constexpr int smem_fixed() {
    return 1024 /*align slack*/ + out_bytes() + bop_bytes<R, BF>() + 8 * (2 * kMaxRawStages + 16) +
           8 * 2 * kTileRing + 4 * (kTileRing + kMaxRawStages + 8);
}
template <int R, bool BF>
__host__ __device__ constexpr int raw_stages() {
    return cmin(kMaxRawStages, (kSmemBudget - smem_fixed<R, BF>()) / raw_stage_bytes<BF>());
}
template <int R, bool BF>
__host__ __device__ constexpr int smem_bytes() {
    return smem_fixed<R, BF>() + raw_stages<R, BF>() * raw_stage_bytes<BF>();
}

struct MxArgs2D {
    const void* bops;          // block operands [part][kchunk][block*16 + q][16 bytes]
    unsigned int* err;         // device error word (host-mapped)
    int* sched;                // [0] tiles handed out beyond the first gridDim.x, [1] CTAs finished (0 between launches)
    int ny, nx;
    int64_t ldx;               // row stride of the grids (elements)
    int nparts;                // operand parts of the input split (1..3)
    int tiles_x, tiles_total;
    int x0, y0, x1, y1;        // grid region the tiles write: rows y0.., columns x0..; the rest are strips
    int rows_even, rows_odd;   // that region's rows of the even / odd row-parity views
    int bc;
    int strip_classes;         // weight classes per axis of the strips (0: no strips)
    const float* strip_w;      // strip weights [y class][x class][2R+1][kStripRow]
    const float* in;
    float* out;
    int bop_copies;
    uint32_t bop_bytes;        // every part
    uint32_t bpart_bytes;      // one part
    int nprod;                 // products per K step (1, 3 or 6)
};

// Tensor-memory stage counts for A operands of a_cols columns and
// accumulator sets of n columns: as many A stages as fit (up to 4) beside two
// accumulator sets, then as many accumulator sets as fit beside those.
__host__ __device__ constexpr int a_stages(int a_cols, int n) {
    return (4 * a_cols + 2 * n <= kTmemCols) ? 4 : (3 * a_cols + 2 * n <= kTmemCols) ? 3 : 2;
}
__host__ __device__ constexpr int d_sets(int a_cols, int n) {
    return (a_stages(a_cols, n) * a_cols + 4 * n <= kTmemCols)   ? 4
           : (a_stages(a_cols, n) * a_cols + 3 * n <= kTmemCols) ? 3
                                                                 : 2;
}

// Boundary strips.  The points within a few rows or columns of a face are not
// a convolution with one set of weights: with a zero halo, a sweep of k > 1
// steps resets the points outside the grid after every step, so the weights
// depend on the distance to the faces; with a periodic boundary the neighbours
// wrap, which the tiles' TMA loads (zeros outside the grid) do not.  One warp
// per CTA computes them from global memory in FP32 beside the tiles: an item
// is four adjacent columns of one row, the weights come from a table by the
// point's distance class in y and x (one class when periodic).  The tiles
// write only the rest of the grid, so the two need no order between them.
// 8192^2, order 4: 32 thousand items over 152 warps cost 5 us of a 130 us
// sweep (issue slots and the load/store pipe shared with the tiles' warps); a
// second kernel over the strips cost 20.  Data comes through L2 (__ldcg): the
// buffer was the output of an earlier sweep of the same stream.
__device__ __forceinline__ int strip_class(int i, int n, int s) {
    return i < s ? i : (n - 1 - i < s ? 2 * s - (n - 1 - i) : s);
}

template <int R>
__device__ __forceinline__ void boundary_strips(const MxArgs2D& a, int first, int stride) {
    constexpr int W = 2 * R + 1;
    constexpr int RB = 3;                     // input rows loaded before the first is used
    const int groups = (a.nx + 3) >> 2;       // column groups per row
    const int xg = a.x1 >> 2;                 // first group right of the tiles' region
    const int left = a.x0 >> 2;               // groups left of the tiles' region
    const int side = left + groups - xg;      // strip groups of a row beside it
    const int mid = a.y1 - a.y0;
    const int full = (a.y0 + a.ny - a.y1) * groups;   // items of whole rows
    const int total = full + mid * side;
    const int s = a.strip_classes >> 1;
    const bool periodic = a.bc == kBcPeriodic;
    for (int item = first; item < total; item += stride) {
        int y, g;
        if (item < full) {
            const int f = item / groups;
            g = item - f * groups;
            y = f < a.y0 ? f : a.y1 + (f - a.y0);
        } else {   // consecutive lanes: consecutive rows of one group
            const int j = item - full, c = j / mid;
            y = a.y0 + j - c * mid;
            g = c < left ? c : xg + c - left;
        }
        const float* wy = a.strip_w + (size_t)strip_class(y, a.ny, s) * a.strip_classes * (W * kStripRow);
        int cx[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) cx[q] = strip_class(min(4 * g + q, a.nx - 1), a.nx, s);
        float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        // Input columns 4 g - 4 .. 4 g + 7: three groups, each wholly inside the
        // grid or wholly outside it (then wrapped, or zero), unless the extent is
        // no multiple of 4 and the item lies at an x face: then column by column.
        // Predicated loads without branches, so that a chunk's are all in flight:
        // with a branch per group the strips outlasted the tiles (8192^2 order 4
        // periodic 135 us, now 130; 128^2 r = 1 2.5 us per step, now 2.2).
        const bool whole = a.nx % 4 == 0 || (g > 0 && 4 * g + 8 <= a.nx);
        for (int d0 = 0; d0 < W; d0 += RB) {
            float v[RB][12];   // v[b][k] = column 4 g - 4 + k of row y - R + d0 + b
#pragma unroll
            for (int b = 0; b < RB; ++b) {
                int yy = y - R + d0 + b;
                const bool wrap_y = yy < 0 || yy >= a.ny;
                const bool use = d0 + b < W && (periodic || !wrap_y);
                if (wrap_y) yy += yy < 0 ? a.ny : -a.ny;
                const float* row = a.in + (int64_t)yy * a.ldx;
                if (whole) {
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        int x = 4 * (g - 1 + k);
                        const bool in = x >= 0 && x < a.nx;
                        x += in ? 0 : x < 0 ? a.nx : -a.nx;
                        float4 u = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                        if (use && (in || periodic)) u = __ldcg(reinterpret_cast<const float4*>(row + x));
                        v[b][4 * k] = u.x;
                        v[b][4 * k + 1] = u.y;
                        v[b][4 * k + 2] = u.z;
                        v[b][4 * k + 3] = u.w;
                    }
                } else {
#pragma unroll
                    for (int k = 0; k < 12; ++k) {
                        int x = 4 * g - 4 + k;
                        const bool in = x >= 0 && x < a.nx;
                        x += in ? 0 : x < 0 ? a.nx : -a.nx;
                        v[b][k] = 0.0f;
                        if (use && (in || periodic)) v[b][k] = __ldcg(row + x);
                    }
                }
            }
#pragma unroll
            for (int b = 0; b < RB; ++b) {
                if (d0 + b >= W) break;
                float w[kStripRow];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (q == 0 || cx[q] != cx[q - 1]) {
                        const float* wr = wy + ((size_t)cx[q] * W + d0 + b) * kStripRow;
#pragma unroll
                        for (int c = 0; c < (W + 3) / 4; ++c) {
                            const float4 u = __ldg(reinterpret_cast<const float4*>(wr) + c);
                            w[4 * c] = u.x;
                            w[4 * c + 1] = u.y;
                            w[4 * c + 2] = u.z;
                            w[4 * c + 3] = u.w;
                        }
                    }
#pragma unroll
                    for (int c = 0; c < W; ++c) acc[q] = fmaf(w[c], v[b][4 + q + c - R], acc[q]);
                }
            }
        }
        float* o = a.out + (int64_t)y * a.ldx + 4 * g;
        if (4 * g + 3 < a.nx) {
            *reinterpret_cast<float4*>(o) = make_float4(acc[0], acc[1], acc[2], acc[3]);
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (4 * g + q < a.nx) o[q] = acc[q];
        }
    }
}

// The products of one item (as issue_products), each row parity's K steps on
// the blocks that use it: N - 16 of the N columns, the even rows' from block 0
// and the odd rows' from block 1 (the first MMA runs on all, to clear them).
// The columns left out would add zeros.  8192^2 TF32x3, us per sweep with all
// columns / without: order 4 128 / 124, order 3 112 / 110.
template <bool BF, int KS, int N, int PA, int PB, bool FIRST>
__device__ __forceinline__ void issue_pair_product(uint32_t d, uint32_t a_base, int part_cols, uint64_t b_desc0,
                                                   uint32_t bpart_bytes) {
    constexpr uint32_t F = OpFmt<BF>::kFmt;
    constexpr uint32_t all = ptx::instr_desc(F, F, 128, (uint32_t)N);
    constexpr uint32_t most = ptx::instr_desc(F, F, 128, (uint32_t)(N - kNb));
    const uint32_t a = a_base + (uint32_t)(PA * part_cols);
    const uint64_t b = b_desc0 + (uint64_t)((PB * bpart_bytes) >> 4);
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
        const uint64_t bd = b + (uint64_t)((2 * ks * N * 16) >> 4);
        if (FIRST && ks == 0)
            ptx::mma_ts<BF, true>(d, a + 8 * ks, bd, all);
        else if (ks < KS / 2)
            ptx::mma_ts<BF, false>(d, a + 8 * ks, bd, most);
        else
            ptx::mma_ts<BF, false>(d + kNb, a + 8 * ks, bd + kNb, most);   // 16 rows of 16 bytes on
    }
}

template <bool BF, int KS, int N>
__device__ __forceinline__ void issue_pair_products(uint32_t d, uint32_t a, int pc, uint64_t b0, uint32_t bpb, int nprod) {
    switch (nprod) {
        case 1:
            issue_pair_product<BF, KS, N, 0, 0, true>(d, a, pc, b0, bpb);
            break;
        case 2:
            issue_pair_product<BF, KS, N, 0, 1, true>(d, a, pc, b0, bpb);
            issue_pair_product<BF, KS, N, 0, 0, false>(d, a, pc, b0, bpb);
            break;
        case 3:
            issue_pair_product<BF, KS, N, 1, 0, true>(d, a, pc, b0, bpb);
            issue_pair_product<BF, KS, N, 0, 1, false>(d, a, pc, b0, bpb);
            issue_pair_product<BF, KS, N, 0, 0, false>(d, a, pc, b0, bpb);
            break;
        case 6:
            issue_pair_product<BF, KS, N, 0, 2, true>(d, a, pc, b0, bpb);
            issue_pair_product<BF, KS, N, 1, 1, false>(d, a, pc, b0, bpb);
            issue_pair_product<BF, KS, N, 2, 0, false>(d, a, pc, b0, bpb);
            issue_pair_product<BF, KS, N, 1, 0, false>(d, a, pc, b0, bpb);
            issue_pair_product<BF, KS, N, 0, 1, false>(d, a, pc, b0, bpb);
            issue_pair_product<BF, KS, N, 0, 0, false>(d, a, pc, b0, bpb);
            break;
    }
}

template <int R, bool BF, int NP>
__global__ void __launch_bounds__(kThreads, 1)
mx2d_kernel(const __grid_constant__ CUtensorMap tmap_e, const __grid_constant__ CUtensorMap tmap_o,
            const __grid_constant__ CUtensorMap omap_e, const __grid_constant__ CUtensorMap omap_o,
            const MxArgs2D args) {
    using F = OpFmt<BF>;
    using G = Pair<R>;
    constexpr int N = G::NBLK * kNb;        // MMA N
    constexpr int W = window<BF>(kNb);      // K window of one input row
    constexpr int KW = 2 * W;               // K: even-row window | odd-row window
    constexpr int KS = KW / F::kKStep;      // MMAs per product
    constexpr int PC = F::part_cols(KW);    // TMEM columns of one operand part
    constexpr int A_COLS = NP * PC;         // NP operand parts (1..3) per A stage
    constexpr int GW = F::kGroup;           // input columns per split group
    constexpr int NG = W / GW;              // split groups per row
    constexpr int KP = raw_pitch(raw_row<BF>(kNb));
    constexpr int SLAB = kLanes * KP * 4;   // one (parity, quarter) box
    constexpr int RSB = raw_stage_bytes<BF>();
    constexpr int kRawStages = raw_stages<R, BF>();
    constexpr int OWB = out_warp_bytes();
    // A stages hide the split -> MMA -> completion -> split round trip,
    // accumulator sets the MMA -> epilogue -> MMA one
    constexpr int AST = a_stages(A_COLS, N);
    constexpr int DST = d_sets(A_COLS, N);
    static_assert(kRawStages * kItems >= 4, "TMA ring too shallow");
    static_assert(N % 16 == 0 && N <= 256, "MMA N");
    static_assert(2 * A_COLS + 2 * N <= kTmemCols, "TMEM budget");
    static_assert(AST * A_COLS + DST * N <= kTmemCols, "TMEM budget");
    static_assert(2 * kRawStages + 2 * AST + 2 * DST + 1 <= 2 * kMaxRawStages + 15, "barrier space");
    static_assert(G::LANES_OUT * kTw * 4 <= OWB && kTw * 4 == 128, "output staging (128-byte swizzle rows)");

    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* outs = smem;                     // [epilogue warp] output buffers (1 KB aligned)
    unsigned char* raw = outs + out_bytes();        // [stage][parity][quarter] 32-row boxes
    unsigned char* bops = raw + kRawStages * RSB;
    uint64_t* bars = (uint64_t*)(bops + args.bop_bytes);
    uint64_t* full = bars;                          // [kRawStages] TMA landed
    uint64_t* rawfree = bars + kRawStages;          // [kRawStages] rows read by the split warps
    uint64_t* afull = bars + 2 * kRawStages;        // [AST] A operand stage written to TMEM
    uint64_t* aempty = afull + AST;                 // [AST] MMAs done reading the A stage
    uint64_t* accf = aempty + AST;                  // [DST] accumulator set ready
    uint64_t* acce = accf + DST;                    // [DST] accumulator set drained
    uint64_t* bop_bar = acce + DST;
    uint64_t* tq_full = bop_bar + 1;                // [kTileRing] tile id written
    uint64_t* tq_empty = tq_full + kTileRing;       // [kTileRing] tile id read by the epilogue warps
    uint32_t* tmem_slot = (uint32_t*)(tq_empty + kTileRing);
    volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
    volatile int* tile_ring = abort_flag + 1;       // [kTileRing] tile ids (-1: no more tiles)
    volatile int* stage_tile = tile_ring + kTileRing;   // [kRawStages] tile of each input stage
    volatile int* a_tile = stage_tile + kMaxRawStages;  // [AST] tile of each A stage (-1: end)

    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;

    if (tid == 0) {
        for (int s = 0; s < kRawStages; ++s) {
            ptx::mbar_init(&full[s], 1);
            ptx::mbar_init(&rawfree[s], kSplitWarps);
        }
        for (int a = 0; a < AST; ++a) {
            ptx::mbar_init(&afull[a], kSplitWarps);
            ptx::mbar_init(&aempty[a], 1);
        }
        for (int a = 0; a < DST; ++a) {
            ptx::mbar_init(&accf[a], 1);
            ptx::mbar_init(&acce[a], kEpiWarps);
        }
        ptx::mbar_init(bop_bar, 1);
        for (int k = 0; k < kTileRing; ++k) {
            ptx::mbar_init(&tq_full[k], 1);
            ptx::mbar_init(&tq_empty[k], kEpiWarps);
        }
        *abort_flag = 0;
        ptx::fence_mbar_init();
    }
    const bool claims = (int)gridDim.x < args.tiles_total;   // more tiles than CTAs
    // A small grid lets the stream's next kernel start at once: on the SMs that
    // this one leaves free its CTAs set themselves up and wait.
    if (!claims && tid == 32 * kStripWarp) ptx::launch_dependents();
    if (warp == 1) {
        ptx::tmem_alloc(tmem_slot, kTmemCols);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const uint32_t tmem_a = tmem;                             // A stages: [AST][parts]
    const uint32_t tmem_d = tmem + (uint32_t)(AST * A_COLS);  // accumulator sets: [DST][N]
    int issued = 0;        // producer: TMA tiles issued
    int committed = -1;    // MMA issuer: last tile whose MMAs were committed

    if (warp == 0) {
        // ------------------------------------------------ TMA producer
        if (lane == 0) {
            ptx::mbar_arrive_expect_tx(bop_bar, args.bop_bytes);
            ptx::bulk_load(bops, (const unsigned char*)args.bops + (size_t)(blockIdx.x % args.bop_copies) * args.bop_bytes,
                           args.bop_bytes, bop_bar);
            ptx::prefetch_tensormap(&tmap_e);
            ptx::prefetch_tensormap(&tmap_o);
            ptx::prefetch_tensormap(&omap_e);
            ptx::prefetch_tensormap(&omap_o);
            // Launched as a programmatic dependent of the stream's previous
            // kernel (the previous sweep, or its boundary-strip kernel): the
            // set-up above (barriers, tensor memory, banded operands) overlapped
            // its tail; the grids and the tile counter are touched only from here.
            ptx::grid_dependency_wait();
            // A CTA's first tile is its index: no claim to wait for, and none at
            // all on a grid with a CTA per tile.
            for (int i = 0;; ++i) {
                const int s = i % kRawStages;
                const uint32_t ph = (uint32_t)(i / kRawStages) & 1u;
                const int tq = i % kTileRing;
                if (!wait_or_abort(&rawfree[s], ph ^ 1u, abort_flag) ||
                    !wait_or_abort(&tq_empty[tq], ((uint32_t)(i / kTileRing) & 1u) ^ 1u, abort_flag))
                    break;
                int t = blockIdx.x;
                if (i > 0) t = claims ? (int)gridDim.x + atomicAdd(&args.sched[0], 1) : args.tiles_total;
                if (t >= args.tiles_total) t = -1;
                stage_tile[s] = t;
                tile_ring[tq] = t;
                ptx::mbar_arrive(&tq_full[tq]);
                if (t < 0) {   // no more tiles: the split warps see the end through the stage
                    ptx::mbar_arrive(&full[s]);
                    break;
                }
                const int X0 = args.x0 + (t % args.tiles_x) * kTw;
                const int Y0 = args.y0 + (t / args.tiles_x) * (kQuarters * G::ROWS_OUT);
                unsigned char* dst = raw + s * RSB;
                ptx::mbar_arrive_expect_tx(&full[s], (uint32_t)RSB);
#pragma unroll
                for (int q = 0; q < kQuarters; ++q) {
                    // quarter q covers input rows Y0 + q*ROWS_OUT - 2*DM + [0, 64): an even start
                    const int yp = (Y0 + q * G::ROWS_OUT - 2 * G::DM) / 2;   // row in the parity views
                    ptx::tma_load_2d(dst + q * SLAB, &tmap_e, X0 - kPad, yp, &full[s]);
                    ptx::tma_load_2d(dst + (kQuarters + q) * SLAB, &tmap_o, X0 - kPad, yp, &full[s]);
                }
                issued = i + 1;
            }
        }
    } else if (warp == 1 || warp == kMma2Warp) {
        // ------------------------------------------------ MMA issuers (items i with i % 2 == u)
        const int u = warp == 1 ? 0 : 1;
        if (lane == 0 && wait_or_abort(bop_bar, 0, abort_flag)) {
            const uint64_t b0 = ptx::smem_desc(ptx::smem_u32(bops), (uint32_t)(N * 16), 128);
            const int pr = args.nprod;
            for (int i = u;; i += 2) {
                const int sa = i % AST;
                const uint32_t pa = (uint32_t)(i / AST) & 1u;
                const int st = i % DST;
                const uint32_t ph = (uint32_t)(i / DST) & 1u;
                if (!wait_or_abort(&afull[sa], pa, abort_flag)) break;
                if (a_tile[sa] < 0) break;   // the split warps passed the end of the tiles
                if (!wait_or_abort(&acce[st], ph ^ 1u, abort_flag)) break;
                ptx::tc_fence_after();
                issue_pair_products<BF, KS, N>(tmem_d + (uint32_t)(st * N), tmem_a + (uint32_t)(sa * A_COLS), PC, b0,
                                               args.bpart_bytes, pr);
                ptx::mma_commit(&aempty[sa]);
                ptx::mma_commit(&accf[st]);
                committed = i;
            }
        }
    } else if (warp < 2 + kSplitWarps) {
        // ------------------------------------------------ split: rows (smem) -> operand parts (TMEM)
        const int q = warp & 3;                        // TMEM lane quarter of this warp
        const int e = (warp - 2) >> 2;                 // input row parity this warp converts
        const uint32_t lane_off = (uint32_t)(q * 32) << 16;
        int i = 0;   // items
        bool ok = true;
        for (int k = 0; ok; ++k) {
            const int rs = k % kRawStages;
            const uint32_t rph = (uint32_t)(k / kRawStages) & 1u;
            if (!wait_or_abort(&full[rs], rph, abort_flag)) break;
            const int t = stage_tile[rs];
            if (t < 0) {
                // End of the tiles: one end marker per MMA issuer through the
                // next two A stages (the issuers take alternate items).
                for (int e2 = 0; e2 < 2; ++e2, ++i) {
                    const int sa = i % AST;
                    if (!wait_or_abort(&aempty[sa], ((uint32_t)(i / AST) & 1u) ^ 1u, abort_flag)) break;
                    if (warp == 2 && lane == 0) a_tile[sa] = -1;
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(&afull[sa]);
                }
                break;
            }
            const float* row =
                reinterpret_cast<const float*>(raw + rs * RSB + (e * kQuarters + q) * SLAB) + (size_t)lane * KP;
            for (int j = 0; j < kItems; ++j, ++i) {
                const int sa = i % AST;
                const uint32_t pa = (uint32_t)(i / AST) & 1u;
                float x[NG][GW];
#pragma unroll
                for (int g = 0; g < NG; ++g) {
#pragma unroll
                    for (int c4 = 0; c4 < GW; c4 += 4) {
                        const float4 v = *reinterpret_cast<const float4*>(row + kNb * j + GW * g + c4);
                        x[g][c4] = v.x;
                        x[g][c4 + 1] = v.y;
                        x[g][c4 + 2] = v.z;
                        x[g][c4 + 3] = v.w;
                    }
                }
                if (j == kItems - 1) {   // every item's rows are in registers: the stage goes back
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(&rawfree[rs]);
                }
                if (!wait_or_abort(&aempty[sa], pa ^ 1u, abort_flag)) {
                    ok = false;
                    break;
                }
                ptx::tc_fence_after();
                const uint32_t abase = tmem_a + lane_off + (uint32_t)(sa * A_COLS);
                split_store_groups<BF, NP, NG>(x, abase, PC, e * W, GW);
                ptx::tc_fence_before();
                if (warp == 2 && lane == 0) a_tile[sa] = t;
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(&afull[sa]);
            }
        }
    } else if (warp == kStripWarp) {
        // ------------------------------------------------ boundary strips (straight from and to global memory)
        if (args.strip_classes > 0) {
            // bring the weights (at most 21 KB) into L1 while the previous kernel
            // drains: read cold, row by row, they were most of a small grid's sweep
            constexpr int kTable = (2 * R + 1) * kStripRow;
            for (int o = lane * 32; o < args.strip_classes * args.strip_classes * kTable; o += 32 * 32)
                ptx::prefetch_l1(args.strip_w + o);
            ptx::grid_dependency_wait();
            boundary_strips<R>(args, blockIdx.x * 32 + lane, gridDim.x * 32);
        }
    } else {
        // ------------------------------------------------ epilogue: accumulators -> outputs (warps 10..17)
        const int q = warp & 3;
        const int p = (warp - 2 - kSplitWarps) >> 2;   // output row parity of this warp
        const uint32_t lane_off = (uint32_t)(q * 32) << 16;
        unsigned char* ost = outs + (warp - 2 - kSplitWarps) * OWB;
        auto drain = [&](auto pc) {
            constexpr int P = decltype(pc)::value;
            constexpr int DLO = G::dlo(P);
            constexpr int I0 = -DLO;                          // the block with lane offset 0
            constexpr int LB = G::NBP <= 3 ? G::NBP : 2;      // blocks per TMEM load batch
            const CUtensorMap* omap = P ? &omap_o : &omap_e;
            const int prows = P ? args.rows_odd : args.rows_even;
            int i = 0;
            bool ok = true;
            for (int k = 0; ok; ++k) {
            const int tq = k % kTileRing;
            if (!wait_or_abort(&tq_full[tq], (uint32_t)(k / kTileRing) & 1u, abort_flag)) break;
            const int t = tile_ring[tq];
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&tq_empty[tq]);
            if (t < 0) break;
            for (int j = 0; j < kItems; ++j, ++i) {
                const int st = i % DST;
                const uint32_t ph = (uint32_t)(i / DST) & 1u;
                if (!wait_or_abort(&accf[st], ph, abort_flag)) {
                    ok = false;
                    break;
                }
                ptx::tc_fence_after();
                const int X0 = (t % args.tiles_x) * kTw;   // in the tiles' region
                const int Y0 = (t / args.tiles_x) * (kQuarters * G::ROWS_OUT);
                const uint32_t dbase = tmem_d + lane_off + (uint32_t)(st * N);
                auto block = [&](int i) { return dbase + (uint32_t)(G::pos(P, i) * kNb); };
                float acc[kNb];
#pragma unroll
                for (int b0 = 0; b0 < G::NBP; b0 += LB) {
                    // Blocks b0 .. b0 + nv - 1 into v (and, with the first batch,
                    // block I0 into v0 when it lies in a later batch), loaded and
                    // waited for in one step.
                    uint32_t v[LB][kNb];
                    uint32_t v0[kNb];
                    const int nv = G::NBP - b0 < LB ? G::NBP - b0 : LB;
                    if (b0 == 0 && I0 >= LB) {
                        if (nv == 2) ptx::tmem_ld_x16_sync(block(0), v[0], block(1), v[1], block(I0), v0);
                        if (nv == 1) ptx::tmem_ld_x16_sync(block(0), v[0], block(I0), v0);
                    } else {
                        if constexpr (LB >= 3) {
                            if (nv == 3) ptx::tmem_ld_x16_sync(block(b0), v[0], block(b0 + 1), v[1], block(b0 + 2), v[2]);
                        }
                        if (nv == 2) ptx::tmem_ld_x16_sync(block(b0), v[0], block(b0 + 1), v[1]);
                        if (nv == 1) ptx::tmem_ld_x16_sync(block(b0), v[0]);
                    }
                    if (b0 + LB >= G::NBP) {   // last batch: the accumulator set is free
                        ptx::tc_fence_before();
                        __syncwarp();
                        if (lane == 0) ptx::mbar_arrive(&acce[st]);
                    }
                    if (b0 == 0) {
                        if constexpr (I0 < LB) {
#pragma unroll
                            for (int c = 0; c < kNb; ++c) acc[c] = __uint_as_float(v[I0][c]);
                        } else {
#pragma unroll
                            for (int c = 0; c < kNb; ++c) acc[c] = __uint_as_float(v0[c]);
                        }
                    }
#pragma unroll
                    for (int j = 0; j < LB; ++j) {
                        if (b0 + j < G::NBP && b0 + j != I0) {
                            const int src = (lane + DLO + b0 + j) & 31;   // lane m + d of this block
                            float tv[kNb];   // a block's shuffles in flight before the adds
#pragma unroll
                            for (int c = 0; c < kNb; ++c)
                                tv[c] = __shfl_sync(0xffffffffu, __uint_as_float(v[j][c]), src);
#pragma unroll
                            for (int c = 0; c < kNb; ++c) acc[c] += tv[c];
                        }
                    }
                }
                // Stage this warp's output rows (one parity of the quarter,
                // item j's 16 columns of the tile's 32) with the TMA 128-byte
                // swizzle (16-byte chunk XOR row bits), then one TMA store per
                // tile through the parity view.
                if (j == 0) {
                    if (lane == 0) ptx::bulk_wait_group_read<0>();   // the previous tile's store has read the buffer
                    __syncwarp();
                }
                if (lane >= G::DM && lane < kLanes - G::DM) {
                    const int o = lane - G::DM;
#pragma unroll
                    for (int c = 0; c < kNb; c += 4) {
                        const int sw = ((kNb * j + c) >> 2) ^ (o & 7);
                        *reinterpret_cast<float4*>(ost + o * (kTw * 4) + sw * 16) =
                            make_float4(acc[c], acc[c + 1], acc[c + 2], acc[c + 3]);
                    }
                }
                if (j == kItems - 1) {
                    ptx::fence_proxy_async_smem();
                    __syncwarp();
                    const int oy = (Y0 + q * G::ROWS_OUT) / 2;   // first output row of the quarter, parity view
                    if (lane == 0 && X0 < args.x1 - args.x0 && oy < prows) {
                        ptx::tma_store_2d(omap, X0, oy, ost);
                        ptx::bulk_commit_group();
                    }
                }
            }
            }
        };
        if (p == 0)
            drain(std::integral_constant<int, 0>{});
        else
            drain(std::integral_constant<int, 1>{});
    }

    // ---- teardown (also after an abort: every role has left its loop)
    // output stores have read their staging buffers (the writes themselves
    // are visible to later work in the stream once the grid completes)
    if (warp >= 2 + kSplitWarps && warp < kMma2Warp && lane == 0) ptx::bulk_wait_group_read<0>();
    if (*abort_flag) {
        // Let copies and MMAs still in flight land before the CTA gives up its
        // shared and tensor memory (each wait bounded again).
        if (warp == 0 && lane == 0) {
            for (int k = issued - kRawStages; k < issued; ++k)
                if (k >= 0) ptx::mbar_wait(&full[k % kRawStages], (uint32_t)(k / kRawStages) & 1u, kWaitCycles / 8);
        }
        if ((warp == 1 || warp == kMma2Warp) && lane == 0 && committed >= 0)
            ptx::mbar_wait(&accf[committed % DST], (uint32_t)(committed / DST) & 1u, kWaitCycles / 8);
    }
    __syncwarp();
    if (tid == 0 && *abort_flag) atomicOr(args.err, 1u);
    ptx::tc_fence_before();
    __syncthreads();
    // every producer of this CTA is done: the last CTA resets the tile counter
    if (tid == 0 && claims) {
        __threadfence();
        if (atomicAdd(&args.sched[1], 1) == (int)gridDim.x - 1) {
            atomicExch(&args.sched[0], 0);
            atomicExch(&args.sched[1], 0);
        }
    }
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem, kTmemCols);
    }
}

// ------------------------------------------------------------------ host side
using MxKernel = void (*)(CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap, MxArgs2D);

struct KernelInfo {
    MxKernel fn = nullptr;
    int smem = 0;
};

template <int R, bool BF, int NP>
KernelInfo kernel_info() {
    return {mx2d_kernel<R, BF, NP>, smem_bytes<R, BF>()};
}

template <int R>
KernelInfo kernel_for_parts(bool bf, int np) {
    if (bf) return np == 1 ? kernel_info<R, true, 1>() : np == 2 ? kernel_info<R, true, 2>() : kernel_info<R, true, 3>();
    return np == 1 ? kernel_info<R, false, 1>() : kernel_info<R, false, 2>();
}

// Kernel of order r for BF16 (else TF32) operands split into np parts.
KernelInfo kernel_for(int r, bool bf, int np) {
    switch (r) {
        case 1: return kernel_for_parts<1>(bf, np);
        case 2: return kernel_for_parts<2>(bf, np);
        case 3: return kernel_for_parts<3>(bf, np);
        case 4: return kernel_for_parts<4>(bf, np);
    }
    return {};
}

// Block list of order r, in their order along N (Pair::pos): block (p, i) (lane
// offset d = dlo(p) + i) stacks line 2d - p + r over line 2d - p + r + 1 (null
// outside 0..2r) and goes into output parity p.
template <int R>
std::vector<PairBlock> pair_blocks(const double* cg) {
    using G = Pair<R>;
    std::vector<PairBlock> out(G::NBLK);
    for (int p = 0; p < 2; ++p)
        for (int i = 0; i < G::NBP; ++i) {
            PairBlock b{{nullptr, nullptr}, p};
            for (int e = 0; e < 2; ++e) {
                const int a = 2 * (G::dlo(p) + i) - p + R + e;
                if (a >= 0 && a <= 2 * R) b.line[e] = cg + a * (2 * R + 1);
            }
            out[G::pos(p, i)] = b;
        }
    return out;
}

std::vector<PairBlock> pair_blocks(int r, const double* cg) {
    switch (r) {
        case 1: return pair_blocks<1>(cg);
        case 2: return pair_blocks<2>(cg);
        case 3: return pair_blocks<3>(cg);
        default: return pair_blocks<4>(cg);
    }
}

// Row-parity view of a row-major grid with rows of ldx elements: rows parity,
// parity + 2, ... (a 2D tensor of rows_p rows of nx elements, row stride two
// grid rows).
bool encode_parity_map(CUtensorMap* map, const float* base, int rows_p, int nx, int64_t ldx, int box_x, int box_y,
                       CUtensorMapSwizzle swz, CUtensorMapL2promotion l2) {
    auto enc = get_encode();
    if (!enc) return false;
    cuuint64_t dims[2] = {(cuuint64_t)nx, (cuuint64_t)rows_p};
    cuuint64_t strides[1] = {(cuuint64_t)ldx * 8};
    cuuint32_t box[2] = {(cuuint32_t)box_x, (cuuint32_t)box_y};
    cuuint32_t es[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, (void*)base, dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, swz, l2, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// What a sweep of one depth needs (offsets into the plan's operand buffer).
struct DepthOps {
    int order = 0;             // order of the composed stencil, depth * r
    size_t bops = 0;           // banded operands
    int copies = 1;            // of the banded operands, one after the other
    uint32_t bop_bytes = 0;
    uint32_t bpart_bytes = 0;
    int strip_rows = 0;        // rows (columns) along each face computed as strips (0: none)
    int strip_classes = 0;
    size_t strip_w = 0;
};

struct MxState {
    unsigned int* err_host = nullptr;  // host-mapped error word
    unsigned int* err_dev = nullptr;
    int* sched = nullptr;              // device tile counter pair (in the operand buffer; zero between launches)
    int num_sms = 0;
    bool bf = false;      // BF16 operands (else TF32)
    DepthOps depth[kMaxDepth + 1];     // [1 .. the plan's tb]
};

constexpr size_t kSchedBytes = 256;    // of the operand buffer: the tile counters

// Tiles of a region of ny x nx outputs for a stencil of order r.
int64_t tiles_2d(int64_t ny, int64_t nx, int r) {
    const int rows = kQuarters * 2 * (kLanes - 2 * ((r + 1) / 2));
    return (nx + kTw - 1) / kTw * ((ny + rows - 1) / rows);
}

// Weights of `k` steps of a 2D stencil as one stencil of order k r: what the
// input at each offset contributes to one output point when the points past
// the given limits (offsets from the output point) are outside the grid, that
// is, zero at every step in between.  Without limits this is the k-fold
// convolution of the weights.
struct Limits {
    int ylo, yhi, xlo, xhi;
};
constexpr int kNoLimit = 1 << 20;

std::vector<double> compose_steps(int r, const double* cg, int k, const Limits& in) {
    const int R = k * r, W = 2 * R + 1, w = 2 * r + 1;
    std::vector<double> cur((size_t)W * W, 0.0), nxt;
    cur[(size_t)R * W + R] = 1.0;
    for (int step = 1; step <= k; ++step) {
        nxt.assign(cur.size(), 0.0);
        const int h = (step - 1) * r;
        for (int y = -h; y <= h; ++y)
            for (int x = -h; x <= h; ++x) {
                const double v = cur[(size_t)(y + R) * W + x + R];
                if (v == 0.0) continue;
                const int a0 = std::max(0, in.ylo - y + r), a1 = std::min(w - 1, in.yhi - y + r);
                const int b0 = std::max(0, in.xlo - x + r), b1 = std::min(w - 1, in.xhi - x + r);
                for (int a = a0; a <= a1; ++a) {
                    double* const row = &nxt[(size_t)(y + a - r + R) * W + x - r + R];
                    for (int b = b0; b <= b1; ++b) row[b] += cg[a * w + b] * v;
                }
            }
        cur.swap(nxt);
    }
    return cur;
}

// Split precisions that stand in for FP32 arithmetic; only these fuse steps.
// In the others the rounding of the weights and of the field at every step is
// part of the result a caller asked for.
bool fp32_class(int prec) { return prec == STENCIL_PREC_TF32X3 || prec == STENCIL_PREC_BF16X3; }

bool strips_in_kernel(const MxRequest& q) {
    return fp32_class(q.prec) && q.n[0] >= kStripMin && q.n[1] >= kStripMin;
}

// Most time steps that one sweep may advance.  k steps of an order-r stencil
// are one step of an order-kr stencil, as long as the largest order built (4)
// holds it.  Only when the composed weights are as safe as the single steps:
// within FP32's range by a wide margin, and with no larger a rounding error
// (the composed weights' absolute sum bounds it; k single steps have k times
// the weights' absolute sum, times the growth of a constant field).
int most_depth(const MxRequest& q) {
    if (q.tb != 0 || !strips_in_kernel(q)) return 1;
    const int w = 2 * q.r + 1;
    double sum = 0.0, abs_sum = 0.0;
    for (int i = 0; i < w * w; ++i) {
        sum += q.cg[i];
        abs_sum += std::fabs(q.cg[i]);
    }
    if (!(abs_sum > std::ldexp(1.0, -24) && abs_sum < std::ldexp(1.0, 24))) return 1;
    for (int k = std::min(kMaxDepth, 4 / q.r); k > 1; --k) {
        double composed = 0.0;
        for (double v : compose_steps(q.r, q.cg, k, {-kNoLimit, kNoLimit, -kNoLimit, kNoLimit})) composed += std::fabs(v);
        if (composed <= 1.0001 * k * abs_sum * std::max(1.0, std::pow(std::fabs(sum), k - 1))) return k;
    }
    return 1;
}

// Grid region of the tiles of a sweep with strips of `rows` points along each
// face (0: none), from an even row (row-parity views) and a 16-byte column
// group, and the strip items: of whole rows, and beside the region.
struct Region {
    int x0 = 0, y0 = 0, x1, y1;
    int64_t row_items = 0, col_items = 0;
    Region(int ny, int nx, int rows) : x1(nx), y1(ny) {
        if (rows <= 0) return;
        x0 = kStripCols;
        y0 = (rows + 1) / 2 * 2;
        x1 = (nx - rows) / 4 * 4;
        y1 = ny - rows;
        const int groups = (nx + 3) / 4;
        row_items = (int64_t)(y0 + ny - y1) * groups;
        col_items = (int64_t)(y1 - y0) * (x0 / 4 + groups - x1 / 4);
    }
    int64_t items() const { return row_items + col_items; }
};

int strip_rows(int r, int bc, int depth) { return bc == kBcPeriodic ? depth * r : (depth - 1) * r; }

// Estimated us per time step of sweeps of `depth` steps, with the faces as
// strips in the sweep's kernel or (depth 1) as the periodic edge kernel's.  A
// sweep's time grows far slower than its order: us per tile of an SM 1.5 / 1.6
// / 1.8 / 2.05 for orders 1 to 4 (8192^2: 89 / 94 / 113 / 125), so many steps at
// once are the faster, unless the strips outlast the tiles: one warp per CTA
// takes about 4 us for 32 items along a row and 7 for 32 down a column
// (periodic: 3.5 and 5.5), and short or narrow grids have many for their size.
// The edge kernel takes a few us and some time per point, more down columns.
// us per step, the rule's choice / the other: 1000000 x 96 r = 2 zero halo single
// sweeps 124 / two steps with strips 1393; 96 x 1000000 r = 3 periodic edge kernel
// 544 / strips 1242; 8192^2 r = 2 two steps with strips 66 / single sweeps 96.
double step_cost(const MxRequest& q, int num_sms, int depth, bool strips) {
    static const double kTile[5] = {0.0, 1.5, 1.6, 1.8, 2.05};
    static const double kEdge[5] = {0.0, 2.5, 4.0, 6.0, 9.0};
    static const double kEdgeRow[5] = {0.0, 15e-6, 23e-6, 40e-6, 60e-6};   // per point of whole rows
    static const double kEdgeCol[5] = {0.0, 58e-6, 50e-6, 90e-6, 145e-6};  // per point down columns
    const bool periodic = q.bc == kBcPeriodic;
    const int ny = (int)q.n[0], nx = (int)q.n[1];
    const Region g(ny, nx, strips ? strip_rows(q.r, q.bc, depth) : 0);
    const int64_t tiles = tiles_2d(g.y1 - g.y0, g.x1 - g.x0, depth * q.r);
    const int64_t ctas = std::min<int64_t>(num_sms, std::max<int64_t>(tiles, (g.items() + 31) / 32));
    const double tile_us = (double)((tiles + ctas - 1) / ctas) * kTile[depth * q.r];
    double strip_us = 0.0;
    if (g.items() > 0) {
        const double us = ((periodic ? 3.5 : 4.0) * g.row_items + (periodic ? 5.5 : 7.0) * g.col_items) / g.items();
        strip_us = us * std::max(1.0, (double)g.items() / (32.0 * ctas));
    }
    const double edge_us =
        periodic && !strips ? kEdge[q.r] + 2.0 * q.r * (ny * kEdgeCol[q.r] + nx * kEdgeRow[q.r]) : 0.0;
    return (4.0 + std::max(tile_us, strip_us) + edge_us) / depth;
}

// Time steps per sweep, and whether its kernel computes the faces as strips.
struct SweepKind {
    int depth = 1;
    bool strips = false;
};

SweepKind sweep_kind(const MxRequest& q, int num_sms) {
    SweepKind best;
    double least = step_cost(q, num_sms, 1, false);
    const int deepest = most_depth(q);
    for (int depth : {1, deepest}) {
        if (!strips_in_kernel(q) || strip_rows(q.r, q.bc, depth) == 0) continue;
        const double us = step_cost(q, num_sms, depth, true);
        if (us < least) {
            least = us;
            best = {depth, true};
        }
    }
    return best;
}

// Strip weights of depth k: [y class][x class][2R+1][kStripRow], classes 0 ..
// s-1 by the distance to the low face, s past both, s+1 .. 2s up to the high
// face (s = (k-1) r for the zero halo, 0 when periodic).
std::vector<float> strip_weights(int r, const double* cg, int k, int s) {
    const int R = k * r, W = 2 * R + 1, n = 2 * s + 1;
    std::vector<float> out((size_t)n * n * W * kStripRow, 0.0f);
    auto lo = [&](int c) { return c < s ? -c : -kNoLimit; };
    auto hi = [&](int c) { return c > s ? 2 * s - c : kNoLimit; };
    for (int cy = 0; cy < n; ++cy)
        for (int cx = 0; cx < n; ++cx) {
            const std::vector<double> c = compose_steps(r, cg, k, {lo(cy), hi(cy), lo(cx), hi(cx)});
            for (int a = 0; a < W; ++a)
                for (int b = 0; b < W; ++b)
                    out[(((size_t)cy * n + cx) * W + a) * kStripRow + b] = (float)c[(size_t)a * W + b];
        }
    return out;
}

}  // namespace

bool mx_supported(const MxRequest& q, std::string* why) {
    if (q.f64) {
        if (why) *why = "FP64 storage runs on the CUDA-core kernel (no FP64 tensor-core path on this GPU)";
        return false;
    }
    if (q.ndim == 3) return mx3d_supported(q, why);
    if (q.cover == STENCIL_COVER_HYBRID) {
        if (why) *why = "the hybrid line cover is built for 3D stars";
        return false;
    }
    if (!mx_precision(q.prec)) {
        if (why) *why = "the outer-product kernels run TF32, TF32X3, BF16, BF16X2, BF16X3 or BF16_W2";
        return false;
    }
    if (q.ldx % 4 != 0) {
        if (why) *why = "the row stride must be a multiple of 4 (16-byte TMA rows)";
        return false;
    }
    if (q.n[0] < 2) {
        if (why) *why = "the matrixized 2D kernel needs at least two rows";
        return false;
    }
    if (q.tb > 1) {
        if (why) *why = "temporal blocking not built for the matrixized kernel";
        return false;
    }
    return true;
}

// Periodic plans also get the boundary-term table of the edge kernel; a plan
// that cannot get it is freed.
static stencil_status with_edges(const MxRequest& q, MxPlan* p, std::string* why) {
    const stencil_status s = mx_edges_build(q, p);
    if (s != STENCIL_OK) {
        mx_plan_free(p);
        if (why) *why = "the periodic boundary-term table holds r <= 4 and at most 120 terms";
    }
    return s;
}

stencil_status mx_plan_build(const MxRequest& q, MxPlan* p, std::string* why) {
    if (!mx_supported(q, why)) return STENCIL_EUNSUPPORTED;
    p->ndim = q.ndim;
    for (int d = 0; d < 3; ++d) p->n[d] = q.n[d];
    p->ldx = q.ldx;
    p->unit_planes = q.unit_planes;
    p->r = q.r;
    p->bc = q.bc;
    p->prec = q.prec;
    p->tb = 1;
    p->n_edge_terms = 0;
    if (q.ndim == 3) {
        const stencil_status s3 = mx3d_plan_build(q, p, why);
        return s3 == STENCIL_OK ? with_edges(q, p, why) : s3;
    }
    const bool bf = is_bf16(q.prec);
    const int W = bf ? window<true>(kNb) : window<false>(kNb);
    int dev = 0, num_sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) {
        if (why) *why = std::string("device: ") + cudaGetErrorString(e);
        return STENCIL_ECUDA;
    }
    const SweepKind kind = sweep_kind(q, num_sms);
    p->nb = kNb;
    p->tb = kind.depth;
    p->n_lines = 2 * q.r + 1;
    p->cover = STENCIL_COVER_PARALLEL;
    p->n_scalar = 0;
    // One buffer: the tile counter pair (zero), each depth's strip weights and
    // banded operands, the whole sweeps' operands last and in several copies
    // (CTA b reads copy b % copies).
    DepthOps depth[kMaxDepth + 1];
    std::vector<unsigned char> all(kSchedBytes, 0);
    for (int k = 1; k <= p->tb; ++k) {
        DepthOps& d = depth[k];
        d.order = k * q.r;
        d.strip_rows = kind.strips ? strip_rows(q.r, q.bc, k) : 0;
        if (d.strip_rows > 0) {
            const int s = q.bc == kBcPeriodic ? 0 : d.strip_rows;
            const std::vector<float> w = strip_weights(q.r, q.cg, k, s);
            d.strip_classes = 2 * s + 1;
            d.strip_w = all.size();
            all.insert(all.end(), (const unsigned char*)w.data(), (const unsigned char*)(w.data() + w.size()));
        }
        const std::vector<double> cg = compose_steps(q.r, q.cg, k, {-kNoLimit, kNoLimit, -kNoLimit, kNoLimit});
        const bool cancel = p->tb > 1;
        const std::vector<PairBlock> blocks = pair_blocks(d.order, cg.data());
        const std::vector<unsigned char> ops = bf ? pack_blocks<true>(d.order, blocks, kNb, W, cancel, &d.bpart_bytes)
                                                  : pack_blocks<false>(d.order, blocks, kNb, W, cancel, &d.bpart_bytes);
        d.bop_bytes = (uint32_t)ops.size();
        if (!kernel_for(d.order, bf, operand_parts(q.prec)).fn || d.bop_bytes != (bf ? 3 : 2) * d.bpart_bytes ||
            d.bop_bytes % 16 != 0) {
            if (why) *why = "internal error: block operand size";
            return STENCIL_EUNSUPPORTED;
        }
        d.bops = all.size();
        all.insert(all.end(), ops.begin(), ops.end());
    }
    DepthOps& last = depth[p->tb];
    const int64_t ctas = std::min<int64_t>(num_sms, tiles_2d(q.n[0], q.n[1], last.order));
    last.copies = (int)std::min<int64_t>(kBopCopies, (ctas + kCtasPerCopy - 1) / kCtasPerCopy);
    last.copies = (int)std::min<int64_t>(last.copies, 1 + (int64_t)(kMostOperands - all.size()) / last.bop_bytes);
    p->operand_bytes = all.size() + (size_t)(last.copies - 1) * last.bop_bytes;
    e = cudaMalloc(&p->d_operands, p->operand_bytes);
    if (e != cudaSuccess) {
        p->d_operands = nullptr;
        if (why) *why = std::string("operand upload: ") + cudaGetErrorString(e);
        return STENCIL_ENOMEM;
    }
    e = cudaMemcpy(p->d_operands, all.data(), all.size(), cudaMemcpyHostToDevice);
    unsigned char* const first = (unsigned char*)p->d_operands + last.bops;
    for (int have = 1; have < last.copies && e == cudaSuccess;) {   // 1 -> 2 -> 4 .. copies
        const int more = std::min(have, last.copies - have);
        e = cudaMemcpyAsync(first + (size_t)have * last.bop_bytes, first, (size_t)more * last.bop_bytes,
                            cudaMemcpyDeviceToDevice, cudaStreamLegacy);
        have += more;
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(cudaStreamLegacy);
    if (e != cudaSuccess) {
        cudaFree(p->d_operands);
        p->d_operands = nullptr;
        if (why) *why = std::string("operand upload: ") + cudaGetErrorString(e);
        return STENCIL_ECUDA;
    }
    MxState* st = new MxState();
    for (int k = 1; k <= p->tb; ++k) st->depth[k] = depth[k];
    st->bf = bf;
    e = cudaHostAlloc((void**)&st->err_host, sizeof(unsigned int), cudaHostAllocMapped);
    if (e == cudaSuccess) e = cudaHostGetDevicePointer((void**)&st->err_dev, st->err_host, 0);
    if (e != cudaSuccess) {
        cudaFree(p->d_operands);
        p->d_operands = nullptr;
        delete st;
        if (why) *why = std::string("error word: ") + cudaGetErrorString(e);
        return STENCIL_ECUDA;
    }
    *st->err_host = 0;
    st->sched = (int*)p->d_operands;
    st->num_sms = num_sms;
    p->tmap_storage = st;
    for (int k = 1; k <= p->tb && e == cudaSuccess; ++k) {
        const KernelInfo ki = kernel_for(k * q.r, bf, operand_parts(q.prec));
        e = cudaFuncSetAttribute(ki.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, ki.smem);
    }
    if (e != cudaSuccess) {
        mx_plan_free(p);
        if (why) *why = std::string("kernel set-up: ") + cudaGetErrorString(e);
        return STENCIL_ECUDA;
    }
    return kind.strips ? STENCIL_OK : with_edges(q, p, why);   // the strips cover the periodic boundary
}

void mx_plan_free(MxPlan* p) {
    if (p->ndim == 3) {
        mx3d_plan_free(p);
        return;
    }
    if (p->d_operands) cudaFree(p->d_operands);
    p->d_operands = nullptr;
    MxState* st = (MxState*)p->tmap_storage;
    if (st) {
        if (st->err_host) cudaFreeHost(st->err_host);
        delete st;
    }
    p->tmap_storage = nullptr;
}

unsigned int mx_device_error(const MxPlan& p) {
    if (p.ndim == 3) return mx3d_device_error(p);
    const MxState* st = (const MxState*)p.tmap_storage;
    return st && st->err_host ? *(volatile unsigned int*)st->err_host : 0u;
}

cudaError_t mx_sweep(const MxPlan& p, const void* src, void* dst, int tb, cudaStream_t s) {
    const cudaError_t e = p.ndim == 3 ? mx3d_sweep(p, src, dst, tb, s) : mx2d_sweep(p, src, dst, tb, s);
    // periodic boundary: the kernels ran with a zero halo in x and y
    return e == cudaSuccess ? mx_periodic_edges(p, src, dst, s) : e;
}

cudaError_t mx2d_sweep(const MxPlan& p, const void* src, void* dst, int tb, cudaStream_t s) {
    if (tb < 1 || tb > p.tb) return cudaErrorInvalidValue;
    if (((uintptr_t)src & 15u) || ((uintptr_t)dst & 15u)) return cudaErrorMisalignedAddress;
    const MxState* st = (const MxState*)p.tmap_storage;
    const DepthOps& d = st->depth[tb];
    const int ny = (int)p.n[0], nx = (int)p.n[1];
    const int dm = (d.order + 1) / 2;
    const int RWD = st->bf ? raw_row<true>(kNb) : raw_row<false>(kNb);
    MxArgs2D a;
    memset(&a, 0, sizeof(a));
    a.bops = (const unsigned char*)p.d_operands + d.bops;
    a.err = st->err_dev;
    a.sched = st->sched;
    a.ny = ny;
    a.nx = nx;
    a.ldx = p.ldx;
    a.nparts = operand_parts(p.prec);
    a.nprod = products_for(p.prec);
    a.bpart_bytes = d.bpart_bytes;
    a.bop_bytes = d.bop_bytes;
    a.bop_copies = d.copies;
    a.bc = p.bc;
    a.in = (const float*)src;
    a.out = (float*)dst;
    // the tiles' region: all of the grid, or what the strips leave
    const Region region(ny, nx, d.strip_rows);
    a.x0 = region.x0;
    a.y0 = region.y0;
    a.x1 = region.x1;
    a.y1 = region.y1;
    if (d.strip_rows > 0) {
        a.strip_classes = d.strip_classes;
        a.strip_w = (const float*)((const unsigned char*)p.d_operands + d.strip_w);
    }
    const int rx = a.x1 - a.x0, ry = a.y1 - a.y0;
    a.tiles_x = (rx + kTw - 1) / kTw;
    a.tiles_total = (int)tiles_2d(ry, rx, d.order);
    a.rows_even = (ry + 1) / 2;
    a.rows_odd = ry / 2;
    const int64_t ld = p.ldx;
    float* const out = a.out + a.y0 * ld + a.x0;
    alignas(64) CUtensorMap te, to, oe, oo;
    const int kp = raw_pitch(RWD);
    if (!encode_parity_map(&te, a.in, (ny + 1) / 2, nx, ld, kp, kLanes, CU_TENSOR_MAP_SWIZZLE_NONE,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B) ||
        !encode_parity_map(&to, a.in + ld, ny / 2, nx, ld, kp, kLanes, CU_TENSOR_MAP_SWIZZLE_NONE,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B) ||
        !encode_parity_map(&oe, out, a.rows_even, rx, ld, kTw, kLanes - 2 * dm, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_NONE) ||
        !encode_parity_map(&oo, out + ld, a.rows_odd, rx, ld, kTw, kLanes - 2 * dm, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_NONE))
        return cudaErrorInvalidValue;
    const KernelInfo ki = kernel_for(d.order, st->bf, operand_parts(p.prec));
    // a CTA per tile or per warp of strip items, up to one per SM
    const int64_t want = std::max<int64_t>(a.tiles_total, (region.items() + 31) / 32);
    const int grid = (int)std::min<int64_t>(want, st->num_sms);
    return launch_dependent(ki.fn, grid, kThreads, ki.smem, s, te, to, oe, oo, a);
}

}  // namespace stx
