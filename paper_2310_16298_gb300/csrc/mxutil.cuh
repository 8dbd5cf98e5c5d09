// Helpers shared by the matrixized kernels (2D and 3D).
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <vector>

#include "plan.h"

#include "../../include/stencil.h"
#include "ptx.cuh"

namespace stx {
namespace mxu {

constexpr long long kWaitCycles = 4000000000LL;  // ~2 s at 2 GHz

// Bounded mbarrier wait that also gives up once another role has failed.
// Between polls the warp sleeps briefly, so that waiting warps leave the
// issue slots (and the shared-memory pipe) to the warps doing the work.
__device__ __forceinline__ bool wait_or_abort(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
    const long long t0 = clock64();
    while (!ptx::mbar_try_wait(bar, parity)) {
        __nanosleep(64);
        if (*abort_flag) return false;
        if (clock64() - t0 > kWaitCycles) {
            *abort_flag = 1;
            return false;
        }
    }
    return true;
}

// TF32 high part by integer rounding (nearest, ties away from zero): the low
// 13 mantissa bits are cleared after adding half of their weight.
__device__ __forceinline__ uint32_t tf32_hi_bits(float x) {
    return (__float_as_uint(x) + 0x1000u) & 0xFFFFE000u;
}

// BF16 bits (upper half of the FP32 pattern) of x rounded to nearest, ties to
// even; finite inputs.
__device__ __forceinline__ uint32_t bf16_rn_bits(float x) {
    const uint32_t u = __float_as_uint(x);
    return (u + 0x7FFFu + ((u >> 16) & 1u)) >> 16;
}


// Operand formats of the matrixized kernels.  Both use, per MMA K-step, 8
// tensor-memory columns of A and two 16-byte chunks of B:
//   TF32 (kind::tf32): one element per column, K = 8 per MMA, parts hi/lo;
//   BF16 (kind::f16):  two elements per column, K = 16 per MMA, parts 0/1/2.
template <bool BF>
struct OpFmt {
    static constexpr int kKStep = BF ? 16 : 8;          // K per MMA
    static constexpr int kGroup = BF ? 16 : 8;          // input columns per tcgen05.st x8
    static constexpr uint32_t kFmt = BF ? 1u : 2u;      // instruction-descriptor A/B format
    static constexpr int kMaxParts = BF ? 3 : 2;
    __host__ __device__ static constexpr int window(int nb) {  // K window for nb outputs
        return ((nb + 8) + kKStep - 1) / kKStep * kKStep;
    }
    __host__ __device__ static constexpr int part_cols(int k) { return BF ? k / 2 : k; }
};

// Products per K step of a precision mode (see issue_products).
inline int products_for(int prec) {
    switch (prec) {
        case STENCIL_PREC_TF32X3: return 3;
        case STENCIL_PREC_BF16X2: return 3;
        case STENCIL_PREC_BF16X3: return 6;
        case STENCIL_PREC_BF16_W2: return 2;
    }
    return 1;
}

// Precisions the outer-product kernels run.
inline bool mx_precision(int prec) { return prec >= STENCIL_PREC_TF32 && prec <= STENCIL_PREC_BF16_W2; }

inline int operand_parts(int prec) {
    switch (prec) {
        case STENCIL_PREC_TF32X3: return 2;
        case STENCIL_PREC_BF16X2: return 2;
        case STENCIL_PREC_BF16X3: return 3;
    }
    return 1;
}

inline bool is_bf16(int prec) {
    return prec == STENCIL_PREC_BF16 || prec == STENCIL_PREC_BF16X2 || prec == STENCIL_PREC_BF16X3 ||
           prec == STENCIL_PREC_BF16_W2;
}

// Issue every K step of one product (A part PA, B part PB) into accumulator
// d; FIRST clears the accumulator with the first step.
template <bool BF, int KS, int PA, int PB, bool FIRST>
__device__ __forceinline__ void issue_product(uint32_t d, uint32_t a_base, int part_cols, uint64_t b_desc0,
                                              uint32_t bpart_bytes, int n, uint32_t idesc) {
    const uint32_t a = a_base + (uint32_t)(PA * part_cols);
    const uint64_t b = b_desc0 + (uint64_t)((PB * bpart_bytes) >> 4);
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
        const uint64_t bd = b + (uint64_t)((2 * ks * n * 16) >> 4);
        if (FIRST && ks == 0)
            ptx::mma_ts<BF, true>(d, a + 8 * ks, bd, idesc);
        else
            ptx::mma_ts<BF, false>(d, a + 8 * ks, bd, idesc);
    }
}

// Issue every product of one tile (A in tensor memory, B in shared memory)
// into accumulator d, smallest products first: nprod = 1 (x0*h0), 2 (x0*h1,
// x0*h0), 3 (x1*h0, x0*h1, x0*h0) or 6 (x0*h2, x1*h1, x2*h0, x1*h0, x0*h1,
// x0*h0).  Each product count is its own fixed sequence.
template <bool BF, int KS>
__device__ __forceinline__ void issue_products(uint32_t d, uint32_t a_base, int pc, uint64_t b0, uint32_t bpb,
                                               int n, uint32_t idesc, int nprod) {
    switch (nprod) {
        case 1:
            issue_product<BF, KS, 0, 0, true>(d, a_base, pc, b0, bpb, n, idesc);
            break;
        case 2:
            issue_product<BF, KS, 0, 1, true>(d, a_base, pc, b0, bpb, n, idesc);
            issue_product<BF, KS, 0, 0, false>(d, a_base, pc, b0, bpb, n, idesc);
            break;
        case 3:
            issue_product<BF, KS, 1, 0, true>(d, a_base, pc, b0, bpb, n, idesc);
            issue_product<BF, KS, 0, 1, false>(d, a_base, pc, b0, bpb, n, idesc);
            issue_product<BF, KS, 0, 0, false>(d, a_base, pc, b0, bpb, n, idesc);
            break;
        case 6:
            issue_product<BF, KS, 0, 2, true>(d, a_base, pc, b0, bpb, n, idesc);
            issue_product<BF, KS, 1, 1, false>(d, a_base, pc, b0, bpb, n, idesc);
            issue_product<BF, KS, 2, 0, false>(d, a_base, pc, b0, bpb, n, idesc);
            issue_product<BF, KS, 1, 0, false>(d, a_base, pc, b0, bpb, n, idesc);
            issue_product<BF, KS, 0, 1, false>(d, a_base, pc, b0, bpb, n, idesc);
            issue_product<BF, KS, 0, 0, false>(d, a_base, pc, b0, bpb, n, idesc);
            break;
    }
}

// Split kGroup input values into NP operand parts and write them to the
// warp's tensor-memory lanes at column c (part p at a_base + p*part_cols).
// The stores have completed when this returns.
template <bool BF, int NP>
__device__ __forceinline__ void split_store(const float* x, uint32_t a_base, int part_cols, int c) {
    if constexpr (!BF) {
        uint32_t h[8], l[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            h[e] = tf32_hi_bits(x[e]);
            if constexpr (NP > 1) l[e] = __float_as_uint(x[e] - __uint_as_float(h[e]));
        }
        if constexpr (NP > 1)
            ptx::tmem_st_x8_sync(a_base + (uint32_t)c, h, a_base + (uint32_t)(part_cols + c), l);
        else
            ptx::tmem_st_x8_sync(a_base + (uint32_t)c, h);
    } else {
        uint32_t w[NP][8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            float r0a = x[2 * e], r0b = x[2 * e + 1];
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                const uint32_t ba = bf16_rn_bits(r0a), bb = bf16_rn_bits(r0b);
                w[k][e] = ba | (bb << 16);
                if (k + 1 < NP) {
                    r0a -= __uint_as_float(ba << 16);
                    r0b -= __uint_as_float(bb << 16);
                }
            }
        }
        const uint32_t a0 = a_base + (uint32_t)(c / 2);
        if constexpr (NP == 1)
            ptx::tmem_st_x8_sync(a0, w[0]);
        else if constexpr (NP == 2)
            ptx::tmem_st_x8_sync(a0, w[0], a0 + (uint32_t)part_cols, w[1]);
        else
            ptx::tmem_st_x8_sync(a0, w[0], a0 + (uint32_t)part_cols, w[1], a0 + (uint32_t)(2 * part_cols), w[2]);
    }
}

// Split NGR groups of kGroup input values (x[g], written at column c0 + g *
// cstep) into NP operand parts each and write them all with one fused
// store-and-wait: the stores have completed when this returns.
template <bool BF, int NP, int NGR>
__device__ __forceinline__ void split_store_groups(const float (&x)[NGR][OpFmt<BF>::kGroup], uint32_t a_base,
                                                   int part_cols, int c0, int cstep) {
    uint32_t addr[NGR * NP];
    uint32_t w[NGR * NP][8];
#pragma unroll
    for (int g = 0; g < NGR; ++g) {
        const int c = c0 + cstep * g;
        if constexpr (!BF) {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const uint32_t h = tf32_hi_bits(x[g][e]);
                w[g * NP][e] = h;
                if constexpr (NP > 1) w[g * NP + 1][e] = __float_as_uint(x[g][e] - __uint_as_float(h));
            }
#pragma unroll
            for (int k = 0; k < NP; ++k) addr[g * NP + k] = a_base + (uint32_t)(k * part_cols + c);
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                float r0a = x[g][2 * e], r0b = x[g][2 * e + 1];
#pragma unroll
                for (int k = 0; k < NP; ++k) {
                    const uint32_t ba = bf16_rn_bits(r0a), bb = bf16_rn_bits(r0b);
                    w[g * NP + k][e] = ba | (bb << 16);
                    if (k + 1 < NP) {
                        r0a -= __uint_as_float(ba << 16);
                        r0b -= __uint_as_float(bb << 16);
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < NP; ++k) addr[g * NP + k] = a_base + (uint32_t)(k * part_cols + c / 2);
        }
    }
    ptx::tmem_st_x8_sync_n<NGR * NP>(addr, w);
}

// Run-time part count (kernels not specialised on it).
template <bool BF>
__device__ __forceinline__ void split_store(const float* x, uint32_t a_base, int part_cols, int c, int nparts) {
    if (nparts == 1)
        split_store<BF, 1>(x, a_base, part_cols, c);
    else if (nparts == 2 || !BF)
        split_store<BF, 2>(x, a_base, part_cols, c);
    else
        split_store<BF, 3>(x, a_base, part_cols, c);
}

inline PFN_cuTensorMapEncodeTiled_v12000 get_encode() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    });
    return fn;
}


// Round to BF16 on the host (nearest, ties to even); finite inputs.
inline float bf16_round(float x) {
    uint32_t u;
    memcpy(&u, &x, 4);
    u += 0x7FFFu + ((u >> 16) & 1u);
    u &= 0xFFFF0000u;
    float y;
    memcpy(&y, &u, 4);
    return y;
}

// Round to TF32 on the host (nearest, ties to even); finite inputs.
inline float tf32_round(float x) {
    uint32_t u;
    memcpy(&u, &x, 4);
    u += 0xFFFu + ((u >> 13) & 1u);
    u &= ~0x1FFFu;
    float y;
    memcpy(&y, &u, 4);
    return y;
}


// One block of the 2D kernel's operand: the lines its even and odd input rows
// are multiplied with (null: none) and the output row parity it goes into.
struct PairBlock {
    const double* line[2];
    int parity;
};

// Banded operand of a block list: block j stacks, along K, the band of its
// first line (K rows 0 .. kh-1) over the band of its second (rows kh ..
// 2kh-1).  Used when one TMEM lane holds two input rows side by side along K.
//
// `cancel` (fused TF32x3 and BF16x3 sweeps): the error of these over many steps
// is a bias of the field's amplitude from two sources, both cancelled here at
// no cost (a composed stencil's sums are longer, so its truncation is larger per
// sweep).
//  * The last parts' rounding changes the weights' sum by up to 2^-24 of it:
//    each output column's rounding errors are carried into its next weights,
//    by at most 2^-23 of any weight.
//  * The tensor core truncates an FP32 accumulator at each MMA that adds to
//    it.  On average over mantissas that loses kTrunc of the accumulator's
//    value, so a weight applied in the t-th last adding MMA of its block loses
//    about t kTrunc of its product and is packed that much larger; by
//    measurement (t - 1/2) kTrunc in TF32x3 and (t - 1) kTrunc in BF16x3, whose
//    MMAs take twice the columns, for every order (the first MMA, on to the
//    small correction products, loses less).  With up to six adding MMAs that
//    is 2.4e-7 of a weight.
// Products of either sign are corrected as if they had the accumulator's:
// measured on signed weights and fields it helps there too.  Relative L2 error
// after 100 steps, single steps / fused without / fused with (256 x 260, zero
// halo and periodic, positive and signed fields):
//   random weights, positive and signed, TF32x3: r = 1 1.2e-6..1.0e-5 single,
//   9.7e-8..8.5e-7 fused with; r = 2 2.0e-6..7.6e-6, 7.8e-8..8.8e-7;
//   BF16x3: r = 1 3.2e-6..4.8e-6 / 8.2e-7..1.7e-6 / 8.2e-8..6.1e-7, r = 2
//   3.4e-6..5.1e-6 / 1.5e-6..2.6e-6 / 8.6e-8..7.5e-7;
//   fourth-order diffusion (r = 2, weights of both signs), BF16x3
//   2.0e-6..2.7e-6 / 2.7e-6..2.8e-6 / 5.7e-7..7.1e-7.
// Weights that are all exact in one part stay as they are: fields of short
// mantissas then have exact products and sums, which truncation leaves alone.
// (Other fields' sums are truncated with such weights too, fused ones less
// often per step: five-point smoothing with 1/2 and 1/8, single / fused, TF32x3
// 2.3e-6..3.2e-6 / 1.0e-6..1.1e-6, BF16x3 2.4e-6..3.3e-6 / 9.9e-7..1.1e-6.)
constexpr double kUlp = 1.0 / (1 << 23);
constexpr double kTrunc = 0.7213475 * 0.5 * kUlp;   // E[2^e / x] / 2 ulp, x's mantissa log-uniform

template <bool bf>
std::vector<unsigned char> pack_blocks(int r, const std::vector<PairBlock>& blocks, int nb, int kh, bool cancel,
                                       uint32_t* part_bytes) {
    const int nblk = (int)blocks.size(), N = nblk * nb, kw = 2 * kh;
    constexpr int epc = bf ? 8 : 4;  // elements per 16-byte chunk
    constexpr int es = bf ? 2 : 4;
    constexpr int parts = bf ? 3 : 2;
    constexpr int kstep = OpFmt<bf>::kKStep;
    constexpr double first = bf ? 1.0 : 0.5;   // what the first MMA spares
    const size_t pb = (size_t)(kw / epc) * N * 16;
    std::vector<unsigned char> out(parts * pb, 0);
    bool exact = true;
    for (const auto& b : blocks)
        for (int e = 0; e < 2; ++e)
            for (int t = 0; b.line[e] && t < 2 * r + 1; ++t)
                exact = exact && (double)(bf ? bf16_round((float)b.line[e][t]) : tf32_round((float)b.line[e][t])) ==
                                     b.line[e][t];
    cancel = cancel && !exact;
    // The columns of a block are independent: they are packed side by side,
    // weight by weight (one after the other, each is a chain of roundings).
    std::vector<double> carries(2 * nb, 0.0);      // per output parity and column
    std::vector<int> adds(nb), step(nb);
    for (int j = 0; j < nblk; ++j) {
        double* const carry = &carries[blocks[j].parity * nb];
        // adds[q]: MMAs (kstep window columns each) that add to this block's column q;
        // weight t of a line stands at window column q + 4 - r + t
        std::fill(adds.begin(), adds.end(), 0);
        for (int e = 0; e < 2; ++e) {
            std::fill(step.begin(), step.end(), -1);
            for (int t = 0; blocks[j].line[e] && t < 2 * r + 1; ++t) {
                if (blocks[j].line[e][t] == 0.0) continue;
                for (int q = 0; q < nb; ++q) {
                    const int s = (q + 4 - r + t) / kstep;
                    adds[q] += step[q] != s;
                    step[q] = s;
                }
            }
        }
        for (int e = 0; e < 2; ++e) {
            std::fill(step.begin(), step.end(), -1);   // last K step of this row that was counted
            for (int t = 0; blocks[j].line[e] && t < 2 * r + 1; ++t) {
                const double w = blocks[j].line[e][t];
                if (w == 0.0) continue;
                const double most = std::fabs(w) * kUlp;
                for (int q = 0; q < nb; ++q) {
                    const int kk = q + 4 - r + t;
                    double rem = (double)(float)w;
                    if (cancel) {
                        adds[q] -= step[q] >= 0 && step[q] != kk / kstep;
                        step[q] = kk / kstep;
                        const double taken = std::min(std::max(carry[q], -most), most);
                        rem = w * (1.0 + (adds[q] - first) * kTrunc) + taken;
                        carry[q] -= taken;
                    }
                    const unsigned k = e * kh + kk;
                    const size_t off = ((size_t)(k / epc) * N + (size_t)(j * nb + q)) * 16 + (size_t)(k % epc) * es;
                    for (int p = 0; p < parts; ++p) {
                        const float v = bf ? bf16_round((float)rem) : tf32_round((float)rem);
                        rem -= v;
                        if (bf) {
                            uint32_t u;
                            memcpy(&u, &v, 4);
                            const uint16_t h = (uint16_t)(u >> 16);
                            memcpy(&out[p * pb + off], &h, 2);
                        } else {
                            memcpy(&out[p * pb + off], &v, 4);
                        }
                    }
                    if (cancel) carry[q] += rem;
                }
            }
            for (int q = 0; q < nb; ++q) adds[q] -= step[q] >= 0;
        }
    }
    *part_bytes = (uint32_t)pb;
    return out;
}

// Pack the banded operands of the given lines (line l: 2r+1 gather weights)
// as the MMA B operand, N = lines x nb rows, K-major 16-byte chunks:
// [part][k chunk][n = l*nb + q][16 bytes].  Row (n, k) holds the band entry
// H_l[k][q] = w_l[k - q - (4 - r)] (zero outside the band and for k >= nb + 8),
// split into TF32 hi/lo parts or three BF16 parts.  Returns the bytes of one
// part in *part_bytes.
inline std::vector<unsigned char> pack_bands(int r, const std::vector<const double*>& lines, int nb, int kwin, bool bf,
                                             uint32_t* part_bytes) {
    const int L = (int)lines.size(), N = L * nb;
    const int epc = bf ? 8 : 4;  // elements per 16-byte chunk
    const int es = bf ? 2 : 4;
    const int parts = bf ? 3 : 2;
    const size_t pb = (size_t)(kwin / epc) * N * 16;
    std::vector<unsigned char> out(parts * pb, 0);
    std::vector<double> band((size_t)(nb + 8) * nb);
    for (int l = 0; l < L; ++l) {
        band_operand(r, lines[l], nb, 4, band.data());
        for (int k = 0; k < nb + 8; ++k)
            for (int q = 0; q < nb; ++q) {
                float rem = (float)band[(size_t)k * nb + q];
                const size_t off = ((size_t)(k / epc) * N + (size_t)(l * nb + q)) * 16 + (size_t)(k % epc) * es;
                for (int p = 0; p < parts; ++p) {
                    const float v = bf ? bf16_round(rem) : tf32_round(rem);
                    rem -= v;
                    if (bf) {
                        uint32_t u;
                        memcpy(&u, &v, 4);
                        const uint16_t h = (uint16_t)(u >> 16);
                        memcpy(&out[p * pb + off], &h, 2);
                    } else {
                        memcpy(&out[p * pb + off], &v, 4);
                    }
                }
            }
    }
    *part_bytes = (uint32_t)pb;
    return out;
}

}  // namespace mxu
}  // namespace stx
