// FP64 block products on the 5th-generation tensor cores.  GB300's FP64 pipe does under two fused
// multiply-adds per clock and SM, its BF16 tensor cores about 4,096, so a product that splits
// every FP64 operand into eight BF16 digits and sums 36 digit products is still many times
// faster, as long as the tensor cores' tiles are not too empty (the scheme is Ozaki's error-free
// splitting; Ozaki, Ogita, Oishi, Rump 2012).
//
//   * The operands are read as group tiles (grouptiles.cuh) of at most 112 x 112 elements.  Row
//     i of an A tile (column j of a B tile) has the common scale 2^e above its largest element,
//     and every element is the 64-bit fixed-point number x 2^(63 - e), cut into eight balanced
//     digits d_0 .. d_7 of eight bits (|d| <= 128, exact in BF16): 63 significant bits below the
//     row's maximum, so an element keeps all its 53 bits down to 2^-10 of that maximum.
//   * One tile product (G, G'') x (G'', G') sums d_s d_t over at most 112 terms.  Products of
//     equal s + t = d go to one FP32 accumulator per element, d = 0 .. 7 (36 of the 64 pairs;
//     the rest lies below 2^-64 of the two maxima).  All are integers of magnitude at most
//     8 * 112 * 2^14 < 2^24, so the FP32 sums are exact, whatever their order.
//   * After every tile product the eight accumulators are combined and added, shifted to the C
//     block's common scale (the largest scale product of its tile rows), to a 96-bit fixed-point
//     sum per element, all in integers.  The sum is rounded to FP64 once, at the end: no FP64
//     operation per term is left.
//
// Accuracy: over whole products the error is smaller than an FP64 chain's (relative Frobenius error of
// H H on water with 13/5 blocks 2.2e-16 against 2.3e-15, of X X in the middle of the sign iteration
// 1.6e-16 against 1.3e-15).  Element by element it is about 2^-61 of the largest scale product 2^E of the
// C block's tile rows, whatever the element's own terms are (nearly all of it the pairs s + t = 8 that are left
// out), while the chain's goes with sum_k |a_ik| |b_kj|.  A block whose terms are far below 2^E (A strong in one
// atom of the tile, B in another), or weak in one of its elements (a row graded against its neighbours, an element
// beside a larger one that meets a zero), would lose bits.  k_oz_guard and k_oz_weak leave such blocks to
// the FP64 pipe: a block runs here only if its largest norm product is above 2^(E - 7) and if the block
// product that gives it, taken of the absolute values, is at least 2^(E - 13) in every element.  Digits
// against chain (emulated; root mean square over elements, in units of 2^-53 sum_k |a_ik| |b_kj|), blocks whose
// weakest element lies at 2^-12 to 2^-13: H H with 13/5 blocks 1.7 against 1.9, with 23/7 2.8 against 2.6, X X
// 0.8 against 1.4 and 1.4 against 1.8; at 2^-13 to 2^-14 up to 5 against 3.  All blocks: 0.3 to 0.9 against
// 1.4 to 2.6.  The FP64 pipe also takes the blocks of tiles too empty to pay, and every block when an operand
// holds a value that is not finite or too large or small for the scales.
#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>
#include <vector>

#include <cuda.h>
#include <cudaTypedefs.h>

#include "common.cuh"
#include "grouptiles.cuh"
#include "tc05.cuh"

namespace dbg {

namespace {

constexpr int kDigits = 8;
constexpr int kSlice = 32;                       // C columns per work item: 8 accumulators of 32 columns, twice
constexpr int kOzRows = 112;                     // rows of the widest packed tile (kGroupWidth rounded to 8)
constexpr int kOzA = kOzRows * 2 * kDigits * 16; // A bytes of a K step of 16: 28 KB
constexpr int kZeroBlocks = 6;                   // zero digit blocks before the B digits, see oz_mmas
constexpr int kDigitBlock = kSlice * 16;         // one digit of one 8-column chunk of a B slice
constexpr int kOzBChunk = (kZeroBlocks + kDigits) * kDigitBlock;
constexpr int kOzStage = kOzA + 2 * kOzBChunk;   // 42 KB
constexpr int kOzStages = 4;
constexpr int kOzEpiWarps = 16;                  // four per TMEM lane quadrant, 8 columns each
constexpr int kOzItems = 4;                      // work items in flight between the warps' roles
constexpr int kOzEpi0 = 2;                       // first epilogue warp: 0 producer, 1 MMA issuer
constexpr int kOzThreads = 32 * (kOzEpi0 + kOzEpiWarps);
constexpr int kOzTmem = 512;                     // two buffers of 8 x 32 accumulator columns
constexpr long long kOzWait = 4000000000ll;      // about 2 s
// Exponents (of the largest element of a tile row) outside this range go to the FP64 pipe: the
// result's exponent is then formed without overflow from the two operands'.
constexpr int kExpLimit = 430;
constexpr int16_t kNoExp = -32768;
// A product's flags on the device.  0: a value outside the scales' range; 1: a planned product's execution has
// blocks to repeat on the FP64 pipe; 2: a wait ran out (1; a planned product's execution then repeats every
// block) or the pattern is asymmetric (2).
constexpr int kFlagRange = 0, kFlagRedo = 1, kFlagFailed = 2, kFlags = 3;
// Clocks of one K step of one 32-column slice charged against the FP64 pipe's flops per clock and SM
// (1.01 TFLOP/s measured on the block products) when a tile is given to one of the two.  A K step takes
// 797 clocks with eight digits (oz_mmas) and fewer on average (most entries run fewer digits); beside the
// FP64 pipe's kernels the balance lies lower still, and hardly matters: sign iteration on 512 waters 222.4 ms at
// 270 and 222.6 at 200, 1,024-water product 28.3 and 28.4, ragged update 3.70 and 3.70 (before k_oz_weak, which
// sends more to the FP64 pipe, 234 ms at 430, 231 at 350, 226 at 270, 227 at 200).
constexpr double kStepClocks = 270.0, kSimtFlopsPerClock = 3.2;

// ------------------------------------------------------------------ symbolic helpers
__global__ void k_oz_role(int64_t nform, const int32_t* __restrict__ f_row, const int32_t* __restrict__ f_col,
                          const int64_t* __restrict__ mirror, int sym, const int32_t* __restrict__ grp,
                          int by_group, uint8_t* __restrict__ comp) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nform; k += (int64_t)gridDim.x * blockDim.x)
        comp[k] = block_role(sym, f_row[k], f_col[k], mirror[k], grp, by_group) == 0 ? 1 : 0;
}

// The operand tile's tables: tab[t][row member][K member] = block, and per 32-row slice the K
// steps of 16 columns that hold a block (8 bits per slice).  transpose: the tile's rows are the
// blocks' columns.
__global__ void k_oz_tiles(int64_t nb, const int32_t* __restrict__ row, const int32_t* __restrict__ col,
                           const int32_t* __restrict__ bs, const int32_t* __restrict__ g_pos,
                           const int32_t* __restrict__ g_midx, const int32_t* __restrict__ blk_tile, int transpose,
                           int32_t* __restrict__ tab, unsigned* __restrict__ smask) {
    for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < nb; b += (int64_t)gridDim.x * blockDim.x) {
        const int32_t t = blk_tile[b];
        const int32_t I = transpose ? col[b] : row[b], K = transpose ? row[b] : col[b];
        tab[(int64_t)t * (kGroupMembers * kGroupMembers) + g_midx[I] * kGroupMembers + g_midx[K]] = (int32_t)b;
        const int p0 = g_pos[K], p1 = p0 + bs[K] - 1;
        const unsigned bits = ((2u << (p1 >> 4)) - 1u) & ~((1u << (p0 >> 4)) - 1u);
        const int q0 = g_pos[I] / kSlice, q1 = (g_pos[I] + bs[I] - 1) / kSlice;
        unsigned m = 0;
        for (int q = q0; q <= q1; ++q) m |= bits << (8 * q);
        atomicOr(smask + t, m);
    }
}

__device__ __forceinline__ unsigned fold8(unsigned m) {
    m |= m >> 16;
    return (m | (m >> 8)) & 255u;
}

// ------------------------------------------------------------------ packing
struct OzPackArgs {
    int64_t nt;
    const int32_t* t_rgrp; const int32_t* t_kgrp;   // row and K group of every tile
    const int32_t* tab; const unsigned* smask;
    const int32_t* g_ptr; const int32_t* g_mrec; const int32_t* g_w;
    const int64_t* off; const double* data;
    int transpose;
    int R, KS;                                      // packed rows and K steps of every tile
    uint8_t* pack; int16_t* rexp; int16_t* mexp;    // digits; exponent per row; largest exponent per member
    int* bad;
};

// One CTA per tile.  Pass 1 finds every row's largest element, pass 2 cuts the elements into
// digits and writes them 8 columns of one row and digit (16 bytes) at a time, threads over
// consecutive rows, so a warp writes 512 contiguous bytes; every element of the K steps in use is
// written, zeros included, and nothing is cleared beforehand.  Bound by its writes (16 bytes per
// padded element) and by the integer work of the digits (about 10 instructions each).
// Packed tile: K step k at k * 2 * 8 * R * 16 bytes, then chunk (8 columns), digit, row.
__global__ void __launch_bounds__(256) k_oz_pack(OzPackArgs P) {
    __shared__ int64_t boff[kGroupMembers][kGroupMembers];
    __shared__ int rmax[kOzRows];
    __shared__ uint8_t rmem[kOzRows], kmem[kOzRows];      // member of every row / K column, 255: none
    __shared__ int rrec[kGroupMembers], krec[kGroupMembers];
    const int tid = threadIdx.x;
    for (int64_t t = blockIdx.x; t < P.nt; t += gridDim.x) {
        const int G = P.t_rgrp[t], K = P.t_kgrp[t];
        const int m0 = P.g_ptr[G], nm = P.g_ptr[G + 1] - m0, n0 = P.g_ptr[K], nn = P.g_ptr[K + 1] - n0;
        const unsigned km = fold8(P.smask[t]);
        {
            const int32_t b = P.tab[t * (kGroupMembers * kGroupMembers) + tid];
            boff[tid >> 4][tid & 15] = b >= 0 ? P.off[b] : -1;
        }
        if (tid < kOzRows) {
            rmax[tid] = 0;
            rmem[tid] = 255;
            kmem[tid] = 255;
        }
        if (tid < nm) rrec[tid] = P.g_mrec[m0 + tid];
        if (tid < nn) krec[tid] = P.g_mrec[n0 + tid];
        __syncthreads();
        if (tid < nm)
            for (int i = 0; i < (rrec[tid] >> 8); ++i) rmem[(rrec[tid] & 255) + i] = (uint8_t)tid;
        if (tid >= 32 && tid - 32 < nn)
            for (int i = 0; i < (krec[tid - 32] >> 8); ++i) kmem[(krec[tid - 32] & 255) + i] = (uint8_t)(tid - 32);
        __syncthreads();
        const int units = P.R * 2 * P.KS;
        // element (row r, K column kc) of the tile; 0 where there is no block
        auto load = [&](int r, int a, int kc) -> uint64_t {
            const int b = kc < kOzRows ? kmem[kc] : 255;
            if (a == 255 || b == 255) return 0ull;
            const int64_t o = boff[a][b];
            if (o < 0) return 0ull;
            const int i = r - (rrec[a] & 255), j = kc - (krec[b] & 255);
            const int64_t p = P.transpose ? (int64_t)j * (rrec[a] >> 8) + i : (int64_t)i * (krec[b] >> 8) + j;
            return (uint64_t)__double_as_longlong(P.data[o + p]);
        };
        for (int u = tid; u < units; u += 256) {
            const int c = u / P.R, r = u - c * P.R;
            if (!((km >> (c >> 1)) & 1u)) continue;
            const int a = rmem[r];
            if (a == 255) continue;
            unsigned m = 0;
#pragma unroll
            for (int x = 0; x < 8; ++x) {
                const uint64_t b = load(r, a, 8 * c + x);
                m = max(m, 2u * ((unsigned)(b >> 52) & 0x7ffu) + ((b << 1) != 0u ? 1u : 0u));
            }
            if (m) atomicMax(&rmax[r], (int)m);
        }
        __syncthreads();
        if (tid < P.R) {
            // (a row of subnormals alone, m = 0 with a nonzero element, is outside the range as well)
            const int any = rmax[tid] & 1, m = rmax[tid] >> 1;
            if (any && (m > 1023 + kExpLimit || m < 1023 - kExpLimit)) atomicExch(P.bad, 1);
            rmax[tid] = m;
            P.rexp[t * P.R + tid] = (int16_t)(m ? m - 1022 : 0);
        }
        __syncthreads();
        if (tid < kGroupMembers) {
            int m = 0;
            if (tid < nm)
                for (int i = 0; i < (rrec[tid] >> 8); ++i) m = max(m, rmax[(rrec[tid] & 255) + i]);
            P.mexp[t * kGroupMembers + tid] = m ? (int16_t)(m - 1022) : kNoExp;
        }
        uint8_t* base = P.pack + t * P.KS * (int64_t)(2 * kDigits * 16) * P.R;
        for (int u = tid; u < units; u += 256) {
            const int c = u / P.R, r = u - c * P.R;
            if (!((km >> (c >> 1)) & 1u)) continue;
            const int a = rmem[r];
            const int em = rmax[r];
            uint32_t w[kDigits][4];
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                float d[kDigits][2];
#pragma unroll
                for (int y = 0; y < 2; ++y) {
                    const uint64_t bits = load(r, a, 8 * c + 2 * x + y);
                    const int be = (int)(bits >> 52) & 0x7ff;
                    const bool neg = (bits >> 63) != 0;
                    const uint64_t M = (bits & 0xfffffffffffffull) | (1ull << 52);
                    const int rs = em - be - 10;                     // |x| 2^(63 - e) = M / 2^rs
                    uint64_t v = 0;                                  // (subnormal elements count as zero)
                    if (be) v = rs <= 0 ? M << (-rs) : rs <= 54 ? (M + (1ull << (rs - 1))) >> rs : 0;
                    if (neg) v = 0ull - v;
                    // adding 128 to each of the low seven digits makes them plain bytes
                    v += 0x0080808080808080ull;
                    const int top = (int)(v >> 56);
                    d[0][y] = (float)(neg ? (int)(int8_t)top : top);
#pragma unroll
                    for (int s = 1; s < kDigits; ++s)
                        d[s][y] = __uint_as_float(0x4B000000u | ((uint32_t)(v >> (56 - 8 * s)) & 255u)) - 8388736.0f;
                }
#pragma unroll
                for (int s = 0; s < kDigits; ++s)                    // exact in BF16: the upper halves
                    w[s][x] = __byte_perm(__float_as_uint(d[s][0]), __float_as_uint(d[s][1]), 0x7632);
            }
            uint4* o = reinterpret_cast<uint4*>(base + ((int64_t)c * kDigits * P.R + r) * 16);
#pragma unroll
            for (int s = 0; s < kDigits; ++s) o[(int64_t)s * P.R] = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------ which blocks
// Executed flops of every C tile's blocks (the FP64 pipe's alternative).
__global__ void k_oz_tile_flops(int64_t nform, const int32_t* __restrict__ blk_tile, const int32_t* __restrict__ f_row,
                                const int32_t* __restrict__ f_col, const int32_t* __restrict__ f_ksum,
                                const int32_t* __restrict__ bs, unsigned long long* __restrict__ flops) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nform; k += (int64_t)gridDim.x * blockDim.x) {
        const int32_t t = blk_tile[k];
        if (t >= 0)
            atomicAdd(flops + t, 2ull * (unsigned long long)(bs[f_row[k]] * bs[f_col[k]]) * (unsigned long long)f_ksum[k]);
    }
}

struct OzGuardArgs {
    int64_t nform;
    const int32_t* blk_tile; const int32_t* f_row; const int32_t* f_col;
    const int32_t* g_midx; const int32_t* g_w; const int32_t* c_tcol;
    const int64_t* s_ptr; const int32_t* st_a; const int32_t* st_b;
    const int16_t* a_mexp; const int16_t* b_mexp;
    const float* f_max;                              // largest |alpha| ||A_IK|| ||B_KJ|| of every block
    const int32_t* f_at;                             // and which block of A's row I that is
    const unsigned long long* tile_flops;
    float abs_alpha;
    const int* bad;
    int16_t* f_exp;                                  // k_oz_guard to k_oz_weak: exponent of the block's scale
    uint8_t* comp;
    int32_t* c_tbl; int16_t* c_exp; unsigned* c_slices;
    const int32_t* g_pos; const int32_t* bs;
    const int64_t* a_rp; const int32_t* a_col; const int64_t* a_off; const double* a_data;
    const int64_t* b_rp; const int32_t* b_col; const int64_t* b_off; const double* b_data;
};

__device__ __forceinline__ bool oz_pays(int64_t entries, int width, unsigned long long flops) {
    const int slices = (width + kSlice - 1) / kSlice;
    return (double)entries * (kGroupWidth / 16) * slices * kStepClocks * kSimtFlopsPerClock <= (double)flops;
}
// Flops of the tiles for which the tensor cores pay.
__global__ void k_oz_pays(int64_t nt, const int64_t* __restrict__ s_ptr, const int32_t* __restrict__ c_tcol,
                          const int32_t* __restrict__ g_w, const unsigned long long* __restrict__ flops,
                          unsigned long long* __restrict__ sum) {
    unsigned long long f = 0;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nt; t += (int64_t)gridDim.x * blockDim.x)
        if (oz_pays(s_ptr[t + 1] - s_ptr[t], g_w[c_tcol[t]], flops[t])) f += flops[t];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
    if ((threadIdx.x & 31) == 0 && f) atomicAdd(sum, f);
}
// Without such tiles nothing is packed.  Nor is it, in a product that need not take the same path in a batch
// (weigh), when packing the operands' tiles takes longer than the FP64 pipe needs for those blocks: tiles of a
// pattern without neighbourhoods hold a block or two each in 200 KB of digits, of which a quarter or less (the K
// steps in use) is written at 4 TB/s (3,000 blocks of 13 with 20 random ones a row: 16.9 ms with the tiles, for a
// few of its 5.8 GF, 12.8 without, 11.0 if the blocks need not be grouped).
constexpr double kPackBytesPerSecond = 16e12, kSimtFlopsPerSecond = 1e12;

// A computed block runs on the tensor cores (comp = 2) unless
//   * its tile's tensor-core time (every stack entry at full width; a rule on the tile alone, so
//     a block takes the same path in any batch) is above the FP64 pipe's time for its blocks;
//   * the largest product of its tile rows' scales, max 2^(e_a + e_b), is at least 2^7 times its
//     largest norm product (Frobenius error of a block in units of the FP64 chain's, root mean square over
//     water products, emulated: 0.1 below 2^4, 0.4 to 0.9 at 2^6 to 2^7, 0.7 to 1.5 above, 1.7 at 2^8);
//   * its weakest element is too far below those scales (k_oz_weak);
//   * an operand holds a value outside the scales' range.
// The blocks that both rules send back cost the FP64 pipe's rate: the sign iteration on 512 waters takes
// 245 ms with them, 204 with 2^8 and no rule on elements, 222 with 2^8 and 2^-14, 239 with 2^8 and 2^-13.
constexpr float kNormRatio = 0.0078125f;             // 2^-7
constexpr int kWeakBits = 13;
constexpr int kNoTerm = -4096;                       // exponent of a block all of whose products are zero
__global__ void k_oz_guard(OzGuardArgs A) {
    const bool bad = *A.bad != 0;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < A.nform; k += (int64_t)gridDim.x * blockDim.x) {
        A.f_exp[k] = kNoExp;                          // FP64 pipe
        const int32_t t = A.blk_tile[k];
        if (bad || t < 0) continue;
        const int64_t e0 = A.s_ptr[t], e1 = A.s_ptr[t + 1];
        if (!oz_pays(e1 - e0, A.g_w[A.c_tcol[t]], A.tile_flops[t])) continue;
        const int a = A.g_midx[A.f_row[k]], b = A.g_midx[A.f_col[k]];
        int E = 2 * kNoExp;
        for (int64_t e = e0; e < e1; ++e)
            E = max(E, (int)A.a_mexp[(int64_t)A.st_a[e] * kGroupMembers + a] +
                           (int)A.b_mexp[(int64_t)A.st_b[e] * kGroupMembers + b]);
        // (a norm product near the ends of FP32's range, or past them, says nothing: FP64 pipe; below, it is
        // rounded up to a denormal while the scales' product underflows to 0)
        if (E > kNoExp / 2 &&
            !(ldexpf(A.abs_alpha, E) * kNormRatio < A.f_max[k] && A.f_max[k] >= 1e-30f && A.f_max[k] <= 3e38f))
            continue;
        A.f_exp[k] = (int16_t)max(E, kNoTerm);
    }
}

// n elements of a block as floats |x| 2^-e, e the exponent above the largest (returned), cut to 21 bits: by
// the high words, since the FP64 pipe converts a few values per clock and SM.
__device__ __forceinline__ int oz_abs(const double* __restrict__ x, int n, int lane, float* out) {
    unsigned mx = 0;
    for (int e = lane; e < n; e += 32) {
        const unsigned hi = __ldg(reinterpret_cast<const unsigned*>(x + e) + 1) & 0x7fffffffu;
        out[e] = __uint_as_float(hi);
        mx = max(mx, hi >> 20);
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    for (int e = lane; e < n; e += 32) {              // (each lane its own elements)
        const int v = (int)__float_as_uint(out[e]) - (((int)mx - 126) << 20);
        out[e] = v >= (1 << 20) ? __int_as_float(v << 3) : 0.f;
    }
    return (int)mx - 1022;
}

// Whether every element of |A_IK| |B_KJ| is at least 2^(E - bits) (one warp; sh: two blocks).
__device__ __forceinline__ bool oz_no_weak(const double* a, const double* b, int m, int kk, int n, int E, int bits,
                                           int lane, float (*sh)[kMaxBlock * kMaxBlock]) {
    __syncwarp();                                     // the last block's elements are read
    const int ea = oz_abs(a, m * kk, lane, sh[0]), eb = oz_abs(b, kk * n, lane, sh[1]);
    __syncwarp();
    float low = 3e38f;
    for (int e = lane; e < m * n; e += 32) {
        const int i = e / n, j = e - i * n;
        float s = 0.f;
        for (int t = 0; t < kk; ++t) s = fmaf(sh[0][i * kk + t], sh[1][t * n + j], s);
        low = fminf(low, s);
    }
    low = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(low)));
    const int x = E - bits - ea - eb;                 // at least -bits: 2^E is a scale product of the same rows
    return x < 100 && low >= ldexpf(1.f, x);
}

// The blocks that k_oz_guard lets through, one warp each: their strongest block product without signs is a
// lower bound of sum_k |a_ik| |b_kj| for every element, 8 times below it on water in the median.  Bound by the
// loads of the two operand blocks and 2 m n k / 32 shared-memory reads a block.
constexpr int kWeakWarps = 4;
__global__ void __launch_bounds__(32 * kWeakWarps) k_oz_weak(OzGuardArgs A) {
    __shared__ float sh[kWeakWarps][2][kMaxBlock * kMaxBlock];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t k = (int64_t)blockIdx.x * kWeakWarps + warp; k < A.nform; k += (int64_t)gridDim.x * kWeakWarps) {
        const int E = A.f_exp[k];
        if (E == kNoExp) continue;
        const int32_t t = A.blk_tile[k], I = A.f_row[k], J = A.f_col[k];
        if (E > kNoTerm) {
            const int64_t p = A.a_rp[I] + A.f_at[k];
            const int32_t K = A.a_col[p];
            int64_t lo = A.b_rp[K], hi = A.b_rp[K + 1];
            const int64_t end = hi;
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                if (A.b_col[mid] < J) lo = mid + 1; else hi = mid;
            }
            if (!(lo < end && A.b_col[lo] == J)) continue;
            if (!oz_no_weak(A.a_data + A.a_off[p], A.b_data + A.b_off[lo], A.bs[I], A.bs[K], A.bs[J], E, kWeakBits, lane,
                            sh[warp]))
                continue;
        }
        if (lane == 0) {
            const int64_t at = (int64_t)t * (kGroupMembers * kGroupMembers) + A.g_midx[I] * kGroupMembers + A.g_midx[J];
            A.comp[k] = 2;
            A.c_tbl[at] = (int32_t)k;
            A.c_exp[at] = (int16_t)E;
            unsigned m = 0;
            for (int q = A.g_pos[J] / kSlice; q <= (A.g_pos[J] + A.bs[J] - 1) / kSlice; ++q) m |= 1u << q;
            atomicOr(A.c_slices + t, m);
        }
    }
}

// Digits per stack entry and slice.  A tile product whose scales lie 2^d below those of every block
// the slice writes may drop the last digits: with 8 - w digits its error grows by 2^(8 w), which
// stays under that of the largest tile product for 8 w <= d - kDepthMargin (the margin for the sum
// over the entries).  Far tiles need few digits (on water half of the digit products go), and an
// entry that needs none leaves the slice's mask (the K steps that both tiles hold in that slice).
// One warp per C tile, lanes over its 256 members.
constexpr int kDepthMargin = 3;
struct OzDepthArgs {
    int64_t ntiles;
    const int32_t* c_tcol; const int32_t* g_ptr; const int32_t* g_mrec;
    const int64_t* s_ptr; const int32_t* st_a; const int32_t* st_b;
    const int16_t* a_mexp; const int16_t* b_mexp;
    const int32_t* c_tbl; const int16_t* c_exp;
    const unsigned* a_sm; const unsigned* b_sm;
    int4* ent;                                       // per entry: A tile, B tile, K steps, digits (8 bits per slice)
};
__global__ void __launch_bounds__(256) k_oz_depth(OzDepthArgs A) {
    constexpr int kPer = kGroupMembers * kGroupMembers / 32;
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    // lane l holds the member pairs (2 u + (l >> 4), l & 15)
    const int b = lane & 15, a0 = lane >> 4;
    for (int64_t t = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < A.ntiles; t += warps) {
        int ex[kPer];
        bool any = false;
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const int64_t p = t * (kGroupMembers * kGroupMembers) + 32 * u + lane;
            ex[u] = A.c_tbl[p] >= 0 ? (int)A.c_exp[p] : 1 << 20;
            any |= ex[u] < (1 << 20);
        }
        unsigned cols = 0;                            // slices that column member b lies in
        {
            const int n0 = A.g_ptr[A.c_tcol[t]], nn = A.g_ptr[A.c_tcol[t] + 1] - n0;
            if (b < nn) {
                const int mr = A.g_mrec[n0 + b], p = mr & 255, w = mr >> 8;
                for (int q = p / kSlice; q <= (p + w - 1) / kSlice; ++q) cols |= 1u << q;
            }
        }
        if (!__any_sync(0xffffffffu, any)) continue;
        for (int64_t e = A.s_ptr[t]; e < A.s_ptr[t + 1]; ++e) {
            const int16_t* pa = A.a_mexp + (int64_t)A.st_a[e] * kGroupMembers;
            const int eb = A.b_mexp[(int64_t)A.st_b[e] * kGroupMembers + b];
            int d = 1 << 20;
#pragma unroll
            for (int u = 0; u < kPer; ++u) {
                const int ea = pa[2 * u + a0];
                if (ex[u] < (1 << 20) && ea != kNoExp && eb != kNoExp) d = min(d, ex[u] - ea - eb);
            }
            const int32_t ta = A.st_a[e], tb = A.st_b[e];
            unsigned m = A.b_sm[tb] & (fold8(A.a_sm[ta]) * 0x01010101u), nd4 = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int dq = __reduce_min_sync(0xffffffffu, (cols >> q) & 1u ? d : 1 << 20);
                const int nd = kDigits - min(kDigits, max(0, dq - kDepthMargin) >> 3);
                if (!nd) m &= ~(255u << (8 * q));
                nd4 |= (unsigned)nd << (8 * q);
            }
            if (lane == 0) A.ent[e] = make_int4(ta, tb, (int)m, (int)nd4);
        }
    }
}

// ------------------------------------------------------------------ the tensor-core kernel
struct OzMaps {
    CUtensorMap m[kDigits];                          // boxes of 1 .. 8 digits of a B slice
};

struct OzArgs {
    int64_t nitems;                                  // C tiles x slices
    int nsl, R, KS;
    const int32_t* c_trow; const int32_t* c_tcol; const int64_t* s_ptr; const unsigned* c_slices;
    const int4* ent;                                 // per stack entry: A tile, B tile, K steps, digits
    const uint8_t* a_pack;
    const int16_t* a_rexp; const int16_t* b_rexp;
    const int32_t* g_ptr; const int32_t* g_mrec;
    const int32_t* c_tbl; const int16_t* c_exp;      // per C tile, 16 x 16: block, exponent of its scale
    const int64_t* f_off; const int64_t* f_cin;
    const int64_t* ci_off; const double* ci_data;
    double alpha, beta;
    double* c_data;
    int* flags;
    unsigned long long* next;                        // the work items' counter
};

struct OzShared {
    alignas(1024) uint8_t stage[kOzStages][kOzStage];
    int64_t koff[kGroupMembers][kGroupMembers];      // element offset of the block, -1: not written
    int64_t kcin[kGroupMembers][kGroupMembers];      // element offset of its C input, -1: none
    int kexp[kGroupMembers][kGroupMembers];          // exponent of its scale
    int colrec[kSlice];                              // member | column inside it << 8 | its width << 16; -1
    int rowrec[128];                                 // member | row inside it << 8; -1
    int64_t item[kOzItems];
    uint64_t item_full[kOzItems], item_empty[kOzItems];
    uint64_t full[kOzStages], empty[kOzStages], acc_full[2], acc_empty[2], fin;
    uint32_t tmem_base;
    int abort, epi_stop;
};

__device__ __forceinline__ void oz_epi_sync() { asm volatile("bar.sync 1, %0;" ::"n"(32 * kOzEpiWarps) : "memory"); }

__device__ __forceinline__ void oz_fail(const OzArgs& A, OzShared& S) {
    *(volatile int*)&S.abort = 1;
    atomicExch(A.flags + kFlagFailed, 1);
}
__device__ __forceinline__ int oz_aborted(const OzShared& S) { return *(volatile const int*)&S.abort; }

// A 96-bit two's-complement sum.
struct Oz96 {
    uint32_t l;
    int64_t h;
};

// acc += (sum_d v[d] 2^(8 (7 - d))) >> sh over the first ND digits' accumulators, 0 <= sh <= 95.  v[d] is an integer of at most (d + 1) * 112 * 2^14 in magnitude.  Adding 1.5 * 2^23
// leaves v[0] and v[1] (below 2^22) in the low bits; v[6] and v[7] are taken to a multiple of 4, far
// below the digits that are not summed; the other four go through the conversion unit (a sixteenth
// of the issue rate: it would bound the epilogue with all eight).
template <int ND>
__device__ __forceinline__ void oz_add(Oz96& acc, const float* v, int sh) {
    const int q = __float_as_int(v[0] + 12582912.0f) * 256 + __float_as_int(v[1] + 12582912.0f) - (int)(0x4B400000u * 257u);
    const int p = __float2int_rn(v[2]) * 256 + __float2int_rn(v[3]);
    uint32_t w0 = 0u, w1, w2;
    if (ND > 4) {
        int64_t lo = (int64_t)__float2int_rn(v[5]) * 65536ll;
        if (ND > 6) {
            const int r = __float_as_int(v[6] + 50331648.0f) * 256 + __float_as_int(v[7] + 50331648.0f) -
                          (int)(0x4C400000u * 257u);
            lo += (int64_t)r * 4ll;
        }
        lo += (int64_t)__float2int_rn(v[4]) * 16777216ll;
        const int64_t hi = (int64_t)q * 65536ll + ((int64_t)p + (lo >> 32));
        w0 = (uint32_t)lo;
        w1 = (uint32_t)hi;
        w2 = (uint32_t)(hi >> 32);
    } else {
        const int64_t hi = (int64_t)q * 65536ll + (int64_t)p;
        w1 = (uint32_t)hi;
        w2 = (uint32_t)(hi >> 32);
    }
    const uint32_t sg = (uint32_t)((int32_t)w2 >> 31);
    if (sh >= 32) {
        w0 = w1;
        w1 = w2;
        w2 = sg;
    }
    if (sh >= 64) {
        w0 = w1;
        w1 = sg;
    }
    w0 = __funnelshift_r(w0, w1, sh);
    w1 = __funnelshift_r(w1, w2, sh);
    w2 = (uint32_t)((int32_t)w2 >> (sh & 31));
    uint32_t h0 = (uint32_t)acc.h, h1 = (uint32_t)((uint64_t)acc.h >> 32);
    asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
        : "+r"(acc.l), "+r"(h0), "+r"(h1)
        : "r"(w0), "r"(w1), "r"(w2));
    acc.h = (int64_t)(((uint64_t)h1 << 32) | h0);
}

// x 2^sc rounded to FP64.
__device__ __forceinline__ double oz_value(const Oz96& x, int sc) {
    uint32_t l = x.l;
    int64_t hi = x.h;
    const bool neg = hi < 0;
    if (neg) {
        l = 0u - l;
        hi = ~hi + (l == 0u ? 1 : 0);
    }
    uint32_t h1 = (uint32_t)((uint64_t)hi >> 32), h0 = (uint32_t)hi;
    int e = 1023 + 95 + sc;
    for (int x2 = 0; x2 < 2; ++x2)
        if (h1 == 0u) {                              // leading word zero: up by a word
            h1 = h0;
            h0 = l;
            l = 0u;
            e -= 32;
        }
    if (h1 == 0u) return 0.0;
    const int n = __clz((int)h1);
    const uint64_t w = ((uint64_t)__funnelshift_l(h0, h1, n) << 32) | __funnelshift_l(l, h0, n);   // leading bit at 63
    const uint64_t bits = ((uint64_t)(uint32_t)(e - n - 1) << 52) + (w >> 11) + ((w >> 10) & 1u);
    return __longlong_as_double((long long)(bits | ((uint64_t)neg << 63)));
}

// 2 consecutive 32-bit columns of one TMEM lane per thread, not waited for.
__device__ __forceinline__ void oz_ld2(uint32_t taddr, float* v) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=f"(v[0]), "=f"(v[1]) : "r"(taddr));
}
// The loaded registers are passed through, so that no use of them moves above the wait.
template <int ND>
__device__ __forceinline__ void oz_ld_wait(float (*v)[2]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int d = 0; d < ND; ++d)
#pragma unroll
        for (int x = 0; x < 2; ++x) asm volatile("" : "+f"(v[d][x]));
}

// A box of a 4-D tensor map into shared memory.
__device__ __forceinline__ void oz_tma4(void* dst, const void* tmap, int c0, int c1, int c2, int c3, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];" ::"r"(tc::smem_u32(dst)),
        "l"(tmap), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(tc::smem_u32(bar))
        : "memory");
}

// The MMAs of one K step with ND digits.  Digit s of A times digits 0 .. ND - 1 - s of the B slice
// (the N dimension, one digit after the other) lands in accumulators s .. ND - 1.  MMAs that
// overlap in tensor memory at another first column wait for each other (about 110 clocks each,
// measured), so up to six digits all MMAs write all ND accumulators, with zero digit blocks before
// digit 0 standing in for the pairs that do not exist.  With seven and eight digits, where that would cost 784 and
// 1,024 clocks (an MMA takes N / 2 clocks, at least 66), there are two groups, s < 4 with all accumulators and
// s >= 4 with the last ND - 4: 776 clocks by the MMAs' own times at eight digits, 797 measured with nothing
// beside them.
// al, bl: the low words of the operands' descriptors at A's digit 0 and at the first zero block of B
// (start address and chunk distance); the high words hold the constant 128 bytes between 8-row
// groups.
// FIRST: the first K step of a tile product (digit 0 overwrites the accumulators).
template <int ND, bool FIRST>
__device__ __forceinline__ void oz_mmas(uint32_t d, uint32_t al, uint32_t a_step, uint32_t bl) {
    constexpr int h = ND >= 7 ? 4 : ND;
    constexpr uint64_t hi = ((uint64_t)(128 >> 4) << 32) | ((uint64_t)1 << 46);
    static_assert(kZeroBlocks >= kDigits - 2, "zero blocks for every shift of B");
    tc::mma_f16_acc<!FIRST>(d, hi | al, hi | (bl + (uint32_t)(kZeroBlocks * (kDigitBlock / 16))),
                            tc::instr_desc(1, 128, kSlice * ND));
#pragma unroll
    for (int s = 1; s < ND; ++s) {
        const int c0 = s < h ? 0 : h;                 // first accumulator
        tc::mma_f16_acc<true>(d + (uint32_t)(c0 * kSlice), hi | (al + (uint32_t)s * a_step),
                              hi | (bl + (uint32_t)((kZeroBlocks + c0 - s) * (kDigitBlock / 16))),
                              tc::instr_desc(1, 128, kSlice * (s < h ? ND : ND - h)));
    }
}
template <bool FIRST>
__device__ __forceinline__ void oz_issue(int nd, uint32_t d, uint32_t al, uint32_t a_step, uint32_t bl) {
    switch (nd) {
        case 8: oz_mmas<8, FIRST>(d, al, a_step, bl); break;
        case 7: oz_mmas<7, FIRST>(d, al, a_step, bl); break;
        case 6: oz_mmas<6, FIRST>(d, al, a_step, bl); break;
        case 5: oz_mmas<5, FIRST>(d, al, a_step, bl); break;
        case 4: oz_mmas<4, FIRST>(d, al, a_step, bl); break;
        case 3: oz_mmas<3, FIRST>(d, al, a_step, bl); break;
        case 2: oz_mmas<2, FIRST>(d, al, a_step, bl); break;
        default: oz_mmas<1, FIRST>(d, al, a_step, bl); break;
    }
}

// One finished tile product into this thread's 8 elements: accumulators of nd (at most ND) digits at
// taddr, the elements' scales ex against the row's exponent ea and the columns' in ew.  free: the
// barrier of the accumulator buffer, arrived on once every value is in registers.
template <int ND>
__device__ __forceinline__ void oz_take(int nd, Oz96* acc, const int* ex, int ea, const int* ew, uint32_t taddr,
                                        uint64_t* free, int lane) {
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        float v[ND][2];
#pragma unroll
        for (int d = 0; d < ND; ++d) {
            if (d < nd) oz_ld2(taddr + (uint32_t)(d * kSlice + 2 * g), v[d]);
            else v[d][0] = v[d][1] = 0.f;
        }
        oz_ld_wait<ND>(v);
        if (g == 3) {                                 // all of it is in registers: the buffer is free
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(free);
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int x = j ? ex[g] >> 16 : (int)(int16_t)(ex[g] & 0xffff);
            const int w = j ? ew[g] >> 16 : (int)(int16_t)(ew[g] & 0xffff);
            const int sh = min(max(x - ea - w, 0), 95);
            float c[ND];
#pragma unroll
            for (int d = 0; d < ND; ++d) c[d] = v[d][j];
            oz_add<ND>(acc[2 * g + j], c, sh);
        }
    }
}

// A warp's next work item (-1: none, or a wait ran out), from the ring the producer fills.
__device__ __forceinline__ int64_t oz_item(const OzArgs& A, OzShared& S, uint32_t n, int lane) {
    const int slot = (int)(n % kOzItems);
    const bool ok = __all_sync(0xffffffffu, tc::mbar_wait(&S.item_full[slot], (n / kOzItems) & 1u, kOzWait));
    if (!ok && lane == 0) oz_fail(A, S);
    const int64_t it = ok && !oz_aborted(S) ? *(volatile const int64_t*)&S.item[slot] : -1;
    return __shfl_sync(0xffffffffu, it, 0);
}
__device__ __forceinline__ void oz_item_done(OzShared& S, uint32_t n, int lane) {
    __syncwarp();
    if (lane == 0) tc::mbar_arrive(&S.item_empty[n % kOzItems]);
}

// One persistent CTA per SM over the work items (C tile, 32-column slice), taken from a global
// counter in order, so that the CTAs running at one time share the A tiles of a few group rows in
// L2, and handed from the producer to the other warps through a small ring (the items' costs
// differ several times: fixed shares left the SMs busy 76% of the time).  Warp 0 streams the K
// steps (A by bulk copies, the B slice through a tensor map) into a ring of stages, warp 1
// issues the MMAs, warps 2-17 combine a finished tile product's accumulators while the next one is
// multiplied.
// 64 registers a thread (a few spills outside the inner loop; 4% slower alone than with 96) leave room for
// 12 and more warps of the FP64 pipe's kernels on the SM: together they finish 16 to 20% sooner than one
// after the other.  For this the accumulators come two columns at a time and the scales' exponents are
// held in pairs; with 96 registers nothing ran beside it, with 80 a third of the gain was there.
__global__ void __maxnreg__(64) k_oz(const __grid_constant__ OzMaps maps, OzArgs A) {
    extern __shared__ __align__(1024) uint8_t oz_dyn[];
    OzShared& S = *reinterpret_cast<OzShared*>((reinterpret_cast<uintptr_t>(oz_dyn) + 1023) & ~(uintptr_t)1023);
    // (a planned product whose blocks the FP64 pipe forms: all of them for these values, or the self-test's)
    if (A.flags[kFlagRange] || A.flags[kFlagFailed] == 1) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < kOzStages * 2 * kZeroBlocks * (kDigitBlock / 16); i += kOzThreads) {
        const int per = kZeroBlocks * (kDigitBlock / 16);
        const int st = i / (2 * per), ch = (i / per) & 1, x = i % per;
        *reinterpret_cast<uint4*>(S.stage[st] + kOzA + ch * kOzBChunk + 16 * x) = make_uint4(0, 0, 0, 0);
    }
    if (threadIdx.x == 0) {
        for (int i = 0; i < kOzStages; ++i) {
            tc::mbar_init(&S.full[i], 1);
            tc::mbar_init(&S.empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&S.acc_full[i], 1);
            tc::mbar_init(&S.acc_empty[i], kOzEpiWarps);
        }
        for (int i = 0; i < kOzItems; ++i) {
            tc::mbar_init(&S.item_full[i], 1);
            tc::mbar_init(&S.item_empty[i], 1 + kOzEpiWarps);
        }
        tc::mbar_init(&S.fin, 1);
        S.abort = 0;
        S.epi_stop = 0;
        tc::fence_barrier_init();
    }
    if (warp == 1) {
        tc::tmem_alloc(&S.tmem_base, kOzTmem);
        tc::tmem_relinquish();
    }
    tc::fence_proxy_async();                          // the zero blocks, for the tensor cores
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = S.tmem_base;
    const int a_bytes = 2 * kDigits * 16 * A.R;

    if (warp == 0) {
        // ---------------- producer (lane 0)
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0, n = 0;
            int64_t armed = 0;
            int64_t ahead = (int64_t)atomicAdd(A.next, 1ull);     // the item after this one, fetched early
            bool ok = true;
            while (ok) {
                const int64_t it = ahead;
                if (it < A.nitems) ahead = (int64_t)atomicAdd(A.next, 1ull);
                const int64_t t = it < A.nitems ? it / A.nsl : 0;
                const int q = (int)(it - t * A.nsl);
                if (it < A.nitems && !((A.c_slices[t] >> q) & 1u)) continue;
                const int slot = (int)(n % kOzItems);
                if (!tc::mbar_wait(&S.item_empty[slot], ((n / kOzItems) & 1u) ^ 1u, kOzWait)) oz_fail(A, S);
                S.item[slot] = it < A.nitems && !oz_aborted(S) ? it : -1;
                tc::mbar_arrive(&S.item_full[slot]);  // releases the item to the other warps
                ++n;
                if (it >= A.nitems || oz_aborted(S)) break;
                const int64_t e1 = A.s_ptr[t + 1];
                int64_t e = A.s_ptr[t];
                int4 nx = e < e1 ? __ldg(A.ent + e) : make_int4(0, 0, 0, 0);
                for (; e < e1 && ok; ++e) {
                    const int4 en = nx;
                    if (e + 1 < e1) nx = __ldg(A.ent + e + 1);
                    unsigned mask = ((unsigned)en.z >> (8 * q)) & 255u;
                    if (!mask) continue;
                    const int nd = (int)(((unsigned)en.w >> (8 * q)) & 255u);
                    const uint32_t ac = (uint32_t)(nd * A.R * 16);            // digits of one chunk of A
                    const uint32_t tx = 2u * ac + (uint32_t)(2 * nd * kDigitBlock);
                    const CUtensorMap* map_b = &maps.m[nd - 1];
                    const uint8_t* pa = A.a_pack + (int64_t)en.x * A.KS * a_bytes;
                    do {
                        const int k = __ffs(mask) - 1;
                        mask &= mask - 1;
                        if (!tc::mbar_wait(&S.empty[stage], phase ^ 1u, kOzWait)) {
                            oz_fail(A, S);
                            ok = false;
                            break;
                        }
                        uint8_t* sa = S.stage[stage];
                        uint8_t* sb = sa + kOzA + kZeroBlocks * kDigitBlock;
                        uint64_t* bar = &S.full[stage];
                        const uint8_t* src = pa + k * a_bytes;
                        tc::mbar_arrive_expect_tx(bar, tx);
                        tc::bulk_g2s(sa, src, ac, bar);
                        tc::bulk_g2s(sa + a_bytes / 2, src + a_bytes / 2, ac, bar);
                        oz_tma4(sb, map_b, q * kSlice * 8, 0, 0, en.y * A.KS + k, bar);
                        oz_tma4(sb + kOzBChunk, map_b, q * kSlice * 8, 0, 1, en.y * A.KS + k, bar);
                        ++armed;
                        if (++stage == kOzStages) {
                            stage = 0;
                            phase ^= 1u;
                        }
                    } while (mask);
                }
            }
            // no copy may still be landing in shared memory when the CTA exits
            for (int64_t x = 0; x < armed && x < kOzStages; ++x) {
                if (--stage < 0) {
                    stage = kOzStages - 1;
                    phase ^= 1u;
                }
                if (!tc::mbar_wait(&S.full[stage], phase, kOzWait)) oz_fail(A, S);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- MMA issuer: the whole warp, every lane with the same values (elect_one)
        int stage = 0;
        uint32_t phase = 0, n = 0;                    // n: tile products started
        const uint32_t a_step = (uint32_t)A.R, a_lbo = (uint32_t)(kDigits * A.R) << 16;     // in 16-byte units
        const uint32_t s0 = tc::smem_u32(S.stage[0]) >> 4;
        bool ok = true;
        for (uint32_t ni = 0; ok; ++ni) {
            const int64_t it = oz_item(A, S, ni, lane);
            if (it < 0) break;
            oz_item_done(S, ni, lane);
            const int64_t t = it / A.nsl;
            const int qs = 8 * (int)(it - t * A.nsl);
            const int64_t e1 = A.s_ptr[t + 1];
            int64_t e = A.s_ptr[t];
            int4 nx = e < e1 ? __ldg(A.ent + e) : make_int4(0, 0, 0, 0);
            for (; e < e1 && ok; ++e) {
                const int4 en = nx;
                if (e + 1 < e1) nx = __ldg(A.ent + e + 1);
                unsigned mask = tc::uniform(((unsigned)en.z >> qs) & 255u);
                if (!mask) continue;
                const int nd = (int)tc::uniform(((unsigned)en.w >> qs) & 255u);
                const uint32_t buf = n & 1u;
                const uint32_t d = tc::uniform(tmem + buf * 256u);
                bool mine = tc::mbar_wait(&S.acc_empty[buf], ((n >> 1) & 1u) ^ 1u, kOzWait);
                // two K steps at a time where there are two: an MMA's issue waits until the tensor cores
                // are nearly through with the ones before it, so what lies between two batches of
                // MMAs leaves them idle
                bool first = true;
                while (mask) {
                    const int st0 = stage, st1 = stage + 1 == kOzStages ? 0 : stage + 1;
                    mask &= mask - 1;
                    const bool two = mask != 0;
                    const uint32_t sa0 = tc::uniform(s0 + (uint32_t)st0 * (kOzStage / 16));
                    const uint32_t sa1 = tc::uniform(s0 + (uint32_t)st1 * (kOzStage / 16));
                    mine = mine && tc::mbar_wait(&S.full[st0], phase, kOzWait);
                    if (two) mine = mine && tc::mbar_wait(&S.full[st1], phase ^ (st1 == 0 ? 1u : 0u), kOzWait);
                    mask &= mask - 1;
                    tc::fence_after_sync();
                    constexpr uint32_t b_off = kOzA / 16, b_lbo = (uint32_t)(kOzBChunk / 16) << 16;
                    if (tc::elect_one() && mine) {
                        if (first) oz_issue<true>(nd, d, sa0 | a_lbo, a_step, (sa0 + b_off) | b_lbo);
                        else oz_issue<false>(nd, d, sa0 | a_lbo, a_step, (sa0 + b_off) | b_lbo);
                        tc::mma_commit(&S.empty[st0]);
                        if (two) {
                            oz_issue<false>(nd, d, sa1 | a_lbo, a_step, (sa1 + b_off) | b_lbo);
                            tc::mma_commit(&S.empty[st1]);
                        }
                        if (!mask) tc::mma_commit(&S.acc_full[buf]);
                    }
                    __syncwarp();
                    first = false;
                    stage += two ? 2 : 1;
                    if (stage >= kOzStages) {
                        stage -= kOzStages;
                        phase ^= 1u;
                    }
                }
                // the lanes stay together, see mbar_wait_warp: one whose wait ran out only stops issuing until here
                // (a vote before the MMAs of every step took the kernel 2% longer, one behind them 1%)
                ok = __all_sync(0xffffffffu, mine);
                ++n;
            }
            if (!ok && lane == 0) oz_fail(A, S);
        }
        // every MMA has completed before the TMEM is released
        if (tc::elect_one()) tc::mma_commit(&S.fin);
        __syncwarp();
        if (!tc::mbar_wait(&S.fin, 0, kOzWait) && lane == 0) oz_fail(A, S);
        __syncwarp();
    } else {
        // ---------------- epilogue: the warp's TMEM lanes 32 (warp % 4) .., 8 columns of the slice
        const int et = threadIdx.x - 32 * kOzEpi0;
        const int quad = warp & 3, part = et >> 7;
        const int r = 32 * quad + lane;
        const uint32_t lane_base = tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)(8 * part);
        uint32_t n = 0;
        for (uint32_t ni = 0;; ++ni) {
            int64_t it = oz_item(A, S, ni, lane);
            // the tables of this item: its blocks and which block every column and row belongs to
            oz_epi_sync();                            // the last item's tables are no longer read
            if (et == 0) S.epi_stop = it < 0 || oz_aborted(S);
            const int64_t t = it < 0 ? 0 : it / A.nsl;
            const int q = it < 0 ? 0 : (int)(it - t * A.nsl);
            const int32_t G = A.c_trow[t], Gc = A.c_tcol[t];
            if (et < kGroupMembers * kGroupMembers) {
                const int32_t k = A.c_tbl[t * (kGroupMembers * kGroupMembers) + et];
                const int64_t ci = (k >= 0 && A.f_cin) ? A.f_cin[k] : -1;
                S.koff[et >> 4][et & 15] = k >= 0 ? A.f_off[k] : -1;
                S.kcin[et >> 4][et & 15] = ci >= 0 ? A.ci_off[ci] : -1;
                S.kexp[et >> 4][et & 15] = k >= 0 ? (int)A.c_exp[t * (kGroupMembers * kGroupMembers) + et] : 4096;
            } else if (et - kGroupMembers * kGroupMembers < kSlice) {
                const int x = et - kGroupMembers * kGroupMembers;
                const int c = q * kSlice + x, n0 = A.g_ptr[Gc], nn = A.g_ptr[Gc + 1] - n0;
                int rec = -1;
                for (int b = 0; b < nn; ++b) {
                    const int mr = A.g_mrec[n0 + b], p = mr & 255, w = mr >> 8;
                    if (c >= p && c < p + w) rec = b | ((c - p) << 8) | (w << 16);
                }
                S.colrec[x] = rec;
            }
            if (et >= kGroupMembers * kGroupMembers + 128) {
                const int x = et - kGroupMembers * kGroupMembers - 128;
                const int m0 = A.g_ptr[G], nm = A.g_ptr[G + 1] - m0;
                int rec = -1;
                for (int a = 0; a < nm; ++a) {
                    const int mr = A.g_mrec[m0 + a], p = mr & 255, w = mr >> 8;
                    if (x >= p && x < p + w) rec = a | ((x - p) << 8);
                }
                S.rowrec[x] = rec;
            }
            oz_epi_sync();
            if (S.epi_stop) break;
            int ex[4];                                // the scales' exponents of this thread's elements, two a word
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int rr = S.rowrec[r], r0 = S.colrec[8 * part + 2 * j], r1 = S.colrec[8 * part + 2 * j + 1];
                const int e0 = rr >= 0 && r0 >= 0 ? S.kexp[rr & 255][r0 & 255] : 4096;
                const int e1 = rr >= 0 && r1 >= 0 ? S.kexp[rr & 255][r1 & 255] : 4096;
                ex[j] = (e0 & 0xffff) | (int)((unsigned)e1 << 16);
            }
            const int bcol = q * kSlice + 8 * part;   // first column of this thread
            Oz96 acc[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[j] = Oz96{0u, 0};
            bool ok = true;
            const int4* ent = A.ent + A.s_ptr[t];
            for (int ne = (int)(A.s_ptr[t + 1] - A.s_ptr[t]); ne > 0; --ne, ++ent) {
                const int4 en = __ldg(ent);
                if (!(((unsigned)en.z >> (8 * q)) & 255u)) continue;
                const int nd = (int)(((unsigned)en.w >> (8 * q)) & 255u);
                const int ea = r < A.R ? (int)__ldg(A.a_rexp + (int64_t)en.x * A.R + r) : 0;
                const int4 ebv = __ldg(reinterpret_cast<const int4*>(A.b_rexp + (int64_t)en.y * A.R + bcol));
                const int ew[4] = {ebv.x, ebv.y, ebv.z, ebv.w};
                const uint32_t buf = n & 1u;
                ok = __all_sync(0xffffffffu, tc::mbar_wait(&S.acc_full[buf], (n >> 1) & 1u, kOzWait) && !oz_aborted(S));
                if (!ok) {
                    oz_fail(A, S);
                    break;
                }
                tc::fence_after_sync();
                const uint32_t ta = lane_base + buf * 256u;
                // accumulators past the entry's digits hold older sums and are not read; two versions
                // of the code (one for each digit count ran slower: they miss the instruction cache)
                if (nd > 4) oz_take<8>(nd, acc, ex, ea, ew, ta, &S.acc_empty[buf], lane);
                else oz_take<4>(nd, acc, ex, ea, ew, ta, &S.acc_empty[buf], lane);
                ++n;
            }
            oz_item_done(S, ni, lane);
            const int rr = S.rowrec[r], ra = rr & 255, ri = rr >> 8;
            if (ok && rr >= 0) {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int rec = S.colrec[8 * part + j];
                    if (rec < 0) continue;
                    const int b = rec & 255, cj = (rec >> 8) & 255, w = rec >> 16;
                    const int64_t o = S.koff[ra][b];
                    if (o < 0) continue;
                    const int64_t p = (int64_t)ri * w + cj, ci = S.kcin[ra][b];
                    double val = A.alpha * oz_value(acc[j], S.kexp[ra][b] - 70);
                    if (ci >= 0) val = val + A.beta * A.ci_data[ci + p];
                    A.c_data[o + p] = val;
                }
            }
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, kOzTmem);
    }
}

// Norms and distances to 1 of the blocks the tensor cores computed (one warp per block; a block's
// columns can lie in two slices, so the kernel above cannot sum them).
__global__ void k_oz_norms(int64_t nform, const uint8_t* __restrict__ comp, const int32_t* __restrict__ row,
                           const int32_t* __restrict__ col, const int32_t* __restrict__ bs,
                           const int64_t* __restrict__ off, const double* __restrict__ data,
                           double* __restrict__ norms, double* __restrict__ dev2) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t b = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); b < nform; b += warps) {
        if (comp[b] != 2) continue;
        const int I = row[b], J = col[b];
        const int n = bs[J], area = bs[I] * n;
        const double* x = data + off[b];
        double s = 0.0, d = 0.0;
        for (int e = lane; e < area; e += 32) {
            const double v = x[e];
            s = fma(v, v, s);
            if (I == J) {
                const double w = (e % (n + 1) == 0) ? v - 1.0 : v;
                d = fma(w, w, d);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            s += __shfl_xor_sync(0xffffffffu, s, o);
            d += __shfl_xor_sync(0xffffffffu, d, o);
        }
        if (lane == 0) {
            norms[b] = sqrt(s);
            dev2[b] = I == J ? d : s;
        }
    }
}

PFN_cuTensorMapEncodeTiled_v12000 oz_map_encoder() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        DBG_CK(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q));
        if (q != cudaDriverEntryPointSuccess || !p) fail(DBCSR_ECUDA, "multiply: cuTensorMapEncodeTiled not found");
        return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }();
    return fn;
}

// Packed tiles as a 4-D tensor: (8 columns x R rows) of a digit, digit, chunk, K step of a tile;
// a box is one chunk of a 32-row slice in the leading digits (rows past R read as zero).
CUtensorMap oz_map(const uint8_t* base, int R, int64_t nsteps, int digits) {
    CUtensorMap m;
    const cuuint64_t dims[4] = {(cuuint64_t)R * 8, kDigits, 2, (cuuint64_t)std::max<int64_t>(nsteps, 1)};
    const cuuint64_t strides[3] = {(cuuint64_t)R * 16, (cuuint64_t)R * 16 * kDigits, (cuuint64_t)R * 32 * kDigits};
    const cuuint32_t box[4] = {kSlice * 8, (cuuint32_t)digits, 1, 1};
    const cuuint32_t es[4] = {1, 1, 1, 1};
    const CUresult r = oz_map_encoder()(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<uint8_t*>(base), dims, strides,
                                        box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) fail(DBCSR_ECUDA, "multiply: cuTensorMapEncodeTiled failed");
    return m;
}

}  // namespace

// One operand packed into digit tiles.
struct OzOperand {
    TilePattern pat;
    int transpose = 0;
    DBuf<int32_t> tab;
    DBuf<unsigned> smask;
    DBuf<uint8_t> pack;
    DBuf<int16_t> rexp, mexp;
};

struct F64TcPlan {
    std::shared_ptr<Groups> groups;
    OzOperand a, b;
    bool b_is_a = false, b_sym = false;
    int R = 0, KS = 0, nsl = 0;
    TilePattern cp;
    DBuf<int32_t> b_map, st_a, st_b, c_tbl;
    DBuf<int16_t> c_exp;
    DBuf<unsigned long long> next;       // counter of the work items
    DBuf<int64_t> s_ptr;
    DBuf<unsigned> c_slices;
    DBuf<int4> ent;
    DBuf<unsigned long long> tile_flops;
    DBuf<int> flags, flags0;             // see kFlag*; what they start with (0 but for the self-test)
    DBuf<uint8_t> redo;                  // planned products: blocks the FP64 pipe repeats
    int64_t nentries = 0;
};

void f64tc_delete(F64TcPlan* p) { delete p; }

namespace {

// The group tiles of up to three block patterns with one host synchronisation.
struct PatternJob {
    const int64_t* rp; const int32_t* col; const uint8_t* use; int64_t nnzb; TilePattern* out;
};
void tile_patterns(const Groups& g, PatternJob* jobs, int n, int64_t* max_c, cudaStream_t s) {
    const int nwords = pattern_words(g.ngrp);
    const size_t sm = (size_t)2 * ((nwords + 1) & ~1) * sizeof(uint32_t);
    GView gv{g.g_of.p, g.g_pos.p, g.g_ptr.p, g.g_mem.p, g.g_w.p};
    allow_dyn_smem(k_gt_pattern, sm);
    const unsigned grid = (unsigned)std::min<int64_t>(g.ngrp, (int64_t)num_sms() * 8);
    DBuf<int64_t> cnt[3];
    const int64_t *src[3], *in[3];
    int64_t h[3], *out[3];
    for (int i = 0; i < n; ++i) {
        cnt[i].alloc(g.ngrp, s);
        jobs[i].out->t_rp.alloc(g.ngrp + 1, s);
        k_gt_pattern<<<grid, 256, sm, s>>>(g.ngrp, gv, jobs[i].rp, jobs[i].col, jobs[i].use, nwords, 0, cnt[i].p, nullptr,
                                           nullptr, nullptr, nullptr);
        DBG_LAUNCH_CK();
        in[i] = cnt[i].p;
        out[i] = jobs[i].out->t_rp.p;
        src[i] = out[i] + g.ngrp;
    }
    scan_exclusive(in, out, n, g.ngrp, s);
    std::vector<int64_t> rows(g.ngrp);
    DBG_CK(cudaMemcpyAsync(rows.data(), cnt[n - 1].p, sizeof(int64_t) * g.ngrp, cudaMemcpyDeviceToHost, s));
    read_i64s(src, n, h, s);
    *max_c = 0;
    for (int64_t v : rows) *max_c = std::max(*max_c, v);
    for (int i = 0; i < n; ++i) {
        TilePattern& P = *jobs[i].out;
        P.nt = h[i];
        P.t_row.alloc(std::max<int64_t>(P.nt, 1), s);
        P.t_col.alloc(std::max<int64_t>(P.nt, 1), s);
        P.blk_tile.alloc(std::max<int64_t>(jobs[i].nnzb, 1), s);
        k_gt_pattern<<<grid, 256, sm, s>>>(g.ngrp, gv, jobs[i].rp, jobs[i].col, jobs[i].use, nwords, 1, nullptr, P.t_rp.p,
                                           P.t_row.p, P.t_col.p, P.blk_tile.p);
        DBG_LAUNCH_CK();
    }
}

int64_t device_memory() {
    static std::mutex mu;
    static auto* bytes = new std::map<int, int64_t>();   // (outlives every static destructor)
    int dev = 0;
    DBG_CK(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(mu);
    int64_t& n = (*bytes)[dev];
    if (!n) {
        size_t fr = 0, all = 0;
        DBG_CK(cudaMemGetInfo(&fr, &all));
        n = (int64_t)all;
    }
    return n;
}

int64_t oz_tile_bytes(const F64TcPlan& L) { return (int64_t)L.KS * 2 * kDigits * 16 * L.R; }

void oz_tables(F64TcPlan& L, OzOperand& o, const dbcsr_matrix_* M, cudaStream_t s) {
    const Groups& g = *L.groups;
    const int64_t nt = std::max<int64_t>(o.pat.nt, 1);
    o.tab.alloc(nt * kGroupMembers * kGroupMembers, s);
    o.smask.alloc(nt, s);
    DBG_CK(cudaMemsetAsync(o.tab.p, 0xff, sizeof(int32_t) * nt * kGroupMembers * kGroupMembers, s));
    o.smask.zero();
    if (M->nnzb) {
        k_oz_tiles<<<grid_for(M->nnzb, 256), 256, 0, s>>>(M->nnzb, M->row.p, M->col.p, M->bs.p, g.g_pos.p, g.g_midx.p,
                                                          o.pat.blk_tile.p, o.transpose, o.tab.p, o.smask.p);
        DBG_LAUNCH_CK();
    }
    o.pack.alloc(nt * oz_tile_bytes(L), s);
    o.rexp.alloc(nt * L.R + 64, s);      // the last slice reads exponents past the last row
    o.rexp.zero();
    o.mexp.alloc(nt * kGroupMembers, s);
}

void oz_pack(F64TcPlan& L, OzOperand& o, const dbcsr_matrix_* M, cudaStream_t s) {
    if (!o.pat.nt) return;
    const Groups& g = *L.groups;
    OzPackArgs p{o.pat.nt, o.transpose ? o.pat.t_col.p : o.pat.t_row.p, o.transpose ? o.pat.t_row.p : o.pat.t_col.p,
                 o.tab.p, o.smask.p, g.g_ptr.p, g.g_mrec.p, g.g_w.p, M->off.p, M->data.p, o.transpose, L.R, L.KS,
                 o.pack.p, o.rexp.p, o.mexp.p, L.flags.p + kFlagRange};
    k_oz_pack<<<(unsigned)std::min<int64_t>(o.pat.nt, (int64_t)num_sms() * 64), 256, 0, s>>>(p);
    DBG_LAUNCH_CK();
}

// K steps and digits of every stack entry, from the operands' current scales.
void oz_depth(F64TcPlan& L, cudaStream_t s) {
    const OzOperand& b = L.b_is_a ? L.a : L.b;
    if (!L.nentries) return;
    OzDepthArgs d{L.cp.nt, L.cp.t_col.p, L.groups->g_ptr.p, L.groups->g_mrec.p, L.s_ptr.p, L.st_a.p, L.st_b.p,
                  L.a.mexp.p, b.mexp.p, L.c_tbl.p, L.c_exp.p, L.a.smask.p, b.smask.p, L.ent.p};
    k_oz_depth<<<grid_for(L.cp.nt, 8), 256, 0, s>>>(d);
    DBG_LAUNCH_CK();
}

}  // namespace

std::unique_ptr<F64TcPlan, void (*)(F64TcPlan*)> f64tc_prepare(dbcsr_matrix_* A, dbcsr_matrix_* B,
                                                               std::shared_ptr<Groups> groups, int64_t nform,
                                                               const int64_t* f_rp, const F64TcBlocks& f, double alpha,
                                                               bool planned, bool weigh, cudaStream_t s) {
    std::unique_ptr<F64TcPlan, void (*)(F64TcPlan*)> P(nullptr, f64tc_delete);
    if (groups->ngrp > kMaxBlockRowsLt || !nform) return P;
    std::unique_ptr<F64TcPlan, void (*)(F64TcPlan*)> up(new F64TcPlan(), f64tc_delete);
    F64TcPlan& L = *up;
    const Groups& g = *groups;
    L.groups = groups;
    const int wmax = *std::max_element(g.h_w.begin(), g.h_w.end());
    L.R = (wmax + 7) & ~7;
    L.KS = (wmax + 15) / 16;
    L.nsl = (int)ceil_div(wmax, kSlice);
    // B's K-major tiles are the tiles of its transpose: with B exactly symmetric those of B itself (not in
    // a planned product, whose later values need not be symmetric)
    L.b_sym = B->exact_sym && !planned;
    L.b_is_a = A == B && L.b_sym;
    k_oz_role<<<grid_for(nform, 256), 256, 0, s>>>(nform, f.row, f.col, f.mirror, f.sym, g.g_of.p, f.by_group, f.comp);
    DBG_LAUNCH_CK();
    PatternJob jobs[3];
    int nj = 0;
    jobs[nj++] = {A->rp.p, A->col.p, nullptr, A->nnzb, &L.a.pat};
    if (!L.b_is_a) jobs[nj++] = {B->rp.p, B->col.p, nullptr, B->nnzb, &L.b.pat};
    jobs[nj++] = {f_rp, f.col, f.comp, nform, &L.cp};
    int64_t max_row = 0;
    tile_patterns(g, jobs, nj, &max_row, s);
    // the packed operands stay within a quarter of the device's memory (and where what is free does not hold
    // them, the product runs again without them: multiply)
    if ((L.a.pat.nt + L.b.pat.nt) * oz_tile_bytes(L) > device_memory() / 4) return P;
    if (!L.cp.nt || (int64_t)(L.a.pat.nt + L.b.pat.nt) * L.KS > 0x7fffffff) return P;
    L.flags.alloc(kFlags, s);
    L.flags0.alloc(kFlags, s);
    L.flags.zero();
    L.flags0.zero();
    OzOperand& b = L.b_is_a ? L.a : L.b;
    if (L.b_sym && b.pat.nt) {
        L.b_map.alloc(b.pat.nt, s);
        k_gt_transpose<<<grid_for(b.pat.nt, 256), 256, 0, s>>>(b.pat.nt, b.pat.t_row.p, b.pat.t_col.p, b.pat.t_rp.p,
                                                               L.b_map.p, L.flags.p + kFlagFailed);
        DBG_LAUNCH_CK();
    }
    // stacks of tile products per C tile
    const int nwords = pattern_words(g.ngrp);
    const size_t sm_base = (size_t)2 * ((nwords + 1) & ~1) * sizeof(uint32_t);
    const bool use_smem = sm_base + (size_t)max_row * sizeof(int32_t) <= (size_t)96 * 1024;
    const size_t sm = use_smem ? sm_base + (size_t)max_row * sizeof(int32_t) : sm_base;
    DBuf<int64_t> cnt;
    DBuf<int32_t> cursor;
    cnt.alloc(L.cp.nt, s);
    L.s_ptr.alloc(L.cp.nt + 1, s);
    if (!use_smem) cursor.alloc(L.cp.nt, s);
    GView gv{g.g_of.p, g.g_pos.p, g.g_ptr.p, g.g_mem.p, g.g_w.p};
    StackArgs sa{gv, L.cp.t_rp.p, L.cp.t_col.p, L.a.pat.t_rp.p, L.a.pat.t_col.p, b.pat.t_rp.p, b.pat.t_col.p,
                 L.b_sym ? L.b_map.p : nullptr, cnt.p, nullptr, nullptr, nullptr, cursor.p, 0, use_smem ? 1 : 0};
    allow_dyn_smem(k_gt_stack, sm);
    const unsigned grid = (unsigned)std::min<int64_t>(g.ngrp, (int64_t)num_sms() * 8);
    k_gt_stack<<<grid, 256, sm, s>>>(g.ngrp, sa, nwords);
    DBG_LAUNCH_CK();
    scan_exclusive(cnt.p, L.s_ptr.p, L.cp.nt, s);
    L.tile_flops.alloc(L.cp.nt, s);
    L.tile_flops.zero();
    k_oz_tile_flops<<<grid_for(nform, 256), 256, 0, s>>>(nform, L.cp.blk_tile.p, f.row, f.col, f.ksum, A->bs.p,
                                                         L.tile_flops.p);
    DBG_LAUNCH_CK();
    L.next.alloc(1, s);
    L.next.zero();
    k_oz_pays<<<grid_for(L.cp.nt, 256), 256, 0, s>>>(L.cp.nt, L.s_ptr.p, L.cp.t_col.p, g.g_w.p, L.tile_flops.p, L.next.p);
    DBG_LAUNCH_CK();
    {
        const int64_t* src[2] = {L.s_ptr.p + L.cp.nt, (const int64_t*)L.next.p};
        int64_t h[2];
        read_i64s(src, 2, h, s);
        L.nentries = h[0];
        const double pays = (double)(unsigned long long)h[1];
        const double pack = (double)(L.a.pat.nt + L.b.pat.nt) * (double)oz_tile_bytes(L);
        if (pays == 0.0 || (weigh && pays / kSimtFlopsPerSecond < pack / kPackBytesPerSecond)) return P;
    }
    oz_tables(L, L.a, A, s);
    oz_pack(L, L.a, A, s);
    if (!L.b_is_a) {
        L.b.transpose = L.b_sym ? 0 : 1;
        oz_tables(L, L.b, B, s);
        oz_pack(L, L.b, B, s);
    }
    const int64_t ne = std::max<int64_t>(L.nentries, 1);
    L.st_a.alloc(ne, s);
    L.st_b.alloc(ne, s);
    L.ent.alloc(ne, s);
    sa.fill = 1;
    sa.s_ptr = L.s_ptr.p;
    sa.st_a = L.st_a.p;
    sa.st_b = L.st_b.p;
    k_gt_stack<<<grid, 256, sm, s>>>(g.ngrp, sa, nwords);
    DBG_LAUNCH_CK();
    // which blocks the tensor cores take
    L.c_slices.alloc(L.cp.nt, s);
    L.c_slices.zero();
    L.c_tbl.alloc(L.cp.nt * kGroupMembers * kGroupMembers, s);
    L.c_exp.alloc(L.cp.nt * kGroupMembers * kGroupMembers, s);
    if (planned) L.redo.alloc(nform, s);
    DBG_CK(cudaMemsetAsync(L.c_tbl.p, 0xff, sizeof(int32_t) * L.cp.nt * kGroupMembers * kGroupMembers, s));
    DBuf<int16_t> f_exp;
    f_exp.alloc(nform, s);
    OzGuardArgs ga{nform, L.cp.blk_tile.p, f.row, f.col, g.g_midx.p, g.g_w.p, L.cp.t_col.p, L.s_ptr.p, L.st_a.p, L.st_b.p,
                   L.a.mexp.p, b.mexp.p, f.max_term, f.max_at, L.tile_flops.p, (float)std::fabs(alpha), L.flags.p + kFlagRange,
                   f_exp.p, f.comp, L.c_tbl.p, L.c_exp.p, L.c_slices.p, g.g_pos.p, A->bs.p,
                   A->rp.p, A->col.p, A->off.p, A->data.p, B->rp.p, B->col.p, B->off.p, B->data.p};
    k_oz_guard<<<grid_for(nform, 256), 256, 0, s>>>(ga);
    DBG_LAUNCH_CK();
    k_oz_weak<<<grid_for(nform, kWeakWarps, (int64_t)num_sms() * 64), 32 * kWeakWarps, 0, s>>>(ga);
    DBG_LAUNCH_CK();
    oz_depth(L, s);
    return up;
}

void f64tc_pack(F64TcPlan& L, const dbcsr_matrix_* A, const dbcsr_matrix_* B, cudaStream_t s) {
    DBG_CK(cudaMemcpyAsync(L.flags.p, L.flags0.p, sizeof(int) * kFlags, cudaMemcpyDeviceToDevice, s));
    oz_pack(L, L.a, A, s);
    if (!L.b_is_a) oz_pack(L, L.b, B, s);
}

namespace {

// A planned product's new values: one warp per tensor-core block, the tests of k_oz_guard and k_oz_weak on
// its stack, with one more bit of room.
__global__ void __launch_bounds__(32 * kWeakWarps) k_oz_recheck(OzGuardArgs A, const int64_t* __restrict__ pbeg,
                                                                const int32_t* __restrict__ prod_a,
                                                                const int32_t* __restrict__ prod_b,
                                                                const double* __restrict__ an,
                                                                const double* __restrict__ bn,
                                                                uint8_t* __restrict__ redo, int* __restrict__ any) {
    __shared__ float sh[kWeakWarps][2][kMaxBlock * kMaxBlock];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t k = (int64_t)blockIdx.x * kWeakWarps + warp; k < A.nform; k += (int64_t)gridDim.x * kWeakWarps) {
        if (A.comp[k] != 2) continue;
        const int32_t t = A.blk_tile[k], I = A.f_row[k], J = A.f_col[k];
        const int a = A.g_midx[I], b = A.g_midx[J];
        int E = 2 * kNoExp;
        for (int64_t e = A.s_ptr[t] + lane; e < A.s_ptr[t + 1]; e += 32)
            E = max(E, (int)A.a_mexp[(int64_t)A.st_a[e] * kGroupMembers + a] +
                           (int)A.b_mexp[(int64_t)A.st_b[e] * kGroupMembers + b]);
        E = __reduce_max_sync(0xffffffffu, E);
        double mx = 0.0;
        int64_t at = -1;                              // the strongest block product (of equal ones any)
        for (int64_t p = pbeg[k] + lane; p < pbeg[k + 1]; p += 32) {
            const double v = an[prod_a[p]] * bn[prod_b[p]];
            if (v > mx) {
                mx = v;
                at = p;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double omx = __shfl_xor_sync(0xffffffffu, mx, o);
            const int64_t oat = __shfl_xor_sync(0xffffffffu, at, o);
            if (omx > mx || (omx == mx && oat > at)) {
                mx = omx;
                at = oat;
            }
        }
        bool ok = *A.bad == 0;                        // (an operand outside the scales: all of them)
        if (ok && E > kNoExp / 2) {
            ok = at >= 0 && ldexp((double)kNormRatio, E - 1) < mx && mx <= 1e300;
            if (ok) {
                const int32_t p = prod_a[at], q = prod_b[at];
                ok = oz_no_weak(A.a_data + A.a_off[p], A.b_data + A.b_off[q], A.bs[I], A.bs[A.a_col[p]], A.bs[J], E,
                                kWeakBits + 1, lane, sh[warp]);
            }
        }
        if (lane == 0) {
            A.c_exp[(int64_t)t * (kGroupMembers * kGroupMembers) + a * kGroupMembers + b] = (int16_t)max(E, kNoTerm);
            redo[k] = ok ? 0 : 1;
            if (!ok) atomicExch(any, 1);
        }
    }
}

}  // namespace

F64TcRedo f64tc_recheck(F64TcPlan& L, const dbcsr_matrix_* A, const dbcsr_matrix_* B, double* an, double* bn,
                        int64_t nform, const F64TcBlocks& f, const int64_t* f_pbeg, const int32_t* prod_a,
                        const int32_t* prod_b, double alpha, cudaStream_t s) {
    const Groups& g = *L.groups;
    const OzOperand& b = L.b_is_a ? L.a : L.b;
    block_norms(A, an, s);
    const double* bnp = an;
    if (B != A) {
        block_norms(B, bn, s);
        bnp = bn;
    }
    OzGuardArgs ga{nform, L.cp.blk_tile.p, f.row, f.col, g.g_midx.p, g.g_w.p, L.cp.t_col.p, L.s_ptr.p, L.st_a.p, L.st_b.p,
                   L.a.mexp.p, b.mexp.p, nullptr, nullptr, L.tile_flops.p, (float)std::fabs(alpha), L.flags.p + kFlagRange,
                   nullptr, f.comp,
                   L.c_tbl.p, L.c_exp.p, nullptr, g.g_pos.p, A->bs.p,
                   A->rp.p, A->col.p, A->off.p, A->data.p, B->rp.p, B->col.p, B->off.p, B->data.p};
    k_oz_recheck<<<grid_for(nform, kWeakWarps, (int64_t)num_sms() * 64), 32 * kWeakWarps, 0, s>>>(
        ga, f_pbeg, prod_a, prod_b, an, bnp, L.redo.p, L.flags.p + kFlagRedo);
    DBG_LAUNCH_CK();
    oz_depth(L, s);
    return F64TcRedo{L.flags.p + kFlagRedo, L.redo.p};
}

void f64tc_run(F64TcPlan& L, const LowTierOut& o, cudaStream_t s) {
    const Groups& g = *L.groups;
    const OzOperand& b = L.b_is_a ? L.a : L.b;
    OzArgs a{};
    a.nitems = L.cp.nt * L.nsl;
    a.nsl = L.nsl;
    a.R = L.R;
    a.KS = L.KS;
    a.c_trow = L.cp.t_row.p;
    a.c_tcol = L.cp.t_col.p;
    a.s_ptr = L.s_ptr.p;
    a.c_slices = L.c_slices.p;
    a.ent = L.ent.p;
    a.a_pack = L.a.pack.p;
    a.a_rexp = L.a.rexp.p;
    a.b_rexp = b.rexp.p;
    a.g_ptr = g.g_ptr.p;
    a.g_mrec = g.g_mrec.p;
    a.c_tbl = L.c_tbl.p;
    a.c_exp = L.c_exp.p;
    a.next = L.next.p;
    a.f_off = o.f_off;
    a.f_cin = o.f_cin;
    a.ci_off = o.ci_off;
    a.ci_data = o.ci_data;
    a.alpha = o.alpha;
    a.beta = o.beta;
    a.c_data = o.c_data;
    a.flags = L.flags.p;
    OzMaps mb;
    for (int d = 0; d < kDigits; ++d) mb.m[d] = oz_map(b.pack.p, L.R, b.pat.nt * L.KS, d + 1);
    const size_t sm = sizeof(OzShared) + 1024;
    allow_dyn_smem(k_oz, sm);
    DBG_CK(cudaMemsetAsync(L.next.p, 0, sizeof(unsigned long long), s));
    k_oz<<<(unsigned)std::min<int64_t>(a.nitems, (int64_t)num_sms()), kOzThreads, sm, s>>>(mb, a);
    DBG_LAUNCH_CK();
}

void f64tc_norms(int64_t nform, const uint8_t* comp, const int32_t* row, const int32_t* col, const int32_t* bs,
                 const int64_t* off, const double* data, double* norms, double* dev2, cudaStream_t s) {
    k_oz_norms<<<grid_for(nform, 8), 256, 0, s>>>(nform, comp, row, col, bs, off, data, norms, dev2);
    DBG_LAUNCH_CK();
}

int64_t f64tc_tiles(const F64TcPlan& L) { return L.cp.nt; }

void f64tc_release(F64TcPlan& L) {
    for (OzOperand* o : {&L.a, &L.b}) {
        o->pack.release();
        o->tab.release();
        o->rexp.release();
    }
    L.st_a.release();
    L.st_b.release();
    L.ent.release();
    L.c_tbl.release();
    L.c_exp.release();
}

void f64tc_selftest(F64TcPlan& L, bool fail_waits, cudaStream_t s) {
    const int v = fail_waits ? 1 : 0;
    DBG_CK(cudaMemcpyAsync(L.flags0.p + kFlagFailed, &v, sizeof v, cudaMemcpyHostToDevice, s));
    DBG_CK(cudaStreamSynchronize(s));
}

void f64tc_check(F64TcPlan& L, cudaStream_t s) {
    int e = 0;
    DBG_CK(cudaMemcpyAsync(&e, L.flags.p + kFlagFailed, sizeof(int), cudaMemcpyDeviceToHost, s));
    DBG_CK(cudaStreamSynchronize(s));
    if (e == 1) fail(DBCSR_ETIMEOUT, "multiply: a wait of the tensor-core kernel ran out");
    if (e == 2) fail(DBCSR_EINVAL, "multiply: an operand marked symmetric has an asymmetric pattern");
}

}  // namespace dbg
