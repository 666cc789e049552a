// Batched dense products of the submatrix method (section "Submatrix Method": each
// submatrix is purified densely), C[b] = alpha A[b] B[b] + beta C[b] for a batch of n x n
// row-major matrices, in the library's own kernels:
//
//   * FP32 storage on the 5th-generation tensor cores (tcgen05.mma kind::tf32, FP32
//     accumulators in tensor memory).  Plain TF32 keeps 10 stored bits of each operand (the
//     tensor cores drop the low 13); split TF32 (hi = x so truncated, lo = x - hi likewise,
//     three products hi*hi + hi*lo + lo*hi) carries about 20 bits, close to FP32 arithmetic.
//     The operands come straight from the matrices through tensor maps (B transposed once;
//     A through a copy with padded rows when its rows do not start on 16-byte boundaries).
//   * FP64 storage on the FP64 pipe: 64 x 64 C tiles, 16-wide K slices in shared memory, a
//     4 x 4 register tile per thread.  GB300's FP64 rate is low enough (about 3.5 flops per
//     SM cycle) that the FMA loop, not memory, bounds it.
#include <algorithm>
#include <cstdint>

#include <cuda.h>
#include <cudaTypedefs.h>

#include "common.cuh"
#include "tc05.cuh"

namespace dbg {
namespace {

constexpr int kDM = 128;                 // M of the MMA and rows of an A tile
constexpr int kDNMax = 256;              // rows of the widest B tile (N of the MMA)
constexpr int kDStepK = 8;               // TF32 elements per MMA K step (32 bytes)
constexpr int kTK = 16;                  // K columns per stage (64-byte rows)
constexpr int kTStageBytes = (kDM + kDNMax) * kTK * 4;  // 24 KB: A 8 KB, B up to 16 KB
constexpr int kDEpiCols = 32;            // accumulator columns staged per pass of an epilogue warp
constexpr int kDEpiWarps = 8;            // two per TMEM lane quadrant, every other pass each
constexpr int kTConvWarps = 8;           // split operands: warps that write the low parts
constexpr long long kDWaitLimit = 4000000000ll;

// TF32 as the tensor cores read an FP32 operand: the 13 low mantissa bits dropped (truncation
// toward zero).
__device__ __forceinline__ float to_tf32(float x) { return __uint_as_float(__float_as_uint(x) & 0xFFFFE000u); }

template <bool SPLIT>
struct TmaShared {
    static constexpr int kStages = SPLIT ? 4 : 7;
    alignas(1024) uint8_t x[kStages][kTStageBytes];
    alignas(1024) uint8_t lo[SPLIT ? kStages : 1][SPLIT ? kTStageBytes : 16];
    float out[kDEpiWarps][32][kDEpiCols + 1];   // odd stride: no bank conflicts
    uint64_t full[kStages], conv[kStages], empty[kStages], acc_full[2], acc_empty[2], fin;
    uint32_t tmem_base;
    int abort;
};

struct TmaArgs {
    int n, ntm, ntn, NT;                 // NT: rows of every B tile (N of the MMA)
    int64_t ntiles;
    float alpha, beta;
    const float* Cin;                    // beta's C (may be C)
    float* C;
    int* err;
};

// One persistent CTA per SM over the 128 x NT tiles of C, the row tiles of a matrix next to each other
// so that the CTAs running at one time share its B tiles in L2.  Warp 0 streams 16 K columns per
// stage of the A and B^T tiles into a ring (3-D tensor maps, 64-byte swizzled K-major rows, read by the
// MMAs as they are: as TF32); for split operands eight converter warps write lo = x - tf32(x) of every
// stage, four of them every other stage (the write, the proxy fence and the arrival take a stage's
// time, so two stages are converted at once); warp 1 issues the MMAs (two K = 8 steps per stage,
// three MMAs each when split) into one of two TMEM accumulators, and eight warps write the other one
// back meanwhile, 32 rows and 32 columns at a time.
// On 400 matrices of 400 x 400 the earlier kernel (one CTA per tile, four converter warps that also
// wrote the result back, MMAs issued behind lane 0) took 0.63 ms split and 0.27 ms plain with the
// tensor cores 28% and 22% busy: loads, products and the write-back followed one another in a CTA.
// Now 0.33 ms (55% busy; the low parts' writes bound it) and 0.17 ms (bytes: 0.11 ms at copy rate).
template <bool SPLIT>
__global__ void __launch_bounds__(32 * (2 + (SPLIT ? kTConvWarps : 0) + kDEpiWarps), 1)
    k_dense_tf32(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_bt, TmaArgs D) {
    extern __shared__ __align__(1024) uint8_t t_dyn[];
    using Sh = TmaShared<SPLIT>;
    constexpr int ST = Sh::kStages;
    auto& S = *reinterpret_cast<Sh*>((reinterpret_cast<uintptr_t>(t_dyn) + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int epi0 = SPLIT ? 2 + kTConvWarps : 2;
    const int NT = D.NT;
    const int a_bytes = kDM * kTK * 4, b_bytes = NT * kTK * 4;
    const int nstage = (D.n + kTK - 1) / kTK;
    auto failed = [&] {
        *(volatile int*)&S.abort = 1;
        atomicExch(D.err, 1);
    };
    auto aborted = [&] { return *(volatile const int*)&S.abort != 0; };
    if (threadIdx.x == 0) {
        for (int i = 0; i < ST; ++i) {
            tc::mbar_init(&S.full[i], 1);
            tc::mbar_init(&S.conv[i], kTConvWarps / 2);
            tc::mbar_init(&S.empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&S.acc_full[i], 1);
            tc::mbar_init(&S.acc_empty[i], kDEpiWarps);
        }
        tc::mbar_init(&S.fin, 1);
        S.abort = 0;
        tc::fence_barrier_init();
    }
    if (warp == 1) {
        tc::tmem_alloc(&S.tmem_base, 2 * kDNMax);
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = S.tmem_base;
    if (warp == 0) {
        // ---- producer (lane 0): a stage is refilled once the MMAs that read it completed
        if (lane == 0) {
            int slot = 0;
            uint32_t phase = 0;
            int64_t issued = 0;
            bool ok = true;
            for (int64_t tile = blockIdx.x; tile < D.ntiles && ok; tile += gridDim.x) {
                const int64_t rest = tile / D.ntm;
                const int tm = (int)(tile - rest * D.ntm), b = (int)(rest / D.ntn), tn = (int)(rest - (int64_t)b * D.ntn);
                for (int s = 0; s < nstage; ++s) {
                    if (!tc::mbar_wait(&S.empty[slot], phase ^ 1u, kDWaitLimit)) failed();
                    if (aborted()) {
                        ok = false;
                        break;
                    }
                    tc::mbar_arrive_expect_tx(&S.full[slot], (uint32_t)(a_bytes + b_bytes));
                    tc::tma_load3d(S.x[slot], &map_a, s * kTK, tm * kDM, b, &S.full[slot]);
                    tc::tma_load3d(S.x[slot] + a_bytes, &map_bt, s * kTK, tn * NT, b, &S.full[slot]);
                    ++issued;
                    if (++slot == ST) {
                        slot = 0;
                        phase ^= 1u;
                    }
                }
            }
            // no copy may still be landing when the CTA exits
            for (int64_t x = 0; x < issued && x < ST; ++x) {
                if (--slot < 0) {
                    slot = ST - 1;
                    phase ^= 1u;
                }
                if (!tc::mbar_wait(&S.full[slot], phase, kDWaitLimit)) failed();
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---- MMA issuer (the whole warp, every lane with the same values)
        const uint32_t idesc = tc::uniform(tc::instr_desc(2, kDM, NT));
        const uint64_t hi = tc::smem_desc_sw64(0);    // all but the start address
        const uint32_t x0 = tc::smem_u32(S.x[0]) >> 4, l0 = SPLIT ? tc::smem_u32(S.lo[0]) >> 4 : 0;
        int slot = 0;
        uint32_t phase = 0, k = 0;
        bool ok = true;
        for (int64_t tile = blockIdx.x; tile < D.ntiles && ok; tile += gridDim.x, ++k) {
            const uint32_t buf = k & 1u;
            const uint32_t d = tc::uniform(tmem + buf * kDNMax);
            ok = tc::mbar_wait_warp(&S.acc_empty[buf], ((k >> 1) & 1u) ^ 1u, kDWaitLimit);
            uint32_t acc = 0;
            for (int s = 0; s < nstage && ok; ++s) {
                ok = tc::mbar_wait(SPLIT ? &S.conv[slot] : &S.full[slot], phase, kDWaitLimit) && !aborted();
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc::fence_after_sync();
                const uint32_t xa = tc::uniform(x0 + (uint32_t)slot * (kTStageBytes / 16));
                const uint32_t la = SPLIT ? tc::uniform(l0 + (uint32_t)slot * (kTStageBytes / 16)) : 0;
                constexpr uint32_t ab = kDM * kTK * 4 / 16;
                if (tc::elect_one()) {
#pragma unroll
                    for (uint32_t j = 0; j < kTK / kDStepK; ++j) {
                        const uint32_t ko = j * (kDStepK * 4 / 16);          // 32 bytes per K = 8 step
                        tc::mma_tf32(d, hi | (xa + ko), hi | (xa + ab + ko), idesc, j ? 1u : acc);
                        if (SPLIT) {
                            tc::mma_tf32(d, hi | (xa + ko), hi | (la + ab + ko), idesc, 1);
                            tc::mma_tf32(d, hi | (la + ko), hi | (xa + ab + ko), idesc, 1);
                        }
                    }
                    tc::mma_commit(&S.empty[slot]);
                    if (s == nstage - 1) tc::mma_commit(&S.acc_full[buf]);
                }
                __syncwarp();
                acc = 1;
                if (++slot == ST) {
                    slot = 0;
                    phase ^= 1u;
                }
            }
            ok = __all_sync(0xffffffffu, ok);
            if (!ok && lane == 0) failed();
        }
        // every MMA has completed before the TMEM is released
        if (tc::elect_one()) tc::mma_commit(&S.fin);
        __syncwarp();
        if (!tc::mbar_wait(&S.fin, 0, kDWaitLimit) && lane == 0) failed();
        __syncwarp();
    } else if (SPLIT && warp < epi0) {
        // ---- converters (split operands): lo = x - tf32(x) of every other stage
        constexpr int kConvThreads = 16 * kTConvWarps, kBatch = 6;
        const int ct = (threadIdx.x - 64) % kConvThreads, group = (threadIdx.x - 64) / kConvThreads;
        const int n4 = (a_bytes + b_bytes) / 16;
        int slot = 0, turn = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int64_t tile = blockIdx.x; tile < D.ntiles && ok; tile += gridDim.x)
            for (int s = 0; s < nstage && ok; ++s, turn ^= 1) {
                if (turn == group) {
                    ok = __all_sync(0xffffffffu, tc::mbar_wait(&S.full[slot], phase, kDWaitLimit) && !aborted());
                    if (!ok) {
                        if (lane == 0) failed();
                        break;
                    }
                    const float4* xs = reinterpret_cast<const float4*>(S.x[slot]);
                    float4* ls = reinterpret_cast<float4*>(S.lo[SPLIT ? slot : 0]);
                    for (int i0 = ct; i0 < n4; i0 += kBatch * kConvThreads) {
                        float4 v[kBatch];
#pragma unroll
                        for (int u = 0; u < kBatch; ++u)
                            if (i0 + u * kConvThreads < n4) v[u] = xs[i0 + u * kConvThreads];
#pragma unroll
                        for (int u = 0; u < kBatch; ++u)
                            if (i0 + u * kConvThreads < n4)
                                ls[i0 + u * kConvThreads] =
                                    make_float4(v[u].x - to_tf32(v[u].x), v[u].y - to_tf32(v[u].y),
                                                v[u].z - to_tf32(v[u].z), v[u].w - to_tf32(v[u].w));
                    }
                    tc::fence_proxy_async();              // the tensor cores read what was written
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(&S.conv[slot]);
                }
                if (++slot == ST) {
                    slot = 0;
                    phase ^= 1u;
                }
            }
    } else {
        // ---- epilogue: TMEM lane quadrant warp % 4 holds rows 32 (warp % 4) ..; kDEpiCols columns per
        // pass through this warp's staging, then whole row segments, eight rows in flight
        const int q = warp & 3, ew = warp - epi0, half = ew >> 2;
        uint32_t k = 0;
        for (int64_t tile = blockIdx.x; tile < D.ntiles; tile += gridDim.x, ++k) {
            const int64_t rest = tile / D.ntm;
            const int tm = (int)(tile - rest * D.ntm), tn = (int)(rest % D.ntn);
            const int64_t b = rest / D.ntn;
            const uint32_t buf = k & 1u;
            const bool ok = __all_sync(0xffffffffu, tc::mbar_wait(&S.acc_full[buf], (k >> 1) & 1u, kDWaitLimit) &&
                                                        !aborted());
            if (!ok) {
                if (lane == 0) failed();
                break;
            }
            tc::fence_after_sync();
            float* Cb = D.C + b * D.n * D.n;
            const float* Ib = D.Cin + b * D.n * D.n;
            const int r0 = tm * kDM + 32 * q;
            const int rows = min(32, D.n - r0);
            for (int c0 = kDEpiCols * half; c0 < NT; c0 += 2 * kDEpiCols) {
                const int cw = min(kDEpiCols, NT - c0);
                __syncwarp();                             // the last pass's rows are written
                for (int c = 0; c < cw; c += 16) {
                    float v[16];
                    tc::tmem_ld16(tmem + buf * kDNMax + (uint32_t)(c0 + c) + ((uint32_t)(32 * q) << 16), v);
#pragma unroll
                    for (int x = 0; x < 16; ++x) S.out[ew][lane][c + x] = v[x];
                }
                if (c0 + 2 * kDEpiCols >= NT) {           // this warp's part of the accumulator is read
                    tc::fence_before_sync();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(&S.acc_empty[buf]);
                }
                __syncwarp();
                const int col = tn * NT + c0 + lane;
                if (lane < cw && col < D.n) {
                    const int64_t o = (int64_t)r0 * D.n + col;
                    for (int rb = 0; rb < rows; rb += 8) {
                        float v[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u) v[u] = D.alpha * S.out[ew][rb + u][lane];
                        if (D.beta != 0.f) {
                            float ci[8];
#pragma unroll
                            for (int u = 0; u < 8; ++u) ci[u] = rb + u < rows ? Ib[o + (int64_t)(rb + u) * D.n] : 0.f;
#pragma unroll
                            for (int u = 0; u < 8; ++u) v[u] = v[u] + D.beta * ci[u];
                        }
#pragma unroll
                        for (int u = 0; u < 8; ++u)
                            if (rb + u < rows) Cb[o + (int64_t)(rb + u) * D.n] = v[u];
                    }
                }
            }
            if (kDEpiCols * half >= NT) {                 // (a narrow tile leaves this warp no pass)
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&S.acc_empty[buf]);
            }
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, 2 * kDNMax);
    }
}

// A batch of n x n matrices with rows of ld floats (a multiple of 4, so that tensor maps can read
// them): transposed (64 x 64 tiles through shared memory, 16 loads in flight per thread) or copied.
__global__ void __launch_bounds__(256) k_dense_transpose(int64_t nb, int n, int ld, const float* __restrict__ B,
                                                         float* __restrict__ Bt) {
    __shared__ float t[64][65];
    const int tiles = (n + 63) / 64, tx = threadIdx.x & 63, ty = threadIdx.x >> 6;
    const int64_t total = nb * tiles * tiles;
    for (int64_t w = blockIdx.x; w < total; w += gridDim.x) {
        const int64_t m = w / ((int64_t)tiles * tiles);
        const int rest = (int)(w - m * tiles * tiles);
        const int ti = rest / tiles, tj = rest - ti * tiles;
        const float* src = B + m * n * n;
        float* dst = Bt + m * n * ld;
        const int j0 = tj * 64 + tx;
        float v[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) {
            const int i = ti * 64 + ty + 4 * u;
            v[u] = (i < n && j0 < n) ? src[(int64_t)i * n + j0] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 16; ++u) t[ty + 4 * u][tx] = v[u];
        __syncthreads();
        const int i0 = ti * 64 + tx;
#pragma unroll
        for (int u = 0; u < 16; ++u) {
            const int j = tj * 64 + ty + 4 * u;
            if (i0 < n && j < n) dst[(int64_t)j * ld + i0] = t[tx][ty + 4 * u];
        }
        __syncthreads();
    }
}
__global__ void __launch_bounds__(256) k_dense_pad(int64_t rows, int n, int ld, const float* __restrict__ A,
                                                   float* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t r = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < rows; r += warps)
        for (int c = lane; c < n; c += 32) out[r * ld + c] = A[r * n + c];
}

// FP64: C tile 64 x 64 per CTA of 256 threads, each a 4 x 4 register tile; K in slices of 16
// through shared memory.
constexpr int kF = 64, kFK = 16;

__global__ void __launch_bounds__(256) k_dense_f64(int n, double alpha, const double* __restrict__ A,
                                                   const double* __restrict__ B, double beta, const double* Cin, double* C) {
    __shared__ double sa[kFK][kF + 1];   // A slice transposed: sa[k][i]
    __shared__ double sb[kFK][kF + 1];
    const int64_t b = blockIdx.z;
    const int i0 = blockIdx.y * kF, j0 = blockIdx.x * kF;
    const double* a = A + b * n * n;
    const double* bb = B + b * n * n;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    double acc[4][4] = {};
    for (int k0 = 0; k0 < n; k0 += kFK) {
        for (int e = threadIdx.x; e < kF * kFK; e += 256) {
            const int r = e / kFK, c = e % kFK;          // A: row i0 + r, column k0 + c
            sa[c][r] = (i0 + r < n && k0 + c < n) ? a[(int64_t)(i0 + r) * n + k0 + c] : 0.0;
            const int kr = e / kF, jc = e % kF;          // B: row k0 + kr, column j0 + jc
            sb[kr][jc] = (k0 + kr < n && j0 + jc < n) ? bb[(int64_t)(k0 + kr) * n + j0 + jc] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kFK; ++k) {
            double av[4], bv[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                av[x] = sa[k][ty + 16 * x];
                bv[x] = sb[k][tx + 16 * x];
            }
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
                for (int y = 0; y < 4; ++y) acc[x][y] = fma(av[x], bv[y], acc[x][y]);
        }
        __syncthreads();
    }
    double* c = C + b * n * n;
    const double* ci = Cin + b * n * n;
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            const int i = i0 + ty + 16 * x, j = j0 + tx + 16 * y;
            if (i < n && j < n) {
                const int64_t p = (int64_t)i * n + j;
                c[p] = beta == 0.0 ? alpha * acc[x][y] : alpha * acc[x][y] + beta * ci[p];
            }
        }
}

}  // namespace

void dense_gemm_f64(int64_t nb, int n, double alpha, const double* A, const double* B, double beta, const double* Cin,
                    double* C, cudaStream_t s) {
    if (nb <= 0 || n <= 0) return;
    if (nb > 65535) fail(DBCSR_ECAPACITY, "dense_gemm: more than 65535 matrices in one batch");
    const dim3 grid((unsigned)ceil_div(n, kF), (unsigned)ceil_div(n, kF), (unsigned)nb);
    k_dense_f64<<<grid, 256, 0, s>>>(n, alpha, A, B, beta, Cin, C);
    DBG_LAUNCH_CK();
}

namespace {

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        DBG_CK(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q));
        if (q != cudaDriverEntryPointSuccess || !p) fail(DBCSR_ECUDA, "dense_gemm: cuTensorMapEncodeTiled not found");
        fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

// Tensor map over a batch of n x n row-major FP32 matrices with rows of ld floats (a multiple of 4):
// boxes of 16 columns x rows rows of one matrix, 64-byte swizzled.
CUtensorMap batch_map(const float* base, int n, int ld, int64_t nb, int rows) {
    CUtensorMap m;
    const cuuint64_t dims[3] = {(cuuint64_t)n, (cuuint64_t)n, (cuuint64_t)nb};
    const cuuint64_t strides[2] = {(cuuint64_t)ld * 4, (cuuint64_t)n * ld * 4};
    const cuuint32_t box[3] = {(cuuint32_t)kTK, (cuuint32_t)rows, 1};
    const cuuint32_t es[3] = {1, 1, 1};
    const CUresult r = tensor_map_encoder()(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(base), dims,
                                            strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                            CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) fail(DBCSR_ECUDA, "dense_gemm: cuTensorMapEncodeTiled failed");
    return m;
}

template <bool SPLIT>
void launch_tf32(const CUtensorMap& ma, const CUtensorMap& mb, const TmaArgs& d, cudaStream_t s) {
    const size_t sm = sizeof(TmaShared<SPLIT>) + 1024;
    allow_dyn_smem(k_dense_tf32<SPLIT>, sm);
    const unsigned grid = (unsigned)std::min<int64_t>(d.ntiles, (int64_t)num_sms());
    k_dense_tf32<SPLIT><<<grid, 32 * (2 + (SPLIT ? kTConvWarps : 0) + kDEpiWarps), sm, s>>>(ma, mb, d);
    DBG_LAUNCH_CK();
}

}  // namespace

DenseScratch::DenseScratch(cudaStream_t s) {
    err.alloc(1, s);
    err.zero();
}

void DenseScratch::check(cudaStream_t s) {
    int e = 0;
    DBG_CK(cudaMemcpyAsync(&e, err.p, sizeof(int), cudaMemcpyDeviceToHost, s));
    DBG_CK(cudaStreamSynchronize(s));
    if (e) fail(DBCSR_ETIMEOUT, "dense_gemm: a wait of the tensor-core kernel ran out");
}

void dense_gemm_tf32(int64_t nb, int n, float alpha, const float* A, const float* B, float beta, const float* Cin,
                     float* C, bool split, DenseScratch& w, cudaStream_t s) {
    if (nb <= 0 || n <= 0) return;
    if (nb > 65535) fail(DBCSR_ECAPACITY, "dense_gemm: more than 65535 matrices in one batch");
    const int ld = (n + 3) & ~3;
    // N tiles of equal width (a multiple of 16, at most 256), as many as give the shortest run of
    // whole waves: an MMA takes NT / 2 clocks, at least about 66 (measured), and a tile about 20 of
    // those clocks per K step besides.  (58 matrices of 432 x 432: 3.05 waves of 224 columns run as
    // 4, 4.6 waves of 144 columns as 5 shorter ones.)
    const int ntm = (int)ceil_div(n, kDM);
    int ntn = 1, NT = 0;
    int64_t best = 0;
    for (int t = (int)ceil_div(n, kDNMax); t <= (int)ceil_div(n, 64) || !NT; ++t) {
        const int w = (int)ceil_div(ceil_div(n, t), 16) * 16;
        const int64_t cost = ceil_div(nb * ntm * t, num_sms()) * (std::max(w / 2, 66) + 20);
        if (!NT || cost < best) {
            best = cost;
            ntn = t;
            NT = w;
        }
    }
    const int64_t need = nb * n * (int64_t)ld;
    if (w.bt.n < need) w.bt.alloc(need, s);
    const int64_t tiles = nb * ceil_div(n, 64) * ceil_div(n, 64);
    k_dense_transpose<<<grid_for(tiles, 1, (int64_t)num_sms() * 8), 256, 0, s>>>(nb, n, ld, B, w.bt.p);
    DBG_LAUNCH_CK();
    const float* a = A;
    // tensor maps want 16-byte rows; and a C over A must not be written while A's tiles are read
    const auto pa = reinterpret_cast<uintptr_t>(A), pc = reinterpret_cast<uintptr_t>(C);
    const uintptr_t bytes = (uintptr_t)nb * n * n * sizeof(float);
    if (ld != n || (pa & 15) != 0 || (pa < pc + bytes && pc < pa + bytes)) {
        if (w.a.n < need) w.a.alloc(need, s);
        k_dense_pad<<<grid_for(nb * n, 8), 256, 0, s>>>(nb * n, n, ld, A, w.a.p);
        DBG_LAUNCH_CK();
        a = w.a.p;
    }
    const CUtensorMap ma = batch_map(a, n, ld, nb, kDM), mb = batch_map(w.bt.p, n, ld, nb, NT);
    const TmaArgs d{n, ntm, ntn, NT, nb * ntm * ntn, alpha, beta, Cin, C, w.err.p};
    if (split) launch_tf32<true>(ma, mb, d, s);
    else launch_tf32<false>(ma, mb, d, s);
}

}  // namespace dbg

extern "C" dbcsr_status dbcsr_dense_multiply(int32_t prec, int64_t nb, int32_t n, double alpha, const void* A,
                                             const void* B, double beta, void* C, void* stream) {
    try {
        if (nb < 0 || n < 0 || (nb > 0 && n > 0 && (!A || !B || !C)))
            dbg::fail(DBCSR_EINVAL, "dense_multiply: bad argument");
        cudaStream_t s = (cudaStream_t)stream;
        if (prec == DBCSR_FP64) {
            dbg::dense_gemm_f64(nb, n, alpha, (const double*)A, (const double*)B, beta, (const double*)C, (double*)C, s);
            DBG_CK(cudaStreamSynchronize(s));
        } else if (prec == DBCSR_TF32 || prec == DBCSR_TF32X3) {
            dbg::DenseScratch w(s);
            dbg::dense_gemm_tf32(nb, n, (float)alpha, (const float*)A, (const float*)B, (float)beta, (const float*)C,
                                 (float*)C, prec == DBCSR_TF32X3, w, s);
            w.check(s);
        } else {
            dbg::fail(DBCSR_EINVAL, "dense_multiply: prec must be DBCSR_FP64, DBCSR_TF32 or DBCSR_TF32X3");
        }
        dbg::set_last_error("");
        return DBCSR_OK;
    } catch (const dbg::Error& e) {
        dbg::set_last_error(e.what());
        return e.code;
    }
}
