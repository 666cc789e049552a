// Group tiles of a block-sparse matrix, shared by the tensor-core tiers: the nonzero tiles (group
// row, group column) of a block pattern, the stacks of operand tiles that each tile of a product
// sums, and the role of a block in a symmetric product.  Internal to the translation units that include it.
#pragma once

#include <algorithm>
#include <cstdint>

#include "common.cuh"

namespace dbg {
namespace {

// role of formed block k: 0 computed, 1 copied from its twin, 2 dropped.
// sym = 1 (mirror): one twin computed, the other copied; sym = 2 (average): both twins
// computed and then replaced by their symmetric mean; blocks without a formed twin
// are dropped in both modes.
// by_group: the twin of the lower group is computed (grp, the groups of the blocks), so that all the
// computed blocks between two groups lie in one group tile; otherwise the block I < J.
__device__ __forceinline__ int block_role(int sym, int32_t I, int32_t J, int64_t mirror, const int32_t* grp,
                                          int by_group) {
    if (!sym || I == J) return 0;
    if (mirror < 0) return 2;
    if (sym == 2) return 0;
    const bool first = by_group ? (grp[I] < grp[J] || (grp[I] == grp[J] && I < J)) : I < J;
    return first ? 0 : 1;
}

__device__ int lt_block_scan(int v, int* sh, int& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int t = lane < nw ? sh[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        sh[lane] = t;
    }
    __syncthreads();
    const int excl = (warp ? sh[warp - 1] : 0) + x - v;
    total = sh[nw - 1];
    __syncthreads();
    return excl;
}

__device__ __forceinline__ int lt_rank(const uint32_t* bm, const int* wpre, int32_t g) {
    return wpre[g >> 5] + __popc(bm[g >> 5] & ((1u << (g & 31)) - 1u));
}

struct GView {
    const int32_t* g_of; const int32_t* g_pos; const int32_t* g_ptr; const int32_t* g_mem; const int32_t* g_w;
};

// Bitmap (and prefix popcounts) of the groups reached by the blocks of group row G of a
// block pattern (rp, col); use[q] (nullable) selects blocks.  Returns the number of groups.
__device__ int lt_group_row(const GView& g, int32_t G, const int64_t* rp, const int32_t* col, const uint8_t* use,
                            uint32_t* bm, int* wpre, int nwords, int* sh) {
    for (int w = threadIdx.x; w < nwords; w += blockDim.x) bm[w] = 0u;
    __syncthreads();
    for (int32_t m = g.g_ptr[G]; m < g.g_ptr[G + 1]; ++m) {
        const int32_t I = g.g_mem[m];
        for (int64_t q = rp[I] + threadIdx.x; q < rp[I + 1]; q += blockDim.x)
            if (!use || use[q]) {
                const int32_t c = g.g_of[col[q]];
                atomicOr(&bm[c >> 5], 1u << (c & 31));
            }
    }
    __syncthreads();
    const int per = (nwords + blockDim.x - 1) / blockDim.x;
    const int lo = min(nwords, (int)threadIdx.x * per), hi = min(nwords, lo + per);
    int s = 0;
    for (int w = lo; w < hi; ++w) s += __popc(bm[w]);
    int total;
    int run = lt_block_scan(s, sh, total);
    for (int w = lo; w < hi; ++w) {
        wpre[w] = run;
        run += __popc(bm[w]);
    }
    __syncthreads();
    return total;
}

// fill == 0: cnt[G] = number of tiles of group row G.  fill == 1: tile rows/columns and the
// tile of every selected block (blk_tile[q], -1 for blocks not selected).
__global__ void k_gt_pattern(int32_t ngrp, GView g, const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                             const uint8_t* __restrict__ use, int nwords, int fill, int64_t* __restrict__ cnt,
                             const int64_t* __restrict__ t_rp, int32_t* __restrict__ t_row,
                             int32_t* __restrict__ t_col, int32_t* __restrict__ blk_tile) {
    extern __shared__ uint32_t lt_smem[];
    __shared__ int sh[32];
    uint32_t* bm = lt_smem;
    int* wpre = (int*)(lt_smem + nwords);
    for (int32_t G = blockIdx.x; G < ngrp; G += gridDim.x) {
        const int n = lt_group_row(g, G, rp, col, use, bm, wpre, nwords, sh);
        if (!fill) {
            if (threadIdx.x == 0) cnt[G] = n;
        } else {
            const int64_t base = t_rp[G];
            for (int w = threadIdx.x; w < nwords; w += blockDim.x) {
                uint32_t bits = bm[w];
                int r = wpre[w];
                while (bits) {
                    const int b = __ffs(bits) - 1;
                    bits &= bits - 1;
                    t_row[base + r] = G;
                    t_col[base + r] = w * 32 + b;
                    ++r;
                }
            }
            if (blk_tile)
                for (int32_t m = g.g_ptr[G]; m < g.g_ptr[G + 1]; ++m) {
                    const int32_t I = g.g_mem[m];
                    for (int64_t q = rp[I] + threadIdx.x; q < rp[I + 1]; q += blockDim.x)
                        blk_tile[q] = (!use || use[q]) ? (int32_t)(base + lt_rank(bm, wpre, g.g_of[col[q]])) : -1;
                }
        }
        __syncthreads();
    }
}

__device__ __forceinline__ int lt_ksteps(int w) { return (w + 15) >> 4; }

__device__ __forceinline__ int lt_rows(int w) { return (w + 7) & ~7; }

// For a symmetric pattern: tT[t] = the tile (c, r) of tile t = (r, c).
__global__ void k_gt_transpose(int64_t nt, const int32_t* __restrict__ t_row, const int32_t* __restrict__ t_col,
                               const int64_t* __restrict__ t_rp, int32_t* __restrict__ tT, int* __restrict__ err) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nt; t += (int64_t)gridDim.x * blockDim.x) {
        const int32_t r = t_row[t], c = t_col[t];
        int64_t lo = t_rp[c], hi = t_rp[c + 1];
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (t_col[mid] < r) lo = mid + 1; else hi = mid;
        }
        const bool ok = lo < t_rp[c + 1] && t_col[lo] == r;
        tT[t] = ok ? (int32_t)lo : -1;
        if (!ok) atomicExch(err, 2);
    }
}

// ------------------------------------------------------------------ product stacks
struct StackArgs {
    GView g;
    const int64_t* c_trp; const int32_t* c_tcol;          // C tiles by group row
    const int64_t* a_trp; const int32_t* a_tcol;          // A tiles by group row (A-style)
    const int64_t* b_trp; const int32_t* b_tcol;          // B tiles by K group row
    const int32_t* b_map;                                 // B operand tile -> packed tile (nullable)
    int64_t* cnt;                                         // count pass: entries per C tile (global)
    const int64_t* s_ptr;                                 // fill pass: stack start of each C tile
    int32_t* st_a; int32_t* st_b;
    int32_t* cursor;                                      // global cursors (when not in shared memory)
    int fill, use_smem;
};

// Per group row G: for every A tile (G, G'') in ascending G'' and every B tile (G'', G')
// whose C tile (G, G') exists, one stack entry of that C tile.  Entries of a C tile are in
// ascending G''.
__global__ void k_gt_stack(int32_t ngrp, StackArgs S, int nwords) {
    extern __shared__ uint32_t lt_smem[];
    __shared__ int sh[32];
    uint32_t* bm = lt_smem;
    int* wpre = (int*)(lt_smem + nwords);
    int32_t* cur = (int32_t*)(wpre + nwords);
    for (int32_t G = blockIdx.x; G < ngrp; G += gridDim.x) {
        for (int w = threadIdx.x; w < nwords; w += blockDim.x) bm[w] = 0u;
        __syncthreads();
        const int64_t c0 = S.c_trp[G], c1 = S.c_trp[G + 1];
        for (int64_t t = c0 + threadIdx.x; t < c1; t += blockDim.x) {
            const int32_t c = S.c_tcol[t];
            atomicOr(&bm[c >> 5], 1u << (c & 31));
        }
        __syncthreads();
        {
            const int per = (nwords + blockDim.x - 1) / blockDim.x;
            const int lo = min(nwords, (int)threadIdx.x * per), hi = min(nwords, lo + per);
            int s = 0;
            for (int w = lo; w < hi; ++w) s += __popc(bm[w]);
            int total;
            int run = lt_block_scan(s, sh, total);
            for (int w = lo; w < hi; ++w) {
                wpre[w] = run;
                run += __popc(bm[w]);
            }
        }
        const int nct = (int)(c1 - c0);
        int32_t* cc = S.use_smem ? cur : S.cursor + c0;
        for (int r = threadIdx.x; r < nct; r += blockDim.x) cc[r] = 0;
        __syncthreads();
        for (int64_t ta = S.a_trp[G]; ta < S.a_trp[G + 1]; ++ta) {
            const int32_t K = S.a_tcol[ta];
            for (int64_t tb = S.b_trp[K] + threadIdx.x; tb < S.b_trp[K + 1]; tb += blockDim.x) {
                const int32_t c = S.b_tcol[tb];
                if (!(bm[c >> 5] & (1u << (c & 31)))) continue;
                // a B tile without its transposed twin (an asymmetric pattern declared symmetric) is
                // left out; the k_gt_transpose error flag reports it
                const int32_t bt = S.b_map ? S.b_map[tb] : (int32_t)tb;
                if (bt < 0) continue;
                const int r = lt_rank(bm, wpre, c);
                const int32_t at = cc[r];
                cc[r] = at + 1;
                if (S.fill) {
                    const int64_t pos = S.s_ptr[c0 + r] + at;
                    S.st_a[pos] = (int32_t)ta;
                    S.st_b[pos] = bt;
                }
            }
            __syncthreads();
        }
        if (!S.fill)
            for (int r = threadIdx.x; r < nct; r += blockDim.x) S.cnt[c0 + r] = cc[r];
        __syncthreads();
    }
}

struct TilePattern {
    int64_t nt = 0;
    DBuf<int64_t> t_rp;          // [ngrp + 1]
    DBuf<int32_t> t_row, t_col;  // [nt]
    DBuf<int32_t> blk_tile;      // [nnzb] tile of every block
};

int pattern_words(int32_t ngrp) { return (ngrp + 31) / 32; }

TilePattern tile_pattern(const Groups& g, const int64_t* rp, const int32_t* col, const uint8_t* use, int64_t nnzb,
                         bool want_blk, cudaStream_t s) {
    TilePattern P;
    const int nwords = pattern_words(g.ngrp);
    const size_t sm = (size_t)2 * ((nwords + 1) & ~1) * sizeof(uint32_t);
    GView gv{g.g_of.p, g.g_pos.p, g.g_ptr.p, g.g_mem.p, g.g_w.p};
    DBuf<int64_t> cnt;
    cnt.alloc(g.ngrp, s);
    P.t_rp.alloc(g.ngrp + 1, s);
    allow_dyn_smem(k_gt_pattern, sm);
    const unsigned grid = (unsigned)std::min<int64_t>(g.ngrp, (int64_t)num_sms() * 8);
    k_gt_pattern<<<grid, 256, sm, s>>>(g.ngrp, gv, rp, col, use, nwords, 0, cnt.p, nullptr, nullptr, nullptr,
                                       nullptr);
    DBG_LAUNCH_CK();
    scan_exclusive(cnt.p, P.t_rp.p, g.ngrp, s);
    P.nt = read_i64(P.t_rp.p + g.ngrp, s);
    P.t_row.alloc(std::max<int64_t>(P.nt, 1), s);
    P.t_col.alloc(std::max<int64_t>(P.nt, 1), s);
    if (want_blk) P.blk_tile.alloc(std::max<int64_t>(nnzb, 1), s);
    k_gt_pattern<<<grid, 256, sm, s>>>(g.ngrp, gv, rp, col, use, nwords, 1, nullptr, P.t_rp.p, P.t_row.p, P.t_col.p,
                                       want_blk ? P.blk_tile.p : nullptr);
    DBG_LAUNCH_CK();
    return P;
}

}  // namespace
}  // namespace dbg
