// Traces and the Gershgorin bound.  All reductions are deterministic: per-block
// or per-row partials in a fixed order, then det_sum's fixed tree.
#include "common.cuh"

namespace dbg {
namespace {

__device__ __forceinline__ int64_t find_block(const int64_t* __restrict__ rp, const int32_t* __restrict__ col, int32_t row,
                                              int32_t c) {
    int64_t lo = rp[row], hi = rp[row + 1];
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (col[mid] < c) lo = mid + 1; else hi = mid;
    }
    return (lo < rp[row + 1] && col[lo] == c) ? lo : -1;
}

// part[I] = trace of diagonal block I (0 if absent).
__global__ void k_trace_rows(int32_t nblk, const int32_t* __restrict__ bs, const int64_t* __restrict__ rp,
                             const int32_t* __restrict__ col, const int64_t* __restrict__ off,
                             const double* __restrict__ data, double* __restrict__ part) {
    for (int32_t I = blockIdx.x * blockDim.x + threadIdx.x; I < nblk; I += gridDim.x * blockDim.x) {
        const int64_t q = find_block(rp, col, I, I);
        double s = 0.0;
        if (q >= 0) {
            const int m = bs[I];
            const double* x = data + off[q];
            for (int i = 0; i < m; ++i) s += x[i * m + i];
        }
        part[I] = s;
    }
}

// One warp per block A_IJ: part[b] = <A_IJ, B_JI^T> (0 if B_JI is absent).
__global__ void k_trace_product_blocks(int64_t nb, const int32_t* __restrict__ bs, const int32_t* __restrict__ a_row,
                                       const int32_t* __restrict__ a_col, const int64_t* __restrict__ a_off,
                                       const double* __restrict__ a_data, const int64_t* __restrict__ b_rp,
                                       const int32_t* __restrict__ b_col, const int64_t* __restrict__ b_off,
                                       const double* __restrict__ b_data, double* __restrict__ part) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t b = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); b < nb; b += warps) {
        const int32_t I = a_row[b], J = a_col[b];
        const int64_t q = find_block(b_rp, b_col, J, I);
        double s = 0.0;
        if (q >= 0) {
            const int m = bs[I], n = bs[J];
            const double* x = a_data + a_off[b];
            const double* y = b_data + b_off[q];
            for (int e = lane; e < m * n; e += 32) {
                const int i = e / n, j = e - i * n;
                s = fma(x[e], y[j * m + i], s);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) part[b] = s;
    }
}

// One CTA per block row I, one lane of its first warp per matrix row i: sum_j |(A - mu 1)_ij| in
// ascending column order; the maximum over rows (of each system, with row_sys) is taken with an integer
// atomicMax on the bits of the non-negative sum.  The sums are serial chains, bound by the latency of
// their loads when each lane reads its own row (0.16 ms for the 736 columns of 32 waters).  The row's
// blocks lie one after the other in memory: all threads fetch a stage of whole blocks into registers
// while the first warp adds up the last one, and lay it out in shared memory by matrix rows: the whole
// call takes 65 us there now.
constexpr int kGershThreads = 256, kGershStage = 2048, kGershPer = kGershStage / kGershThreads;
__global__ void __launch_bounds__(kGershThreads)
    k_gershgorin(int32_t nblk, const int32_t* __restrict__ bs, const int64_t* __restrict__ rp,
                 const int32_t* __restrict__ col, const int64_t* __restrict__ off,
                 const double* __restrict__ data, double mu, const int32_t* __restrict__ row_sys,
                 const double* __restrict__ mu_sys, unsigned long long* __restrict__ maxbits) {
    static_assert(kGershStage >= kMaxBlock * kMaxBlock, "a stage holds at least one block");
    __shared__ double rows[kGershStage + kMaxBlock];    // matrix row i of the stage at i (columns | 1): odd strides
    __shared__ int s_n[kGershThreads], s_c[kGershThreads];   // a staged block's width and first column; n < 0: diagonal
    const int t = threadIdx.x;
    for (int32_t I = blockIdx.x; I < nblk; I += gridDim.x) {
        const int m = bs[I], sys = row_sys ? row_sys[I] : 0;
        const double shift = mu_sys ? mu_sys[sys] : mu;
        const int64_t q1 = rp[I + 1];
        double s = 0.0, v[kGershPer];
        bool has_diag = false;
        int cols = 0;                                    // columns of the stage in shared memory
        for (int64_t q = rp[I];; ) {
            // the next stage: as many whole blocks as fit, at most one per thread, into registers
            int nb = 0, cnt = 0;
            if (q < q1) {
                const int64_t o0 = off[q], o = q + t < q1 ? off[q + t] : 0, e = q + t < q1 ? off[q + t + 1] : 0;
                nb = __syncthreads_count(q + t < q1 && e - o0 <= kGershStage);
                if (t < nb) {
                    const int32_t J = col[q + t];
                    const int n = (int)(e - o) / m;
                    s_n[t] = J == I ? -n : n;
                    s_c[t] = (int)(o - o0) / m;
                }
                cnt = (int)(off[q + nb] - o0);
#pragma unroll
                for (int u = 0; u < kGershPer; ++u)
                    if (t + u * kGershThreads < cnt) v[u] = data[o0 + t + u * kGershThreads];
            }
            // the first warp adds up the stage in shared memory
            if (t < m) {
                const double* x = rows + t * (cols | 1);
                int c = 0;
                for (; c + 8 <= cols; c += 8) {
                    double w[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) w[u] = x[c + u];
#pragma unroll
                    for (int u = 0; u < 8; ++u) s += w[u];
                }
                for (; c < cols; ++c) s += x[c];
            }
            if (!nb) break;
            __syncthreads();
            cols = cnt / m;
#pragma unroll
            for (int u = 0; u < kGershPer; ++u) {
                const int x = t + u * kGershThreads;
                if (x >= cnt) continue;
                int lo = 0, hi = nb - 1;                 // the block that holds element x
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (s_c[mid] * m <= x) lo = mid; else hi = mid - 1;
                }
                const int n = abs(s_n[lo]), r = x - s_c[lo] * m, i = r / n, j = r - i * n;
                if (s_n[lo] < 0 && i == j) v[u] -= shift;
                rows[i * (cols | 1) + s_c[lo] + j] = fabs(v[u]);
            }
            if (t < m)
                for (int b = 0; b < nb; ++b) has_diag |= s_n[b] < 0;
            __syncthreads();
            q += nb;
        }
        if (t < m) {
            if (!has_diag) s += fabs(shift);
            atomicMax(maxbits + sys, (unsigned long long)__double_as_longlong(s));
        }
        __syncthreads();
    }
}

}  // namespace

double trace(dbcsr_matrix_* m) {
    check_finalized(m);
    cudaStream_t s = m->stream;
    DBuf<double> part, out;
    part.alloc(m->nblk, s);
    out.alloc(1, s);
    k_trace_rows<<<grid_for(m->nblk, 128), 128, 0, s>>>(m->nblk, m->bs.p, m->rp.p, m->col.p, m->off.p, m->data.p,
                                                        part.p);
    DBG_LAUNCH_CK();
    det_sum(part.p, m->nblk, out.p, s);
    return read_f64(out.p, s);
}

double trace_product(dbcsr_matrix_* a, dbcsr_matrix_* b) {
    check_finalized(a);
    check_finalized(b);
    if (a->h_bs != b->h_bs) fail(DBCSR_EINVAL, "trace_product: block sizes differ");
    cudaStream_t s = a->stream;
    if (b->stream != s) DBG_CK(cudaStreamSynchronize(b->stream));
    DBuf<double> part, out;
    part.alloc(std::max<int64_t>(a->nnzb, 1), s);
    out.alloc(1, s);
    if (a->nnzb) {
        k_trace_product_blocks<<<grid_for(a->nnzb, 8), 256, 0, s>>>(a->nnzb, a->bs.p, a->row.p, a->col.p, a->off.p,
                                                                    a->data.p, b->rp.p, b->col.p, b->off.p, b->data.p,
                                                                    part.p);
        DBG_LAUNCH_CK();
    }
    det_sum(part.p, a->nnzb, out.p, s);
    return read_f64(out.p, s);
}

double gershgorin(dbcsr_matrix_* m, double mu) {
    check_finalized(m);
    cudaStream_t s = m->stream;
    DBuf<double> out;
    out.alloc(1, s);
    out.zero();
    k_gershgorin<<<grid_for(m->nblk, 1), kGershThreads, 0, s>>>(m->nblk, m->bs.p, m->rp.p, m->col.p, m->off.p, m->data.p,
                                                                mu, nullptr, nullptr, (unsigned long long*)out.p);
    DBG_LAUNCH_CK();
    return read_f64(out.p, s);
}

void gershgorin_sys(const dbcsr_matrix_* m, const int32_t* row_sys, const double* mu, double* bound, cudaStream_t s) {
    k_gershgorin<<<grid_for(m->nblk, 1), kGershThreads, 0, s>>>(m->nblk, m->bs.p, m->rp.p, m->col.p, m->off.p, m->data.p,
                                                                0.0, row_sys, mu, (unsigned long long*)bound);
    DBG_LAUNCH_CK();
}

void trace_product_parts_into(dbcsr_matrix_* a, dbcsr_matrix_* b, double* part, cudaStream_t s) {
    if (a->nnzb == 0) return;
    k_trace_product_blocks<<<grid_for(a->nnzb, 8), 256, 0, s>>>(a->nnzb, a->bs.p, a->row.p, a->col.p, a->off.p,
                                                                a->data.p, b->rp.p, b->col.p, b->off.p, b->data.p,
                                                                part);
    DBG_LAUNCH_CK();
}

}  // namespace dbg
