// rw_solve.cu -- the solve step of Algorithm 1: PCG with M = Y^T diag(D) Y.
//
//   z = M^-1 r:  Y^T w = r (backward), v = w / D, Y z = v (forward).
//
// Vectors are node-major [n, nrhs], so one node's right-hand sides share a
// DRAM sector and every gather serves all of them.  The triangular solves are
// sync-free: rows are visited in level order by a co-resident grid, each
// row's warp waits (bounded) until the values it depends on have left the
// "pending" state, computes its row and publishes it with one relaxed store.
// Scalars (alpha, beta, norms) stay on the device; the host reads one small
// status record per iteration.
#include <algorithm>
#include <cmath>
#include <mutex>

#include "rw_internal.h"

namespace rw {

constexpr int kDotParts = 1024;  // blocks of the dot-product producing kernels

// ---------------------------------------------------------------------------
// SpMV: y = A x for node-major vectors.  Optionally accumulates per-block
// partial dot products x.y (per right-hand side) for the PCG step.
//
// A block takes rows_per_pass consecutive rows at a time: their entries are
// one contiguous piece of the CSR arrays, copied to shared memory by all
// threads (every column and value is read from memory once, coalesced); then a
// group of G = NR * ES lanes per row sums it: lane (es, j) owns right-hand
// side j and entries es, es + ES, ... .  What bounds it is the FP64 pipe (2
// lane-FMAs per cycle and SM) and the gathers of x, one sector each, so a row
// gets few lanes: a warp-wide FMA then carries entries of 32 / G rows, and
// log2(ES) of the expensive FP64 additions across lanes serve them all.  With
// 32 / NR lanes per row, rows loaded one dependent access after the other, a
// call took 586 us on the 101 x 97 x 89 27-point grid with three right-hand
// sides and 406 us with one; now 249 and 237 us (1.0e11 gathers/s).
// Passes whose entries exceed the copy or that hold a row of more than
// kLongRow entries per lane sum their rows with all 32 lanes each, straight
// from memory; matrices of long rows take a warp per row throughout (k_spmv_rows).
//
// DIFF (the FP32 operator of the mixed mode): val holds A_ij (j != i) and, at
// the diagonal position, the excess e_i = A_ii + sum_j A_ij, and the row is
// applied as e_i x_i + sum_{j != i} A_ij (x_j - x_i).  Rounding an R-matrix to
// FP32 this way perturbs edge weights and excesses by a relative 2^-24 each,
// so the operator keeps the near-null space of a weakly grounded matrix
// (rounding A_ii itself would move a row sum by 2^-24 A_ii).
// ---------------------------------------------------------------------------
constexpr int kSpmvEntries = 2048;  // entries of a pass (24 KB of columns and FP64 values: eight blocks per SM)
constexpr int kSpmvRows = 512;      // rows of a pass
constexpr int kLongRow = 64;
// Average entries per row times right-hand sides (four at least) from which
// every row is summed by a warp (k_spmv_rows).  A pass of k_spmv then holds too
// few rows for the copy to pay, and from 1000 entries a row only one or two, so
// that most of the block idles.  k_spmv | k_spmv_rows, us: 6000 rows of 920
// entries 60 | 27 (one right-hand side), 430 | 180 (16); 8000 of 497 35 | 27 and
// 163 | 141; 30,000 of 129 42 | 36 and 154 | 132; 16 right-hand sides on 40,000 of
// 65 100 | 96 and on 60,000 of 33 88 | 83.  Below the line: 200,000 of 65 with one
// 89 | 134, with three 146 | 206.
constexpr int kLongRows = 512;

// RES: the true residual b - A x of PCG instead of A x: stored as FP32
// (out32) or FP64 where y is given, its squares in place of the dot products.
template <typename TA, typename TV, int NR, int ES, bool DIFF, bool RES>
__global__ void __launch_bounds__(256) k_spmv(int32_t n, const int32_t* __restrict__ rp,
                                              const int32_t* __restrict__ col,
                                              const TA* __restrict__ val, const TV* __restrict__ x,
                                              TV* __restrict__ y, int nrhs, int rows_per_pass, double* part,
                                              const double* __restrict__ b, int out32) {
    constexpr int G = NR * ES;
    static_assert(G <= 32 && 32 % G == 0, "lane group");
    __shared__ __align__(16) TA sval[kSpmvEntries];
    __shared__ int32_t scol[kSpmvEntries];
    __shared__ int32_t srp[kSpmvRows + 1];
    const int tid = (int)threadIdx.x, lane = (int)lane_id();
    double mydot = 0.0, wdot = 0.0;
    // lanes of right-hand side j, slice es of an ESX-lane row sum entries [s + es, e) of (c, a)
    auto term = [&](int32_t c, TA av, int32_t row, int j, TV xi) -> TV {
        const TV a = (TV)av;
        const TV xc = x[(size_t)c * nrhs + j];
        if (DIFF) return c == row ? a * xi : a * (xc - xi);
        return a * xc;
    };
    // the row's sum is complete: stores it, adds its part of the dot product
    auto finish = [&](size_t at, TV acc, double& dot) {
        if constexpr (RES) {
            const double t = b[at] - (double)acc;
            if (y && out32) reinterpret_cast<float*>(y)[at] = (float)t;
            else if (y) y[at] = (TV)t;
            dot += t * t;
        } else {
            y[at] = acc;
            if (part) dot += (double)x[at] * (double)acc;
        }
    };
    const int64_t npass = ((int64_t)n + rows_per_pass - 1) / rows_per_pass;
    for (int64_t ps = blockIdx.x; ps < npass; ps += gridDim.x) {
        const int32_t base = (int32_t)(ps * rows_per_pass);
        const int nr = min(rows_per_pass, n - base);
        for (int i = tid; i <= nr; i += 256) srp[i] = rp[base + i];
        __syncthreads();
        int longest = 0;
        for (int i = tid; i < nr; i += 256) longest = max(longest, srp[i + 1] - srp[i]);
        const int32_t s0 = srp[0];
        const int cnt = srp[nr] - s0;
        const bool direct = __syncthreads_or(longest > kLongRow * ES || cnt > kSpmvEntries || cnt < 0);
        if (!direct) {
            for (int i = tid; i < cnt; i += 256) {
                scol[i] = col[s0 + i];
                sval[i] = val[s0 + i];
            }
            __syncthreads();
            // one slice: nrhs lanes per row, no lane left over for a right-hand side past nrhs
            const int lanes = ES == 1 ? nrhs : G, set = 256 / lanes, mine = tid / lanes;
            const int j = ES == 1 ? tid - mine * lanes : tid % NR, es = ES == 1 ? 0 : (tid % G) / NR;
            const bool jok = mine < set && j < nrhs;
            for (int r0 = 0; r0 < nr; r0 += set) {
                const int r = r0 + mine;
                TV acc = TV(0);
                if (r < nr && jok) {
                    const int32_t row = base + r;
                    const TV xi = DIFF ? x[(size_t)row * nrhs + j] : TV(0);
                    const int e = srp[r + 1] - s0;
                    for (int p = srp[r] - s0 + es; p < e; p += 4 * ES) {  // four gathers in flight
                        TV t[4];
                        int32_t c[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            c[u] = p + u * ES < e ? scol[p + u * ES] : row;
                            t[u] = x[(size_t)c[u] * nrhs + j];
                        }
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            if (p + u * ES >= e) break;
                            const TV a = (TV)sval[p + u * ES];
                            if (DIFF) acc += c[u] == row ? a * xi : a * (t[u] - xi);
                            else acc += a * t[u];
                        }
                    }
                }
                if constexpr (ES > 1) {
#pragma unroll
                    for (int o = NR; o < G; o <<= 1) acc += __shfl_xor_sync(kFull, acc, o);
                }
                if (r < nr && jok && es == 0) finish((size_t)(base + r) * nrhs + j, acc, mydot);
            }
        } else {
            constexpr int EW = 32 / NR;
            const int j = lane % NR, es = lane / NR;
            const bool jok = j < nrhs;
            for (int r = tid >> 5; r < nr; r += 8) {
                const int32_t row = base + r;
                const TV xi = (DIFF && jok) ? x[(size_t)row * nrhs + j] : TV(0);
                TV acc = TV(0);
                if (jok)
                    for (int32_t p = srp[r] + es; p < srp[r + 1]; p += EW) acc += term(col[p], val[p], row, j, xi);
#pragma unroll
                for (int o = NR; o < 32; o <<= 1) acc += __shfl_xor_sync(kFull, acc, o);
                if (es == 0 && jok) finish((size_t)row * nrhs + j, acc, wdot);
            }
        }
        __syncthreads();
    }
    if (part) {
        // per right-hand side, the threads that hold it in thread order: mydot in the copied passes, wdot
        // (lanes l, l + NR, ... of a warp: right-hand side l % NR) in the others
        static_assert(sizeof(sval) >= 512 * sizeof(double), "the copy's room holds the sums");
        double* sdot = reinterpret_cast<double*>(sval);
        sdot[tid] = mydot;
        sdot[256 + tid] = wdot;
        __syncthreads();
        const int lanes = ES == 1 ? nrhs : NR;
        if (tid < nrhs) {
            double t = 0.0;
            for (int i = tid; i < 256; i += lanes) t += sdot[i];
            for (int i = tid; i < 256; i += NR) t += sdot[256 + i];
            part[(size_t)blockIdx.x * 16 + tid] = t;
        }
    }
}

// Matrices of long rows: a warp per row, straight from memory.  A kernel of its
// own: in k_spmv the loop cost every other matrix registers (spills, 253 -> 263 us
// on the 27-point grid above), and without the copy's shared memory L1 holds more
// of x.
template <typename TA, typename TV, int NR, bool DIFF, bool RES>
__global__ void __launch_bounds__(256) k_spmv_rows(int32_t n, const int32_t* __restrict__ rp,
                                                   const int32_t* __restrict__ col, const TA* __restrict__ val,
                                                   const TV* __restrict__ x, TV* __restrict__ y, int nrhs,
                                                   double* part, const double* __restrict__ b, int out32) {
    constexpr int EW = 32 / NR;
    __shared__ double sdot[8][NR];
    const int lane = (int)lane_id(), warp = (int)threadIdx.x >> 5;
    const int j = lane % NR, es = lane / NR;
    const bool jok = j < nrhs;
    double dot = 0.0;
    for (int64_t row = (int64_t)blockIdx.x * 8 + warp; row < n; row += (int64_t)gridDim.x * 8) {
        const int32_t s = rp[row], e = rp[row + 1];
        const size_t at = (size_t)row * nrhs + j;
        const TV xi = (DIFF && jok) ? x[at] : TV(0);
        TV acc = TV(0);
        if (jok)
            for (int32_t p = s + es; p < e; p += EW) {
                const int32_t c = col[p];
                const TV a = (TV)val[p], xc = x[(size_t)c * nrhs + j];
                if (DIFF) acc += c == row ? a * xi : a * (xc - xi);
                else acc += a * xc;
            }
#pragma unroll
        for (int o = NR; o < 32; o <<= 1) acc += __shfl_xor_sync(kFull, acc, o);
        if (es == 0 && jok) {
            if constexpr (RES) {
                const double t = b[at] - (double)acc;
                if (y && out32) reinterpret_cast<float*>(y)[at] = (float)t;
                else if (y) y[at] = (TV)t;
                dot += t * t;
            } else {
                y[at] = acc;
                if (part) dot += (double)x[at] * (double)acc;
            }
        }
    }
    if (part) {
        if (es == 0) sdot[warp][j] = dot;
        __syncthreads();
        if ((int)threadIdx.x < nrhs) {
            double t = 0.0;
            for (int w = 0; w < 8; ++w) t += sdot[w][threadIdx.x];
            part[(size_t)blockIdx.x * 16 + threadIdx.x] = t;
        }
    }
}

// FP32 operator of the mixed mode (see k_spmv): off-diagonals rounded, the
// diagonal slot replaced by the row's excess (FP64 sum of the row in column
// order, then rounded).  One thread per row.
__global__ void k_to_fp32_diff(int32_t n, const int32_t* __restrict__ rp, const int32_t* __restrict__ col,
                               const double* __restrict__ val, float* __restrict__ a32) {
    for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int32_t s = rp[i], e = rp[i + 1];
        double ex = 0.0;
        for (int32_t p = s; p < e; ++p) ex = __dadd_rn(ex, val[p]);
        for (int32_t p = s; p < e; ++p) a32[p] = col[p] == i ? (float)ex : (float)val[p];
    }
}

void launch_to_fp32_diff(int32_t n, const int32_t* rp, const int32_t* col, const double* val, float* a32,
                         cudaStream_t s, int num_sms) {
    RW_COUNT_LAUNCH();
    k_to_fp32_diff<<<grid_for(n, 256, num_sms * 8), 256, 0, s>>>(n, rp, col, val, a32);
}

// ---------------------------------------------------------------------------
// PCG vector kernels and device scalars.
// ---------------------------------------------------------------------------
struct PcgScalars {
    double bnorm2[16];
    double rho[16];
    double pq[16];
    double alpha[16];
    double rr[16];
    double tt[16];
    double beta[16];
    int active[16];
    int check[16];
    int iters[16];
    int broke;
    int any_active;
    int any_check;
    int pad;
};
static_assert(sizeof(PcgScalars) <= kSmallBytes, "the host copy lies in the context's pinned scratch");

// Threads of a block that work on an [n][nrhs] array element by element, each
// on one right-hand side (tid % nrhs): whole groups of nrhs threads.
__device__ __forceinline__ int rhs_threads(int nrhs) { return 256 / nrhs * nrhs; }

// Sum of v over the block's rhs_threads, per right-hand side, in a fixed order;
// threads j < nrhs hold the sums.
__device__ __forceinline__ double block_rhs_sum(double v, int nrhs) {
    __shared__ double red[256];
    const int tid = (int)threadIdx.x, groups = 256 / nrhs, g = tid / nrhs;
    red[tid] = v;
    __syncthreads();
    int w = 1;
    while (w < groups) w <<= 1;
    for (w >>= 1; w > 0; w >>= 1) {
        if (g < w && g + w < groups) red[tid] += red[tid + w * nrhs];
        __syncthreads();
    }
    const double r = red[tid];
    __syncthreads();
    return r;
}

enum ScalarOp { kOpBnorm = 0, kOpRho0, kOpAlpha, kOpResid, kOpTrue, kOpBeta, kOpReport };

// One block of 1024 threads: the partials part[nparts][16] of all right-hand
// sides in one round of loads (a thread takes partials b, b + 64, ... of one),
// then a fixed tree, then the step of Algorithm 1 by one thread each.  (Summed
// one right-hand side after the other the kernel took 10 us of every step.)
__global__ void __launch_bounds__(1024) k_scalars(PcgScalars* S, const double* part, int nparts,
                                                  int nrhs, int op, double tol, int it) {
    __shared__ double red[1024];
    const int tid = (int)threadIdx.x;
    double sum = 0.0;
    if (tid % 16 < nrhs)
        for (int b = tid / 16; b < nparts; b += 64) sum += part[(size_t)b * 16 + tid % 16];
    red[tid] = sum;
    __syncthreads();
    for (int w = 32; w > 0; w >>= 1) {
        if (tid < w * 16) red[tid] += red[tid + w * 16];
        __syncthreads();
    }
    if (tid < nrhs) {
        const int j = tid;
        const double v = red[j];
        switch (op) {
            case kOpBnorm:
                S->bnorm2[j] = v;
                S->active[j] = v > 0.0;
                S->iters[j] = 0;
                break;
            case kOpRho0:
                S->rho[j] = v;
                break;
            case kOpAlpha:
                S->pq[j] = v;
                if (S->active[j]) {
                    if (!(v > 0.0)) {
                        S->broke = 1;
                        S->active[j] = 0;
                        S->alpha[j] = 0.0;
                    } else {
                        S->alpha[j] = S->rho[j] / v;
                    }
                } else {
                    S->alpha[j] = 0.0;
                }
                break;
            case kOpResid:
                S->rr[j] = v;
                S->check[j] = S->active[j] && (sqrt(v) < tol * sqrt(S->bnorm2[j]));
                break;
            case kOpTrue:
                S->tt[j] = v;
                if (S->check[j] && sqrt(v) < tol * sqrt(S->bnorm2[j])) {
                    S->active[j] = 0;
                    S->iters[j] = it;
                }
                break;
            case kOpBeta:
                S->beta[j] = S->active[j] ? v / S->rho[j] : 0.0;
                S->rho[j] = v;
                break;
            case kOpReport:
                S->tt[j] = v;
                break;
        }
    }
    __syncthreads();
    if (tid == 0) {
        int a = 0, c = 0;
        for (int j = 0; j < nrhs; ++j) {
            a |= S->active[j];
            c |= S->check[j];
        }
        S->any_active = a;
        S->any_check = c;
        if (op == kOpTrue)
            for (int j = 0; j < nrhs; ++j) S->check[j] = 0;
    }
}

// The vector kernels of PCG work element by element over the node-major arrays
// (coalesced; a thread keeps one right-hand side, so its scalar and its one
// accumulator stay in registers) and are bound by memory: with a thread per node
// and accumulators for sixteen right-hand sides, reduced one after the other on
// the FP64 pipe, a dot product of 261,568 entries took 49 us and now takes 5.
template <typename F>
__device__ __forceinline__ void for_elements(int64_t n, int nrhs, F f) {
    const int t = rhs_threads(nrhs);
    if ((int)threadIdx.x >= t) return;
    const int64_t cnt = n * nrhs, step = (int64_t)gridDim.x * t;
    for (int64_t i = (int64_t)blockIdx.x * t + threadIdx.x; i < cnt; i += step) f(i);
}

// Per-block partial sums of a.b (and with a2 given a2.b2) per right-hand side
// into part[blockIdx][j] (and part2).
template <typename TA, typename TB>
__global__ void __launch_bounds__(256) k_dot(const TA* __restrict__ a, const TB* __restrict__ b, int64_t n, int nrhs,
                                             double* part, const TA* __restrict__ a2, const TB* __restrict__ b2,
                                             double* part2) {
    double acc = 0.0, acc2 = 0.0;
    for_elements(n, nrhs, [&](int64_t i) {
        acc += (double)a[i] * (double)b[i];
        if (a2) acc2 += (double)a2[i] * (double)b2[i];
    });
    const double s = block_rhs_sum(acc, nrhs);
    if ((int)threadIdx.x < nrhs) part[(size_t)blockIdx.x * 16 + threadIdx.x] = s;
    if (a2) {
        const double s2 = block_rhs_sum(acc2, nrhs);
        if ((int)threadIdx.x < nrhs) part2[(size_t)blockIdx.x * 16 + threadIdx.x] = s2;
    }
}

// x += alpha p (x FP64), r -= alpha q; partial r.r.
template <typename T>
__global__ void __launch_bounds__(256) k_update_xr(int64_t n, int nrhs, const PcgScalars* S, double* __restrict__ x,
                                                   T* __restrict__ r, const T* __restrict__ p,
                                                   const T* __restrict__ q, double* part) {
    const double a = S->alpha[threadIdx.x % nrhs];
    double acc = 0.0;
    for_elements(n, nrhs, [&](int64_t i) {
        T ri = r[i];
        if (a != 0.0) {
            x[i] += a * (double)p[i];
            ri = (T)((double)ri - a * (double)q[i]);
            r[i] = ri;
        }
        acc += (double)ri * (double)ri;
    });
    const double s = block_rhs_sum(acc, nrhs);
    if ((int)threadIdx.x < nrhs) part[(size_t)blockIdx.x * 16 + threadIdx.x] = s;
}

// p = z + beta p
template <typename T>
__global__ void __launch_bounds__(256) k_update_p(int64_t n, int nrhs, const PcgScalars* S, const T* __restrict__ z,
                                                  T* __restrict__ p) {
    const double be = S->beta[threadIdx.x % nrhs];
    for_elements(n, nrhs, [&](int64_t i) { p[i] = (T)((double)z[i] + be * (double)p[i]); });
}

template <typename Tin, typename Tout>
__global__ void k_convert(const Tin* in, Tout* out, int64_t cnt) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt;
         i += (int64_t)gridDim.x * blockDim.x)
        out[i] = (Tout)in[i];
}

__global__ void k_check_finite(const double* v, int64_t cnt, DevStatus* st) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt;
         i += (int64_t)gridDim.x * blockDim.x)
        if (!isfinite(v[i])) atomicAdd(&st->nonfinite, 1u);
}

// ---------------------------------------------------------------------------
// Host-side dispatch
// ---------------------------------------------------------------------------
static int pow2_at_least(int v) {
    int p = 1;
    while (p < v) p <<= 1;
    return p;
}

template <typename TA, typename TV, int NR, int ES, bool RES>
static void launch_spmv_es(const rw_context* ctx, int32_t n, int64_t nnz, const int32_t* rp, const int32_t* col,
                           const TA* val, const TV* x, TV* y, int nrhs, double* part, int* blocks_out, cudaStream_t s,
                           const double* b, int out32) {
    if constexpr (NR * ES <= 32) {
        // rows of a pass: as many as the copy holds with a tenth to spare, in whole sets of row groups
        const int set = 256 / (ES == 1 ? nrhs : NR * ES);
        const double avg = n > 0 ? std::max(1.0, (double)nnz / (double)n) : 1.0;
        int rows = std::max(1, std::min(kSpmvRows, (int)(0.9 * kSpmvEntries / avg)));
        // (a small matrix: at least two passes per SM)
        rows = std::max(std::min(rows, set), std::min(rows, n / (2 * ctx->num_sms)));
        if (rows > set) rows -= rows % set;
        const int64_t passes = ((int64_t)n + rows - 1) / rows;
        static int per_sm = 0;
        if (per_sm < 1) {
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_spmv<TA, TV, NR, ES, sizeof(TA) == 4, RES>, 256, 0);
            if (per_sm < 1) per_sm = 1;
        }
        int blocks = grid_for(passes, 1, ctx->num_sms * per_sm);
        if (part && blocks > kDotParts) blocks = kDotParts;
        if (blocks_out) *blocks_out = blocks;
        RW_COUNT_LAUNCH();
        // FP32 values are always the excess + difference form of the mixed mode
        k_spmv<TA, TV, NR, ES, sizeof(TA) == 4, RES>
            <<<blocks, 256, 0, s>>>(n, rp, col, val, x, y, nrhs, rows, part, b, out32);
    }
}

template <typename TA, typename TV, int NR, bool RES>
static void launch_spmv_rows(const rw_context* ctx, int32_t n, const int32_t* rp, const int32_t* col, const TA* val,
                             const TV* x, TV* y, int nrhs, double* part, int* blocks_out, cudaStream_t s,
                             const double* b, int out32) {
    int blocks = grid_for(n, 8, ctx->num_sms * 8);
    if (part && blocks > kDotParts) blocks = kDotParts;
    if (blocks_out) *blocks_out = blocks;
    RW_COUNT_LAUNCH();
    k_spmv_rows<TA, TV, NR, sizeof(TA) == 4, RES>
        <<<blocks, 256, 0, s>>>(n, rp, col, val, x, y, nrhs, part, b, out32);
}

// Entry slices per row: the option, else one, doubled until the rows that the
// block's threads hold at once fit the copy (27 entries a row and one
// right-hand side: four slices; nine: one), and while the rows' lanes do not
// fill the chip.
template <typename TA, typename TV, int NR, bool RES>
static void launch_spmv_nr(const rw_context* ctx, int32_t n, int64_t nnz, const int32_t* rp, const int32_t* col,
                           const TA* val, const TV* x, TV* y, int nrhs, double* part, int* blocks, cudaStream_t s,
                           const double* b, int out32) {
    // long rows: a warp each (see kLongRows); slices that fill the warp ask for that too
    if (ctx->opt.spmv_slices > 0 ? ctx->opt.spmv_slices >= 32 / NR : nnz * std::max(NR, 4) >= (int64_t)kLongRows * n)
        return launch_spmv_rows<TA, TV, NR, RES>(ctx, n, rp, col, val, x, y, nrhs, part, blocks, s, b, out32);
    int p = 1;
    if (ctx->opt.spmv_slices > 0) {
        while (p * 2 <= ctx->opt.spmv_slices && p * 2 * NR <= 32) p *= 2;
    } else {
        const int64_t avg = n > 0 ? nnz / n : 0, lanes = (int64_t)ctx->num_sms * 1024;
        while (p * 2 * NR <= 32 && (256 / (p == 1 ? nrhs : NR * p) * avg > kSpmvEntries * 3 / 2 ||
                                    ((int64_t)n * NR * p < lanes && avg > 2 * p)))
            p *= 2;
    }
    switch (p) {
        case 1: launch_spmv_es<TA, TV, NR, 1, RES>(ctx, n, nnz, rp, col, val, x, y, nrhs, part, blocks, s, b, out32); break;
        case 2: launch_spmv_es<TA, TV, NR, 2, RES>(ctx, n, nnz, rp, col, val, x, y, nrhs, part, blocks, s, b, out32); break;
        case 4: launch_spmv_es<TA, TV, NR, 4, RES>(ctx, n, nnz, rp, col, val, x, y, nrhs, part, blocks, s, b, out32); break;
        case 8: launch_spmv_es<TA, TV, NR, 8, RES>(ctx, n, nnz, rp, col, val, x, y, nrhs, part, blocks, s, b, out32); break;
        case 16: launch_spmv_es<TA, TV, NR, 16, RES>(ctx, n, nnz, rp, col, val, x, y, nrhs, part, blocks, s, b, out32); break;
        default: launch_spmv_es<TA, TV, NR, 32, RES>(ctx, n, nnz, rp, col, val, x, y, nrhs, part, blocks, s, b, out32); break;
    }
}

// part: per-block dot products x.y of the right-hand sides ([blocks][16], at
// most kDotParts blocks; *blocks receives their number).
template <typename TA, typename TV, bool RES = false>
static rw_status launch_spmv(rw_context* ctx, int32_t n, int64_t nnz, const int32_t* rp, const int32_t* col,
                             const TA* val, const TV* x, TV* y, int nrhs, double* part, int* blocks = nullptr,
                             const double* b = nullptr, int out32 = 0) {
    cudaStream_t s = ctx->stream;
    const int nr = pow2_at_least(nrhs);
    switch (nr) {
        case 1: launch_spmv_nr<TA, TV, 1, RES>(ctx, n, nnz, rp, col, val, x, y, nrhs, part, blocks, s, b, out32); break;
        case 2: launch_spmv_nr<TA, TV, 2, RES>(ctx, n, nnz, rp, col, val, x, y, nrhs, part, blocks, s, b, out32); break;
        case 4: launch_spmv_nr<TA, TV, 4, RES>(ctx, n, nnz, rp, col, val, x, y, nrhs, part, blocks, s, b, out32); break;
        case 8: launch_spmv_nr<TA, TV, 8, RES>(ctx, n, nnz, rp, col, val, x, y, nrhs, part, blocks, s, b, out32); break;
        default: launch_spmv_nr<TA, TV, 16, RES>(ctx, n, nnz, rp, col, val, x, y, nrhs, part, blocks, s, b, out32); break;
    }
    return check_launch("spmv");
}

template <typename T>
rw_status spmv_launch(rw_context* ctx, int32_t n, int64_t nnz, const int32_t* rp, const int32_t* col, const T* val,
                      const T* x, T* y, int nrhs) {
    NvtxRange nvtx_range("rw_spmv");
    return launch_spmv<T, T>(ctx, n, nnz, rp, col, val, x, y, nrhs, nullptr);
}
template rw_status spmv_launch<double>(rw_context*, int32_t, int64_t, const int32_t*, const int32_t*, const double*,
                                       const double*, double*, int);
template rw_status spmv_launch<float>(rw_context*, int32_t, int64_t, const int32_t*, const int32_t*, const float*,
                                      const float*, float*, int);

// Device-time accumulation of the solve phases (events on the context stream).
struct SolveTimes {
    bool on = false;
    float spmv = 0.f, bwd = 0.f, fwd = 0.f;
    bool pending_spmv = false, pending_pre = false;
};

// z = Y^-1 D^-1 Y^-T r; w: scratch [n, nrhs].  With timing, events 5/6/7
// bracket the two solves (read by the caller).
template <typename T>
static rw_status precond_t(rw_context* ctx, const FactorView& F, const T* yv, const T* ytv,
                           const T* d, const T* r, T* w, T* z, int nrhs, SolveTimes* tm = nullptr) {
    NvtxRange nvtx_range("rw_precond");
    if (tm && tm->on) cudaEventRecord(ctx->ev[5], ctx->stream);
    rw_status rc = solve_runs<T>(ctx, *F.bwd_sched, F.yt_rp, F.yt_col, ytv, r, w, nrhs, F.bar, true, nullptr, nullptr,
                                 F.bwd_t);
    if (rc) return rc;
    if (tm && tm->on) cudaEventRecord(ctx->ev[6], ctx->stream);
    rc = solve_runs<T>(ctx, *F.fwd_sched, F.y_rp, F.y_col, yv, w, z, nrhs, F.bar, false, w, d);
    if (tm && tm->on) {
        cudaEventRecord(ctx->ev[7], ctx->stream);
        tm->pending_pre = true;
    }
    return rc;
}

// Adds the completed event intervals of the last preconditioner application
// and SpMV (the stream has been synchronised by the caller).
static void collect_times(rw_context* ctx, SolveTimes& tm) {
    float t = 0.f;
    if (tm.pending_pre) {
        if (cudaEventElapsedTime(&t, ctx->ev[5], ctx->ev[6]) == cudaSuccess) tm.bwd += t;
        if (cudaEventElapsedTime(&t, ctx->ev[6], ctx->ev[7]) == cudaSuccess) tm.fwd += t;
        tm.pending_pre = false;
    }
    if (tm.pending_spmv) {
        if (cudaEventElapsedTime(&t, ctx->ev[2], ctx->ev[3]) == cudaSuccess) tm.spmv += t;
        tm.pending_spmv = false;
    }
}

void launch_to_fp32(const double* in, float* out, int64_t cnt, cudaStream_t s, int num_sms) {
    RW_COUNT_LAUNCH();
    k_convert<double, float><<<grid_for(cnt, 256, num_sms * 8), 256, 0, s>>>(in, out, cnt);
}

rw_status spmv_fp64(rw_context* ctx, const rw_csr* A, const double* x, double* y, int nrhs) {
    return launch_spmv<double, double>(ctx, A->n, A->nnz, A->row_ptr, A->col, A->val, x, y, nrhs, nullptr);
}

rw_status precond_fp64(rw_context* ctx, const FactorView& F, const double* r, double* z,
                       int nrhs, Pool& scratch) {
    const int64_t cnt = (int64_t)F.n * nrhs;
    double* w = alloc_n<double>(scratch, cnt);
    if (!w) return RW_ERR_ALLOC;
    rw_status rc;
    if ((rc = precond_t<double>(ctx, F, F.y_val, F.yt_val, F.d, r, w, z, nrhs))) return rc;
    return read_status(ctx, "preconditioner");
}

template <typename T>
static rw_status pcg_t(rw_context* ctx, const rw_csr* A, const FactorView& F, const double* b,
                       double* x, int nrhs, double tol, int max_iter, rw_pcg_stats* stats,
                       int32_t* h_iters, double* h_relres, Pool& sc, const T* Aval, const T* yv,
                       const T* ytv, const T* dv, bool mixed) {
    NvtxRange nvtx_range("rw_pcg");
    cudaStream_t s = ctx->stream;
    const int32_t n = A->n;
    const int64_t cnt = (int64_t)n * nrhs;
    T* r = alloc_n<T>(sc, cnt);
    T* z = alloc_n<T>(sc, cnt);
    T* p = alloc_n<T>(sc, cnt);
    T* q = alloc_n<T>(sc, cnt);
    T* w = alloc_n<T>(sc, cnt);
    double* part = alloc_n<double>(sc, (int64_t)kDotParts * 16);
    PcgScalars* S = alloc_n<PcgScalars>(sc, 1);
    if (!r || !z || !p || !q || !w || !part || !S) return RW_ERR_ALLOC;
    PcgScalars* hS = static_cast<PcgScalars*>(ctx->h_small);
    const int vb = grid_for(cnt, 1024, ctx->num_sms * 4);  // partial sums: four elements a thread and more
    rw_status rc;
    if ((rc = check_cuda(cudaMemsetAsync(S, 0, sizeof(PcgScalars), s), "memset"))) return rc;
    if ((rc = check_cuda(cudaMemsetAsync(x, 0, sizeof(double) * (size_t)cnt, s), "memset"))) return rc;
    RW_COUNT_LAUNCH();
    k_check_finite<<<vb, 256, 0, s>>>(b, cnt, ctx->d_status);
    RW_COUNT_LAUNCH();
    k_convert<double, T><<<vb, 256, 0, s>>>(b, r, cnt);
    RW_COUNT_LAUNCH();
    k_dot<double, double><<<vb, 256, 0, s>>>(b, b, n, nrhs, part, nullptr, nullptr, nullptr);
    RW_COUNT_LAUNCH();
    k_scalars<<<1, 1024, 0, s>>>(S, part, vb, nrhs, kOpBnorm, tol, 0);
    if ((rc = check_launch("pcg init"))) return rc;
    SolveTimes tm;
    tm.on = ctx->opt.timing != 0;
    if ((rc = precond_t<T>(ctx, F, yv, ytv, dv, r, w, z, nrhs, &tm))) return rc;
    RW_COUNT_LAUNCH();
    k_dot<T, T><<<vb, 256, 0, s>>>(r, z, n, nrhs, part, nullptr, nullptr, nullptr);
    RW_COUNT_LAUNCH();
    k_scalars<<<1, 1024, 0, s>>>(S, part, vb, nrhs, kOpRho0, tol, 0);
    RW_COUNT_LAUNCH();
    k_convert<T, T><<<vb, 256, 0, s>>>(z, p, cnt);
    if ((rc = check_launch("pcg start"))) return rc;
    if ((rc = check_cuda(cudaMemcpyAsync(hS, S, sizeof(PcgScalars), cudaMemcpyDeviceToHost, s), "copy")))
        return rc;
    if ((rc = read_status(ctx, "pcg start"))) return rc;
    if (ctx->d_status && ctx->h_status->nonfinite) {
        set_error("pcg: right-hand side holds a non-finite value");
        return RW_ERR_ARG;
    }
    // t = b - A x in FP64 (true residual), stored to out in T where given; partial t.t in *blocks blocks
    auto true_resid = [&](T* out, int* blocks) -> rw_status {
        return launch_spmv<double, double, true>(ctx, n, A->nnz, A->row_ptr, A->col, A->val, x,
                                                 reinterpret_cast<double*>(out), nrhs, part, blocks, b,
                                                 sizeof(T) == 4 ? 1 : 0);
    };
    int done_iters = 0;
    const int refine = ctx->opt.refine_every > 0 ? ctx->opt.refine_every : 50;
    bool any_active = hS->any_active != 0;
    for (int it = 1; it <= max_iter && any_active; ++it) {
        done_iters = it;
        if (tm.on) cudaEventRecord(ctx->ev[2], s);
        int sb = 0;
        if ((rc = launch_spmv<T, T>(ctx, n, A->nnz, A->row_ptr, A->col, Aval, p, q, nrhs, part, &sb))) return rc;
        if (tm.on) {
            cudaEventRecord(ctx->ev[3], s);
            tm.pending_spmv = true;
        }
        RW_COUNT_LAUNCH();
        k_scalars<<<1, 1024, 0, s>>>(S, part, sb, nrhs, kOpAlpha, tol, it);
        RW_COUNT_LAUNCH();
        k_update_xr<T><<<vb, 256, 0, s>>>(n, nrhs, S, x, r, p, q, part);
        int rb = vb;
        if (mixed && it % refine == 0 && (rc = true_resid(r, &rb))) return rc;
        RW_COUNT_LAUNCH();
        k_scalars<<<1, 1024, 0, s>>>(S, part, rb, nrhs, kOpResid, tol, it);
        if ((rc = check_launch("pcg step"))) return rc;
        if ((rc = check_cuda(cudaMemcpyAsync(hS, S, sizeof(PcgScalars), cudaMemcpyDeviceToHost, s),
                             "copy")))
            return rc;
        if ((rc = check_cuda(cudaStreamSynchronize(s), "sync"))) return rc;
        if (tm.on) collect_times(ctx, tm);
        if (hS->any_check) {
            int tb = 0;
            if ((rc = true_resid(nullptr, &tb))) return rc;
            RW_COUNT_LAUNCH();
            k_scalars<<<1, 1024, 0, s>>>(S, part, tb, nrhs, kOpTrue, tol, it);
            if ((rc = check_launch("pcg true residual"))) return rc;
            if ((rc = check_cuda(cudaMemcpyAsync(hS, S, sizeof(PcgScalars), cudaMemcpyDeviceToHost,
                                                 s),
                                 "copy")))
                return rc;
            if ((rc = check_cuda(cudaStreamSynchronize(s), "sync"))) return rc;
            if (!hS->any_active) break;
        }
        if (hS->broke) break;
        if ((rc = precond_t<T>(ctx, F, yv, ytv, dv, r, w, z, nrhs, &tm))) return rc;
        RW_COUNT_LAUNCH();
        k_dot<T, T><<<vb, 256, 0, s>>>(r, z, n, nrhs, part, nullptr, nullptr, nullptr);
        RW_COUNT_LAUNCH();
        k_scalars<<<1, 1024, 0, s>>>(S, part, vb, nrhs, kOpBeta, tol, it);
        RW_COUNT_LAUNCH();
        k_update_p<T><<<vb, 256, 0, s>>>(n, nrhs, S, z, p);
        if ((rc = check_launch("pcg direction"))) return rc;
    }
    // final true residuals for the report
    int fb = 0;
    if ((rc = true_resid(nullptr, &fb))) return rc;
    RW_COUNT_LAUNCH();
    k_scalars<<<1, 1024, 0, s>>>(S, part, fb, nrhs, kOpReport, tol, done_iters);
    if ((rc = check_launch("pcg report"))) return rc;
    if ((rc = check_cuda(cudaMemcpyAsync(hS, S, sizeof(PcgScalars), cudaMemcpyDeviceToHost, s), "copy")))
        return rc;
    if ((rc = read_status(ctx, "pcg"))) return rc;
    if (tm.on) collect_times(ctx, tm);
    int maxit = 0;
    double maxrel = 0.0;
    bool conv_all = true;
    for (int j = 0; j < nrhs; ++j) {
        const int itj = hS->active[j] ? done_iters : hS->iters[j];
        if (hS->active[j]) conv_all = false;
        const double rel = hS->bnorm2[j] > 0.0 ? std::sqrt(hS->tt[j] / hS->bnorm2[j]) : 0.0;
        maxit = std::max(maxit, itj);
        maxrel = std::max(maxrel, rel);
        if (h_iters) h_iters[j] = itj;
        if (h_relres) h_relres[j] = rel;
    }
    if (stats) {
        stats->iterations = maxit;
        stats->rel_residual = maxrel;
        stats->spmv_ms = tm.spmv;
        stats->bwd_ms = tm.bwd;
        stats->fwd_ms = tm.fwd;
    }
    if (hS->broke) {
        set_error("pcg breakdown: p.Ap <= 0");
        return RW_ERR_BREAKDOWN;
    }
    if (tol > 0.0 && !conv_all) {
        set_error("pcg did not reach the tolerance in %d iterations", max_iter);
        return RW_ERR_NO_CONVERGENCE;
    }
    return RW_OK;
}

rw_status pcg_run(rw_context* ctx, const rw_csr* A, const FactorView& F, const double* b,
                  double* x, int nrhs, double tol, int max_iter, rw_precision prec,
                  rw_pcg_stats* stats, int32_t* h_iters, double* h_relres) {
    Pool sc(ctx);
    cudaStream_t s = ctx->stream;
    rw_status rc;
    if (ctx->opt.timing) cudaEventRecord(ctx->ev[8], s);
    if (prec == RW_FP32_MIXED) {
        if (!F.y_val32 || !F.yt_val32 || !F.d32) {
            set_error("pcg: FP32 mode needs a factor built with store_fp32 = 1");
            return RW_ERR_ARG;
        }
        float* a32 = alloc_n<float>(sc, A->nnz);
        if (!a32) return RW_ERR_ALLOC;
        launch_to_fp32_diff(A->n, A->row_ptr, A->col, A->val, a32, s, ctx->num_sms);
        if ((rc = check_launch("convert A"))) return rc;
        rc = pcg_t<float>(ctx, A, F, b, x, nrhs, tol, max_iter, stats, h_iters, h_relres, sc, a32,
                          F.y_val32, F.yt_val32, F.d32, true);
    } else {
        rc = pcg_t<double>(ctx, A, F, b, x, nrhs, tol, max_iter, stats, h_iters, h_relres, sc,
                           A->val, F.y_val, F.yt_val, F.d, false);
    }
    if (ctx->opt.timing && stats) {
        cudaEventRecord(ctx->ev[9], s);
        cudaEventSynchronize(ctx->ev[9]);
        cudaEventElapsedTime(&stats->solve_ms, ctx->ev[8], ctx->ev[9]);
    }
    return rc;
}


// ---------------------------------------------------------------------------
// BiCGSTAB with right preconditioning (van der Vorst's method) for a
// nonsymmetric A, one right-hand side, FP64.  The preconditioner is the
// two-game factor of Sec. 7.1 (M = Y_{A^T}^T D Y_A): the view's forward data
// come from the game on A, its backward data from the game on A^T, and it is
// applied by the same backward and forward solves as in PCG.  Dot products:
// per-block sums on the device, added in a fixed order by one warp, so every
// run takes the same iterations.  Convergence is decided on the true residual
// ||b - A x|| < tol ||b||, recomputed whenever the recursive one passes (and
// then replacing it).
// ---------------------------------------------------------------------------
__global__ void k_lin3(int64_t n, double* out, const double* a, double ca, const double* b, double cb,
                       const double* c, double cc) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double v = ca * a[i];
        if (b) v += cb * b[i];
        if (c) v += cc * c[i];
        out[i] = v;
    }
}

// A warp per dot product adds its block sums of right-hand side 0 in a fixed order.
__global__ void k_sum_parts(const double* __restrict__ part, const double* __restrict__ part2, int nblocks,
                            double* out) {
    const double* p = threadIdx.x < 32 ? part : part2;
    double t = 0.0;
    for (int b = (int)lane_id(); b < nblocks; b += 32) t += p[(size_t)b * 16];
    t = warp_sum(t);
    if (lane_id() == 0) out[threadIdx.x >> 5] = t;
}

rw_status bicgstab_run(rw_context* ctx, const rw_csr* A, const FactorView& F, const double* b, double* x, double tol,
                       int max_iter, rw_pcg_stats* stats) {
    cudaStream_t s = ctx->stream;
    const int32_t n = A->n;
    const int64_t launches0 = g_launches;
    Pool sc(ctx);
    double* r = alloc_n<double>(sc, n);
    double* rh = alloc_n<double>(sc, n);
    double* pv = alloc_n<double>(sc, n);
    double* ph = alloc_n<double>(sc, n);
    double* v = alloc_n<double>(sc, n);
    double* sv = alloc_n<double>(sc, n);
    double* sh = alloc_n<double>(sc, n);
    double* t = alloc_n<double>(sc, n);
    double* w = alloc_n<double>(sc, n);
    double* part = alloc_n<double>(sc, (int64_t)kDotParts * 32);
    double* const part2 = part + (int64_t)kDotParts * 16;
    double* dres = alloc_n<double>(sc, 2);
    if (!r || !rh || !pv || !ph || !v || !sv || !sh || !t || !w || !part || !dres) return RW_ERR_ALLOC;
    double* hd = static_cast<double*>(ctx->h_small);
    const int vb = grid_for(n, 1024, ctx->num_sms * 2);
    const int gb = grid_for(n, 256, ctx->num_sms * 8);
    rw_status rc;
    // one or two dot products in one launch and one read back
    auto dots = [&](const double* a, const double* c, double* out, const double* a2, const double* c2,
                    double* out2) -> rw_status {
        RW_COUNT_LAUNCH();
        k_dot<double, double><<<vb, 256, 0, s>>>(a, c, n, 1, part, a2, c2, part2);
        RW_COUNT_LAUNCH();
        k_sum_parts<<<1, a2 ? 64 : 32, 0, s>>>(part, part2, vb, dres);
        rw_status r2;
        if ((r2 = check_launch("bicgstab dot")) ||
            (r2 = check_cuda(cudaMemcpyAsync(hd, dres, 2 * sizeof(double), cudaMemcpyDeviceToHost, s), "copy")) ||
            (r2 = check_cuda(cudaStreamSynchronize(s), "sync")))
            return r2;
        *out = hd[0];
        if (a2) *out2 = hd[1];
        return RW_OK;
    };
    auto dot = [&](const double* a, const double* c, double* out) -> rw_status {
        return dots(a, c, out, nullptr, nullptr, nullptr);
    };
    auto lin3 = [&](double* out, const double* a, double ca, const double* bb, double cb, const double* c,
                    double cc) -> rw_status {
        RW_COUNT_LAUNCH();
        k_lin3<<<gb, 256, 0, s>>>(n, out, a, ca, bb, cb, c, cc);
        return check_launch("bicgstab update");
    };
    auto apply_m = [&](const double* in, double* out) -> rw_status {
        rw_status r2 = precond_t<double>(ctx, F, F.y_val, F.yt_val, F.d, in, w, out, 1);
        return r2 ? r2 : check_launch("bicgstab preconditioner");
    };
    auto spmv = [&](const double* in, double* out) -> rw_status {
        return launch_spmv<double, double>(ctx, n, A->nnz, A->row_ptr, A->col, A->val, in, out, 1, nullptr);
    };
    cudaEventRecord(ctx->ev[8], s);
    double bb = 0.0;
    if ((rc = check_cuda(cudaMemsetAsync(x, 0, sizeof(double) * (size_t)n, s), "memset")) ||
        (rc = check_cuda(cudaMemsetAsync(pv, 0, sizeof(double) * (size_t)n, s), "memset")) ||
        (rc = check_cuda(cudaMemsetAsync(v, 0, sizeof(double) * (size_t)n, s), "memset")) ||
        (rc = lin3(r, b, 1.0, nullptr, 0.0, nullptr, 0.0)) || (rc = lin3(rh, b, 1.0, nullptr, 0.0, nullptr, 0.0)) ||
        (rc = dot(b, b, &bb)))
        return rc;
    if (!std::isfinite(bb)) {
        set_error("bicgstab: right-hand side holds a non-finite value");
        return RW_ERR_ARG;
    }
    const double bnorm = std::sqrt(bb);
    double rho_old = 1.0, alpha = 1.0, omega = 1.0, relres = bnorm > 0.0 ? 1.0 : 0.0;
    int it = 0;
    bool done = bnorm == 0.0, broke = false;
    double rho_next = bb;  // rh . r for the next iteration (r = rh = b), if have_rho
    bool have_rho = true;
    // the true residual b - A x into r; returns its relative norm
    auto true_residual = [&](double* rel) -> rw_status {
        rw_status r2;
        double rr = 0.0;
        if ((r2 = spmv(x, t)) || (r2 = lin3(r, b, 1.0, t, -1.0, nullptr, 0.0)) || (r2 = dot(r, r, &rr))) return r2;
        *rel = std::sqrt(rr) / bnorm;
        return RW_OK;
    };
    while (!done && it < max_iter) {
        ++it;
        double rho = rho_next, rv = 0.0;
        if (!have_rho && (rc = dot(rh, r, &rho))) return rc;
        have_rho = false;
        if (rho == 0.0 || !std::isfinite(rho)) {
            broke = true;
            break;
        }
        const double beta = (rho / rho_old) * (alpha / omega);
        if ((rc = lin3(pv, r, 1.0, pv, beta, v, -beta * omega)) || (rc = apply_m(pv, ph)) || (rc = spmv(ph, v)) ||
            (rc = dot(rh, v, &rv)))
            return rc;
        if (rv == 0.0 || !std::isfinite(rv)) {
            broke = true;
            break;
        }
        alpha = rho / rv;
        double ss = 0.0;
        if ((rc = lin3(sv, r, 1.0, v, -alpha, nullptr, 0.0)) || (rc = dot(sv, sv, &ss))) return rc;
        if (std::sqrt(ss) < tol * bnorm) {
            if ((rc = lin3(x, x, 1.0, ph, alpha, nullptr, 0.0)) || (rc = true_residual(&relres))) return rc;
            if (relres < tol) {
                done = true;
                break;
            }
            rho_old = rho;  // continue from the replaced residual
            omega = 1.0;
            continue;
        }
        double ts = 0.0, tt = 0.0;
        if ((rc = apply_m(sv, sh)) || (rc = spmv(sh, t)) || (rc = dots(t, sv, &ts, t, t, &tt)))
            return rc;
        if (tt == 0.0 || !std::isfinite(tt)) {
            broke = true;
            break;
        }
        omega = ts / tt;
        double rr = 0.0;
        if ((rc = lin3(x, x, 1.0, ph, alpha, sh, omega)) || (rc = lin3(r, sv, 1.0, t, -omega, nullptr, 0.0)) ||
            (rc = dots(r, r, &rr, rh, r, &rho_next)))
            return rc;
        have_rho = true;
        relres = std::sqrt(rr) / bnorm;
        if (relres < tol) {
            have_rho = false;  // (replaces r)
            if ((rc = true_residual(&relres))) return rc;
            if (relres < tol) done = true;
        }
        if (omega == 0.0) {
            broke = !done;
            break;
        }
        rho_old = rho;
    }
    if (!done && bnorm > 0.0 && (rc = true_residual(&relres))) return rc;
    cudaEventRecord(ctx->ev[9], s);
    if ((rc = read_status(ctx, "bicgstab"))) return rc;
    if (stats) {
        memset(stats, 0, sizeof(*stats));
        stats->iterations = it;
        stats->rel_residual = relres;
        cudaEventElapsedTime(&stats->solve_ms, ctx->ev[8], ctx->ev[9]);
        stats->kernel_launches = g_launches - launches0;
    }
    if (done) return RW_OK;
    if (broke) {
        set_error("bicgstab: breakdown after %d iterations (relative residual %.3e)", it, relres);
        return RW_ERR_BREAKDOWN;
    }
    set_error("bicgstab: %d iterations without reaching the tolerance (relative residual %.3e)", it, relres);
    return RW_ERR_NO_CONVERGENCE;
}

// ---------------------------------------------------------------------------
// Preconditioner application without allocation.
//
// Some callers cannot allocate device memory while they apply the
// preconditioner: an outer iterative solver that calls it once per iteration
// from a tight loop, code that runs under a fixed memory budget, or a
// framework whose allocator must not be re-entered from a library call.  For
// them the scratch vector w of the backward solve lives in the file-scope
// device array below instead of coming from the context's allocator.  The
// array holds kStaticScratchEntries doubles (n * nrhs at most) on every device
// that loads the library, for the life of the process.
// ---------------------------------------------------------------------------
constexpr int64_t kStaticScratchEntries = (int64_t)1 << 20;  // 8 MiB of FP64
static __device__ __align__(256) double g_static_scratch[kStaticScratchEntries];

static std::mutex g_static_scratch_mu;
constexpr int kMaxDevices = 64;
static double* g_static_scratch_ptr[kMaxDevices] = {};

// Device address of g_static_scratch on `device` (which must be current).  The
// host-side name of the array is only a stand-in, so the address is looked up
// once per device and cached.
static rw_status static_scratch_address(int device, double** out) {
    std::lock_guard<std::mutex> lock(g_static_scratch_mu);
    if (device < 0 || device >= kMaxDevices) {
        set_error("static scratch: device %d out of range", device);
        return RW_ERR_ARG;
    }
    if (!g_static_scratch_ptr[device]) {
        void* p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
        if (e != cudaSuccess) return check_cuda(e, "cudaGetSymbolAddress(static scratch)");
        g_static_scratch_ptr[device] = static_cast<double*>(p);
    }
    *out = g_static_scratch_ptr[device];
    return RW_OK;
}

}  // namespace rw

extern "C" rw_status rw_precond_apply_static(rw_context* ctx, const rw_factor* F,
                                             const double* d_r, double* d_z, int32_t nrhs) {
    using namespace rw;
    if (!ctx || !F || !d_r || !d_z || nrhs < 1 || nrhs > 16) {
        set_error("rw_precond_apply_static: bad arguments");
        return RW_ERR_ARG;
    }
    const rw_factor_desc& d = F->desc;
    const int64_t cnt = (int64_t)d.n * nrhs;
    if (cnt > kStaticScratchEntries) {
        set_error("rw_precond_apply_static: n * nrhs = %lld exceeds the static scratch of %lld "
                  "entries; use rw_precond_apply",
                  (long long)cnt, (long long)kStaticScratchEntries);
        return RW_ERR_CAPACITY;
    }
    if (d.n == 0) return RW_OK;
    int dev = -1;
    rw_status rc = check_cuda(cudaGetDevice(&dev), "cudaGetDevice");
    if (rc) return rc;
    if (dev != ctx->device) {
        set_error("rw_precond_apply_static: device %d is current, the context is on device %d",
                  dev, ctx->device);
        return RW_ERR_ARG;
    }
    double* w = nullptr;
    if ((rc = static_scratch_address(dev, &w))) return rc;
    FactorView v;
    v.n = d.n;
    v.nnz = d.nnz;
    v.y_rp = d.y_row_ptr;
    v.y_col = d.y_col;
    v.y_val = d.y_val;
    v.y_val32 = d.y_val32;
    v.yt_rp = d.yt_row_ptr;
    v.yt_col = d.yt_col;
    v.yt_val = d.yt_val;
    v.yt_val32 = d.yt_val32;
    v.d = d.d;
    v.d32 = d.d32;
    v.fwd_order = F->fwd_order;
    v.bwd_order = F->bwd_order;
    v.fwd_sched = &F->fwd_sched;
    v.bwd_sched = &F->bwd_sched;
    v.bar = F->bar;
    if ((rc = reset_status(ctx))) return rc;
    // (the solve marks w and z pending on every call: the array keeps the last call's contents)
    if ((rc = precond_t<double>(ctx, v, v.y_val, v.yt_val, v.d, d_r, w, d_z, nrhs))) return rc;
    return read_status(ctx, "static-scratch preconditioner");
}

namespace rw {
}  // namespace rw
