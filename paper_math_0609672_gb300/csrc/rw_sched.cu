// rw_sched.cu -- schedule and kernels of the triangular solves.
//
// The paper applies the factor by forward/backward substitution (Sec. 4);
// row r of a strict triangular system (CSR rp/col/val) gives
//   x_r = rhs_r - sum_p val_p * x_{col_p}
// (the D^-1 between the two solves is an element-wise pass).  Rows are visited
// in level order (level = 1 + the largest level of a dependency).  The DAGs of
// the walk factor are tall and thin: hundreds of levels hold a handful of rows
// each, where the time is the chain of dependent memory round trips (a value
// handed from one SM to another through L2, 0.33 us at least), not arithmetic.
//
// The default schedule (solve_mode 2) cuts the level order into stretches:
//   narrow stretch: consecutive levels of at most kNarrow rows, cut into blocks
//     of 256 consecutive positions.  The schedule holds the inverse of each
//     block's unit triangle L_BB, so that with t = rhs - (dependencies outside
//     the block) all rows of the block follow in one step, x_B = L_BB^-1 t: a
//     block costs two grid barriers instead of a hand-off per level (k_blocks);
//   wide stretch: row by row, every warp of a co-resident grid taking every W-th
//     row of the level order and waiting (bounded) for the values it reads
//     (k_rows).
// Y = I - N with N >= 0 for an R-matrix, so the blocks' inverses have no
// negative entries and are computed and applied without cancellation; they are
// computed in FP64 whatever the solve's precision.  An entry of an inverse is
// zero exactly where its row does not depend on its column, and zero entries
// are not multiplied: 0 x infinity or NaN would carry a non-finite value to rows
// that do not depend on it (of other matrices, in a batch).
// One application of the preconditioner, before (narrow levels one after the
// other in one thread block, the others sync-free with every lane polling its
// own values) and now: 32^2 grid, 709 levels each way, 1.65 -> 0.076 ms; 300^2
// grid in natural order, 48,350 levels, 109 -> 4.0 ms; 64^3 7-point, 1198
// levels, four right-hand sides 6.9 -> 2.4 ms, sixteen 28 -> 6.3 ms; 1000^2
// with long-range edges, 2229 levels, FP32 8.5 -> 4.6 ms.
//
// solve_mode 1 takes every row as in a wide stretch; solve_mode 0 solves the
// narrow stretches as blocks too and the other levels one after another over the
// whole grid (with the narrow levels one after another too, a 100^2 grid of 5,594
// levels takes 26.1 ms per application; with blocks 0.48 ms).  Every row sums its
// terms in a fixed order, so results do not depend on timing.
#include <algorithm>

#include "rw_internal.h"

namespace rw {

// Rows of a narrow level at most.  A block's step takes 5 to 7 us, a wide level
// 2 to 3 us, so the line lies where a block holds two to three levels: 32, 64,
// 128 and 256 gave 2.33, 1.95, 2.05 and 2.58 ms per application on the 64^3
// 7-point grid and 2.94, 2.41, 2.42 and 3.10 ms on a 56^3 27-point one.
constexpr int kNarrow = 96;
// Levels of a narrow stretch at least: shorter ones cost more in launches
// (about 10 us) than they save.
constexpr int kNarrowLevels = 16;
// Rows of a block.  With 512 the inversion takes twice as long (both directions
// of the 64^3 7-point grid: 2.3 against 1.2 ms of a 23 ms build).
constexpr int kBlockRows = 256;
// Thread blocks that solve a block's slots (see k_blocks); smaller devices take
// every row by itself.
constexpr int kMainBlocks = 64;

// Memory of the blocks of one direction, in bytes of inverses and workspace
// (a full block: 263 KB of FP64 inverse, 132 KB of FP32 copies and 42 KB of
// slots, 1.7 KB per row; beside it the schedule holds at most one more copy of
// the rows' entries).  A factor whose levels are all narrow would take several
// times its own size, so the blocks end at a sixteenth of the device's memory
// (10 million rows on 284 GB) and the rows after them are solved one by one.
// Beyond kBlockBytesSure they are also given up when their memory is not to be
// had: the factor then keeps the blocks of that many bytes only.
constexpr int64_t kBlockBytesSure = (int64_t)32 << 20;
constexpr int kBlockMemoryPart = 16;

// Rows of a wide level at least: with more rows than warps (16 on each of 152
// SMs) a level takes several rounds, and a round of packed rows four at a time
// (see k_rows_pack).  Below, a level is one round either way and a row is
// faster with 32 lanes.
constexpr int kWideRows = 2432;
constexpr int kWideLevels = 4;  // levels of a packed stretch at least (a launch of its own)
constexpr int kPackLanes = 8;
constexpr int kPackRows = 32 / kPackLanes;

__device__ __forceinline__ bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

__host__ __device__ __forceinline__ int64_t tri(int64_t m) { return m * (m + 1) / 2; }

// An entry of an inverse that is not the structural zero (integer tests: the
// FP64 pipe is what bounds these kernels).
__device__ __forceinline__ bool nonzero(double v) { return __double_as_longlong(v) != 0; }
__device__ __forceinline__ bool nonzero(float v) { return __float_as_uint(v) != 0u; }

// ---------------------------------------------------------------------------
// Schedule construction
// ---------------------------------------------------------------------------
__global__ void k_pos_of(int32_t n, const int32_t* __restrict__ order, int32_t* pos_of) {
    for (int32_t p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x)
        pos_of[order[p]] = p;
}

// The entries of a block slot's row, by where their column lies: in the block
// (0), in the block before it (1), earlier in the stretch (2), before it (3).
constexpr int kClasses = 4;
// Place of a class in the common numbering of the entries: the in-block ones,
// which only the inversion reads, come last.
__host__ __device__ __forceinline__ int class_place(int k) { return (k + kClasses - 1) % kClasses; }
__device__ __forceinline__ int entry_class(int64_t p, const SolveBlock& b) {
    return p >= b.pos0 ? 0 : p >= b.prev0 ? 1 : p >= b.stretch0 ? 2 : 3;
}

// Warp per slot: its row, and the entries of each class.
__global__ void __launch_bounds__(256) k_block_count(int64_t nslots, const SolveBlock* __restrict__ blocks,
                                                     const int32_t* __restrict__ order,
                                                     const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                                                     const int32_t* __restrict__ pos_of, uint32_t* cnt,
                                                     int32_t* trow) {
    const int lane = (int)lane_id();
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t t = gw; t < nslots; t += nw) {
        const SolveBlock b = blocks[t / kBlockRows];
        const int slot = (int)(t % kBlockRows);
        int row = -1;
        unsigned c[kClasses] = {};
        if (slot < b.rows) {
            row = order[b.pos0 + slot];
            const int64_t s = rp[row], e = rp[row + 1];
            for (int64_t q = s + lane; q < e; q += 32) {
                const int cl = entry_class(pos_of[col[q]], b);
#pragma unroll
                for (int k = 0; k < kClasses; ++k) c[k] += cl == k;
            }
#pragma unroll
            for (int k = 0; k < kClasses; ++k) c[k] = __reduce_add_sync(kFull, c[k]);
        }
        if (lane == 0) {
#pragma unroll
            for (int k = 0; k < kClasses; ++k) cnt[class_place(k) * nslots + t] = c[k];
            trow[t] = row;
        }
    }
}

// The entries of each class, in the row's order: slots and values inside the
// block (from `inside` of the common numbering on), columns, values and FP32
// copies of the others.
struct BlockEntries {
    const int64_t* ptr[kClasses];  // [nslots + 1] first entry of each slot
    int64_t inside;
    int32_t *slot, *col;
    double *yval, *val;
    float* val32;  // (NULL without FP32 copies)
};

__global__ void __launch_bounds__(256) k_block_split(int64_t nslots, const SolveBlock* __restrict__ blocks,
                                                     const int32_t* __restrict__ trow,
                                                     const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                                                     const double* __restrict__ val,
                                                     const float* __restrict__ val32,
                                                     const int32_t* __restrict__ pos_of, const BlockEntries E) {
    const int lane = (int)lane_id();
    const unsigned lt = lanemask_lt();
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t t = gw; t < nslots; t += nw) {
        const int32_t row = trow[t];
        if (row < 0) continue;
        const SolveBlock b = blocks[t / kBlockRows];
        const int64_t s = rp[row], e = rp[row + 1];
        int64_t o[kClasses];
#pragma unroll
        for (int k = 0; k < kClasses; ++k) o[k] = E.ptr[k][t];
        for (int64_t base = s; base < e; base += 32) {
            const int64_t q = base + lane;
            const int32_t c = q < e ? col[q] : 0;
            const int64_t p = q < e ? (int64_t)pos_of[c] : 0;
            const int cl = q < e ? entry_class(p, b) : -1;
#pragma unroll
            for (int k = 0; k < kClasses; ++k) {
                const unsigned m = __ballot_sync(kFull, cl == k);
                if (cl == k) {
                    const int64_t at = o[k] + __popc(m & lt);
                    if (k == 0) {
                        E.slot[at - E.inside] = (int32_t)(p - b.pos0);
                        E.yval[at - E.inside] = val[q];
                    } else {
                        E.col[at] = c;
                        E.val[at] = val[q];
                        if (E.val32) E.val32[at] = val32[q];
                    }
                }
                o[k] += __popc(m);
            }
        }
    }
}

// Inverse of each block's unit triangle L (L_ss = 1, L_su = the in-block
// entries), row s as s + 1 values from tri(s) on.  A warp takes
// eight columns: X_sc = [s == c] - sum_u L_su X_uc, row by row, the panel of X
// in shared memory, lane (q, j) summing entries q, q + 4, ... of column j.  The
// FP64 pipe's latency along the rows bounds it (an FP64 FMA waits 64 cycles), so
// the panels are narrow: many warps per SM, and the columns of a block are
// spread over many SMs.
// An entry to which some product contributes is stored as the least positive
// number when it underflows, so that zero means that no product does.
// One direction's blocks leave most SMs idle on small factors, so both
// directions share a launch (24 factors of random geometric
// graphs: 50 launches of 152 us, now 25 of 157 us).
constexpr int kPanel = 8;
struct InvertJob {
    int64_t nb;
    const SolveBlock* blocks;
    const int64_t* ptr;  // first entry of each slot, the in-block ones from `inside` on
    int64_t inside;
    const int32_t* slot;
    const double* val;
    double* inv;
    float* inv32;
};

__global__ void __launch_bounds__(32) k_block_invert(const InvertJob J0, const InvertJob J1, int64_t b0) {
    __shared__ double X[kBlockRows * kPanel];  // [rows - c0][kPanel]
    const int lane = (int)lane_id(), j = lane % kPanel, q = lane / kPanel;
    const InvertJob& J = blockIdx.z ? J1 : J0;
    const int64_t b = b0 + blockIdx.y;
    if (b >= J.nb) return;
    const int rows = J.blocks[b].rows, c0 = (int)blockIdx.x * kPanel;
    if (c0 >= rows) return;
    const int64_t* __restrict__ iptr = J.ptr;
    const int32_t* __restrict__ islot = J.slot;
    const double* __restrict__ ival = J.val;
    const int64_t inside = J.inside;
    double* const inv = J.inv;
    float* const inv32 = J.inv32;
    const int64_t t0 = b * kBlockRows, out0 = J.blocks[b].inv0;
    constexpr int U = 4;  // entries per lane read ahead
    int32_t sl[U];
    double y[U];
    int64_t e0, e1;
    auto fetch = [&](int r) {
        e0 = e1 = 0;
        if (r < rows) {
            e0 = iptr[t0 + r] - inside;
            e1 = iptr[t0 + r + 1] - inside;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t p = e0 + q + 4 * u;
            sl[u] = p < e1 ? islot[p] : -1;
            y[u] = p < e1 ? ival[p] : 0.0;
        }
    };
    fetch(c0);
    for (int r = c0; r < rows; ++r) {
        int32_t cs[U];
        double cy[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            cs[u] = sl[u];
            cy[u] = y[u];
        }
        const int64_t p0 = e0, p1 = e1;
        fetch(r + 1);  // in flight while this row is summed
        double acc = 0.0;
        int bits = 0;  // of the factors: zero when no product contributes (no branches: they cost more than the products)
        auto term = [&](int s, double yv) {
            const double xv = s >= c0 ? X[(s - c0) * kPanel + j] : 0.0;
            acc += yv * xv;
            bits |= __double2hiint(xv) | __double2loint(xv);
        };
#pragma unroll
        for (int u = 0; u < U; ++u) term(cs[u], cy[u]);
        for (int64_t p = p0 + q + 4 * U; p < p1; p += 4) term(islot[p], ival[p]);
        const unsigned hits = __ballot_sync(kFull, bits != 0);
        acc += __shfl_xor_sync(kFull, acc, 8);
        acc += __shfl_xor_sync(kFull, acc, 16);
        const int c = c0 + j;
        double v = (r == c ? 1.0 : 0.0) - (r >= c ? acc : 0.0);
        const bool hit = ((hits >> j) & 0x01010101u) != 0u;  // in any of the column's four lanes
        v = __hiloint2double(__double2hiint(v), __double2loint(v) | (hit && !nonzero(v) ? 1 : 0));
        if (q == 0) X[(r - c0) * kPanel + j] = v;
        __syncwarp();
        if (q == 0 && c <= r) {
            inv[out0 + tri(r) + c] = v;
            if (inv32) {
                const float f = (float)v;
                inv32[out0 + tri(r) + c] = nonzero(v) && !nonzero(f) ? __uint_as_float(1u) : f;
            }
        }
    }
}

// Thread per position: its row as the row solves take it, in the slot of its
// level (padding slots stay all ones: no row, no entries).
__global__ void k_fill_rows(int32_t n, int32_t depth, const int64_t* __restrict__ lptr,
                            const int64_t* __restrict__ slot0, const int32_t* __restrict__ order,
                            const int32_t* __restrict__ last, const int64_t* __restrict__ rp, SolveRow* rows) {
    for (int32_t p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
        int lo = 0, hi = depth - 1;  // the level of position p
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (lptr[mid] <= p) lo = mid;
            else hi = mid - 1;
        }
        const int32_t row = order[p];
        const int64_t s = rp[row];
        rows[slot0[lo] + (p - lptr[lo])] = SolveRow{s, (int32_t)(rp[row + 1] - s), row, last[row], 0};
    }
}

// A schedule under construction.  The host arrays live until their uploads are
// done (a GPU that shares the CPU's page tables may read them in place).
struct ScheduleWork {
    std::vector<SolveBlock> blocks;
    int64_t inverse = 0;         // entries of the blocks' inverses
    std::vector<int64_t> slot0;  // of each level in the rows array
    int32_t* pos_of = nullptr;
    int64_t* ptr = nullptr;
};

// Entries of the inverses of a stretch of `rows` rows, and the bytes that its
// blocks take (see kBlockBytesSure).
static int64_t inverse_entries(int64_t rows) {
    return rows / kBlockRows * tri(kBlockRows) + tri(rows % kBlockRows);
}
static int64_t block_bytes(int64_t rows, bool fp32) {
    const int64_t nb = (rows + kBlockRows - 1) / kBlockRows;
    return inverse_entries(rows) * (fp32 ? 12 : 8) +
           nb * (int64_t)(kBlockRows * (16 * sizeof(double) + kClasses * sizeof(int64_t) + sizeof(int32_t)) +
                          sizeof(SolveBlock));
}

// The stretches, rows and blocks (of `room` bytes at most; *used receives them)
// of one direction, and (on their way to totals[0..1]) the numbers of its
// blocks' entries outside and in all.
static rw_status schedule_plan(rw_context* ctx, const ScheduleInput& in, SolveSchedule& S, ScheduleWork& W,
                               int64_t* totals, int64_t room, int64_t* used, Pool& pool, Pool& scratch) {
    cudaStream_t s = ctx->stream;
    rw_status rc;
    // stretches: narrow ones as blocks, the others row by row, the widest levels packed
    std::vector<SolveBlock>& blocks = W.blocks;
    const int32_t n = S.n, depth = S.depth;
    std::vector<int64_t>& slot0 = W.slot0;
    slot0.resize((size_t)depth);
    int64_t slots = 0;
    bool full = ctx->num_sms <= kMainBlocks;  // no (further) blocks
    const bool fp32 = in.val32 != nullptr;
    auto kind_of = [&](int32_t l) {
        const int64_t w = S.lptr_h[l + 1] - S.lptr_h[l];
        return w <= kNarrow && !full ? 0 : w < kWideRows ? 1 : 2;
    };
    for (int32_t l = 0; l < depth;) {
        // the longest stretch of one kind; one too short for a launch of its own joins the row by row levels
        int kind = kind_of(l);
        int32_t e = l + 1;
        auto stretch_end = [&](int32_t f, int k) {
            while (f < depth && kind_of(f) == k) ++f;
            return f;
        };
        e = stretch_end(l, kind);
        if (kind == 0 && *used + block_bytes(S.lptr_h[e] - S.lptr_h[l], fp32) > room) {
            int32_t lo = l, hi = e;  // the last level that still has room, by bisection
            while (hi - lo > 1) {
                const int32_t mid = lo + (hi - lo) / 2;
                (*used + block_bytes(S.lptr_h[mid] - S.lptr_h[l], fp32) > room ? hi : lo) = mid;
            }
            full = true;
            if (lo - l < kNarrowLevels) continue;
            e = lo;
        }
        if ((kind == 0 && e - l < kNarrowLevels) || (kind == 2 && e - l < kWideLevels)) kind = 1;
        if (kind == 1) {  // up to the next long enough stretch of another kind
            while (e < depth) {
                const int k = kind_of(e);
                const int32_t f = stretch_end(e, k);
                if ((k == 0 && f - e >= kNarrowLevels) || (k == 2 && f - e >= kWideLevels)) break;
                e = f;
            }
        }
        if (kind == 2) slots = (slots + kPackRows - 1) / kPackRows * kPackRows;
        SolveStretch st{S.lptr_h[l], S.lptr_h[e], slots, 0, W.inverse, l, e, (int32_t)blocks.size(), 0,
                        kind == 2};
        for (int32_t i = l; i < e; ++i) {
            slot0[i] = slots;
            slots += S.lptr_h[i + 1] - S.lptr_h[i];
            if (kind == 2) slots = (slots + kPackRows - 1) / kPackRows * kPackRows;
        }
        st.slot1 = slots;
        if (kind == 0) {
            for (int64_t pos = st.pos0, prev = pos; pos < st.pos1;) {
                const int32_t r = (int32_t)std::min<int64_t>(kBlockRows, st.pos1 - pos);
                blocks.push_back(SolveBlock{pos, prev, st.pos0, W.inverse, r, 0});
                W.inverse += tri(r);
                prev = pos;
                pos += r;
            }
            st.nblocks = (int32_t)blocks.size() - st.block0;
            *used += block_bytes(st.pos1 - st.pos0, fp32);
        }
        S.stretches.push_back(st);
        l = e;
    }
    S.nrows = slots;
    const int g = grid_for(n, 256, ctx->num_sms * 8);
    S.rows = alloc_n<SolveRow>(pool, slots);
    int64_t* d_slot0 = alloc_n<int64_t>(scratch, depth);
    if (!S.rows || !d_slot0) return RW_ERR_ALLOC;
    if ((rc = check_cuda(cudaMemcpyAsync(d_slot0, slot0.data(), sizeof(int64_t) * (size_t)depth,
                                         cudaMemcpyHostToDevice, s),
                         "copy")) ||
        (slots > n &&
         (rc = check_cuda(cudaMemsetAsync(S.rows, 0xFF, sizeof(SolveRow) * (size_t)slots, s), "memset"))))
        return rc;
    RW_COUNT_LAUNCH();
    k_fill_rows<<<g, 256, 0, s>>>(n, depth, S.lptr, d_slot0, S.order, in.last, in.rp, S.rows);
    if ((rc = check_launch("schedule rows"))) return rc;
    const int64_t nb = (int64_t)blocks.size(), nslots = nb * kBlockRows;
    if (nb == 0) return RW_OK;
    int32_t* const pos_of = W.pos_of = alloc_n<int32_t>(scratch, n);
    uint32_t* cnt = alloc_n<uint32_t>(scratch, kClasses * nslots);
    int64_t* const ptr = W.ptr = alloc_n<int64_t>(pool, kClasses * nslots + 1);
    S.blocks = alloc_n<SolveBlock>(pool, nb);
    S.trow = alloc_n<int32_t>(pool, nslots);
    S.inv = alloc_n<double>(pool, W.inverse);
    S.inv32 = fp32 ? alloc_n<float>(pool, W.inverse) : nullptr;
    S.slots = nslots;
    S.t = pool.get((size_t)nslots * 16 * sizeof(double));
    if (!pos_of || !cnt || !ptr || !S.blocks || !S.trow || !S.inv || (fp32 && !S.inv32) || !S.t) return RW_ERR_ALLOC;
    if ((rc = check_cuda(cudaMemcpyAsync(S.blocks, blocks.data(), sizeof(SolveBlock) * (size_t)nb,
                                         cudaMemcpyHostToDevice, s),
                         "copy")))
        return rc;
    const int gw = grid_for(nslots * 32, 256, ctx->num_sms * 8);
    RW_COUNT_LAUNCH();
    k_pos_of<<<g, 256, 0, s>>>(n, S.order, pos_of);
    RW_COUNT_LAUNCH();
    k_block_count<<<gw, 256, 0, s>>>(nslots, S.blocks, S.order, in.rp, in.col, pos_of, cnt, S.trow);
    if ((rc = check_launch("schedule count"))) return rc;
    if ((rc = check_cuda(scan_u32_to_i64(cnt, ptr, kClasses * nslots, s, scratch), "scan")) ||
        (rc = check_cuda(cudaMemcpyAsync(totals, ptr + class_place(0) * nslots, 8, cudaMemcpyDeviceToHost, s),
                         "copy")))
        return rc;
    return check_cuda(cudaMemcpyAsync(totals + 1, ptr + kClasses * nslots, 8, cudaMemcpyDeviceToHost, s), "copy");
}

// The entries of the blocks by class; J: the inversion of their triangles.
static rw_status schedule_split(rw_context* ctx, const ScheduleInput& in, SolveSchedule& S, const ScheduleWork& W,
                                const int64_t* totals, InvertJob& J, Pool& pool, Pool& scratch) {
    cudaStream_t s = ctx->stream;
    const int64_t nb = (int64_t)W.blocks.size(), nslots = nb * kBlockRows;
    if (nb == 0) return RW_OK;
    const int gw = grid_for(nslots * 32, 256, ctx->num_sms * 8);
    BlockEntries E{};
    for (int k = 0; k < kClasses; ++k) E.ptr[k] = W.ptr + class_place(k) * nslots;
    E.inside = totals[0];
    E.slot = alloc_n<int32_t>(scratch, totals[1] - E.inside);
    E.yval = alloc_n<double>(scratch, totals[1] - E.inside);
    E.col = alloc_n<int32_t>(pool, E.inside);
    E.val = alloc_n<double>(pool, E.inside);
    E.val32 = in.val32 ? alloc_n<float>(pool, E.inside) : nullptr;
    if (!E.slot || !E.yval || !E.col || !E.val || (in.val32 && !E.val32)) return RW_ERR_ALLOC;
    for (int k = 0; k + 1 < kClasses; ++k) S.ext[k] = SolveEntries{E.ptr[k + 1], E.col, E.val, E.val32};
    RW_COUNT_LAUNCH();
    k_block_split<<<gw, 256, 0, s>>>(nslots, S.blocks, S.trow, in.rp, in.col, in.val, in.val32, W.pos_of, E);
    J = InvertJob{nb, S.blocks, E.ptr[0], E.inside, E.slot, E.yval, S.inv, S.inv32};
    return check_launch("schedule split");
}

// Both directions with blocks of `room` bytes each at most; *used: the larger
// of what they take.
static rw_status schedules_in(rw_context* ctx, const ScheduleInput* const in[2], SolveSchedule* const S[2],
                              int64_t room, int64_t* used, ScheduleWork (&W)[2], Pool& pool, Pool& scratch) {
    cudaStream_t s = ctx->stream;
    const int32_t n = S[0]->n;
    rw_status rc;
    InvertJob J[2]{};
    int64_t* totals = static_cast<int64_t*>(ctx->h_small);
    for (int k = 0; k < 2; ++k) {
        *S[k] = SolveSchedule{n, in[k]->depth, in[k]->order, in[k]->lptr, std::move(S[k]->lptr_h)};
        int64_t bytes = 0;
        rc = schedule_plan(ctx, *in[k], *S[k], W[k], totals + 2 * k, room, &bytes, pool, scratch);
        *used = std::max(*used, bytes);
        if (rc) return rc;
    }
    const int64_t nb = (int64_t)std::max(W[0].blocks.size(), W[1].blocks.size());
    if ((rc = check_cuda(cudaStreamSynchronize(s), "sync")) || nb == 0) return rc;
    const int64_t counts[4] = {totals[0], totals[1], totals[2], totals[3]};
    for (int k = 0; k < 2; ++k)
        if ((rc = schedule_split(ctx, *in[k], *S[k], W[k], counts + 2 * k, J[k], pool, scratch))) return rc;
    for (int64_t b0 = 0; b0 < nb; b0 += 65535) {
        const unsigned nbl = (unsigned)std::min<int64_t>(nb - b0, 65535);
        RW_COUNT_LAUNCH();
        k_block_invert<<<dim3(kBlockRows / kPanel, nbl, 2), 32, 0, s>>>(J[0], J[1], b0);
    }
    return check_launch("block inverses");
}

rw_status build_schedules(rw_context* ctx, int32_t n, const ScheduleInput& fwd, SolveSchedule& F,
                          const ScheduleInput& bwd, SolveSchedule& B, Pool& pool, Pool& scratch) {
    NvtxRange nvtx_range("rw_schedule");
    cudaStream_t s = ctx->stream;
    rw_status rc;
    const ScheduleInput* const in[2] = {&fwd, &bwd};
    SolveSchedule* const S[2] = {&F, &B};
    for (int k = 0; k < 2; ++k) {
        *S[k] = SolveSchedule{};
        S[k]->n = n;
        S[k]->depth = in[k]->depth;
        S[k]->order = in[k]->order;
        S[k]->lptr = in[k]->lptr;
    }
    if (n == 0) return RW_OK;
    for (int k = 0; k < 2; ++k) {
        S[k]->lptr_h.resize((size_t)S[k]->depth + 1);
        if ((rc = check_cuda(cudaMemcpyAsync(S[k]->lptr_h.data(), S[k]->lptr, sizeof(int64_t) * (S[k]->depth + 1),
                                             cudaMemcpyDeviceToHost, s),
                             "copy")))
            return rc;
    }
    if ((rc = check_cuda(cudaStreamSynchronize(s), "sync"))) return rc;
    for (int64_t room = std::max(kBlockBytesSure, (int64_t)(ctx->mem_bytes / kBlockMemoryPart));;
         room = kBlockBytesSure) {
        ScheduleWork W[2];
        Pool mine(ctx), work(ctx);
        int64_t used = 0;
        rc = schedules_in(ctx, in, S, room, &used, W, mine, work);
        if (rc == RW_OK) {
            pool.absorb(mine);
            scratch.absorb(work);
            return RW_OK;
        }
        cudaStreamSynchronize(s);  // nothing reads the host arrays any more
        if (rc != RW_ERR_ALLOC || used <= kBlockBytesSure) return rc;
        cudaGetLastError();  // (the failed allocation's)
    }
}

// ---------------------------------------------------------------------------
// Wide run: level-synchronous over the co-resident grid.
// ---------------------------------------------------------------------------
template <typename T>
struct WideParams {
    int32_t lev_begin, lev_end;
    const int64_t* __restrict__ lptr;
    const int32_t* __restrict__ order;
    const int64_t* __restrict__ rp;
    const int32_t* __restrict__ col;
    const T* __restrict__ val;
    const T* __restrict__ rhs;
    T* x;
    int nrhs;
    unsigned* bar;
    DevStatus* st;
};

// Wide and cluster runs: a group of G = NR * ES lanes per row, 32 / G rows
// per warp.  Lane (es, j) of a group owns right-hand side j and entries
// s + es, s + es + ES, ...: the NR values of x a row entry needs arrive in one
// contiguous load, and only the ES entry slices are summed across lanes.
//
// A level's own chain after the barrier is one round of x loads; the row
// structure it reads (position -> row -> row pointers -> first entries) does
// not depend on x and is loaded two levels ahead, so its dependent loads
// overlap the levels in between.
constexpr int kPreEntries = 4;  // entries per lane held ahead

template <typename T>
struct RowPre {
    int32_t row;  // -1: no row for this group in that level
    int64_t s, e;
    int32_t c[kPreEntries];
    T y[kPreEntries];
};

template <typename T, int NR, int ES>
struct RowGroup {
    static constexpr int G = NR * ES;
    static constexpr int R = 32 / G;
    int j, es;
    unsigned gmask;
    bool jok;
    __device__ RowGroup(int lane, int nrhs) {
        const int gl = lane % G;
        j = gl % NR;
        es = gl / NR;
        gmask = G == 32 ? kFull : (((1u << G) - 1u) << (lane - gl));
        jok = j < nrhs;
    }
    __device__ __forceinline__ void load(const WideParams<T>& P, int32_t row, RowPre<T>& R0) const {
        R0.row = row;
        R0.s = P.rp[row];
        R0.e = P.rp[row + 1];
#pragma unroll
        for (int u = 0; u < kPreEntries; ++u) {
            const int64_t q = R0.s + es + (int64_t)u * ES;
            R0.c[u] = q < R0.e ? P.col[q] : 0;
            R0.y[u] = q < R0.e ? P.val[q] : T(0);
        }
    }
    // x_row = rhs_row - sum_q val_q x_{col_q}
    __device__ __forceinline__ void row(const WideParams<T>& P, const RowPre<T>& R0) const {
        const T* __restrict__ x = P.x;
        const int nr = P.nrhs;
        T acc = T(0);
        T v[kPreEntries];
#pragma unroll
        for (int u = 0; u < kPreEntries; ++u)
            v[u] = (jok && R0.s + es + (int64_t)u * ES < R0.e) ? __ldcg(x + (size_t)R0.c[u] * nr + j) : T(0);
#pragma unroll
        for (int u = 0; u < kPreEntries; ++u) acc += R0.y[u] * v[u];
        int64_t q = R0.s + es + (int64_t)kPreEntries * ES;
        for (; q + 3 * ES < R0.e; q += 4 * ES) {
            int32_t c[4];
            T y[4], w[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                c[u] = P.col[q + u * ES];
                y[u] = P.val[q + u * ES];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) w[u] = jok ? __ldcg(x + (size_t)c[u] * nr + j) : T(0);
#pragma unroll
            for (int u = 0; u < 4; ++u) acc += y[u] * w[u];
        }
        for (; q < R0.e; q += ES) {
            const int32_t c = P.col[q];
            const T y = P.val[q];
            if (jok) acc += y * __ldcg(x + (size_t)c * nr + j);
        }
#pragma unroll
        for (int o = NR; o < G; o <<= 1) acc += __shfl_xor_sync(gmask, acc, o);
        if (es == 0 && jok) {
            __stcg(P.x + (size_t)R0.row * nr + j, P.rhs[(size_t)R0.row * nr + j] - acc);
        }
    }
};

// Vector rows (rw_options.wide_slices = -1): one warp per row; lane l owns
// entries s + l, s + l + 32, ... and reads all right-hand sides of each entry
// in one vector load, so each entry's column and value are loaded once (not
// once per right-hand side) and 4 entries per lane prefetched cover rows of
// up to 128 entries: a long row costs one round of x loads like a short one.
// The NR partial sums are reduced by the halving butterfly of warp_sums;
// lane j * 32 / NR ends with the sum of right-hand side j.
template <typename T, int NR>
struct RowVec {
    static constexpr int G = 32;
    static constexpr int R = 1;
    int lane;
    __device__ RowVec(int lane_, int) : lane(lane_) {}
    __device__ __forceinline__ void load(const WideParams<T>& P, int32_t row, RowPre<T>& R0) const {
        R0.row = row;
        R0.s = P.rp[row];
        R0.e = P.rp[row + 1];
#pragma unroll
        for (int u = 0; u < kPreEntries; ++u) {
            const int64_t q = R0.s + lane + (int64_t)u * 32;
            R0.c[u] = q < R0.e ? P.col[q] : 0;
            R0.y[u] = q < R0.e ? P.val[q] : T(0);
        }
    }
    // the nrhs values of x at node c (vector loads when nrhs == NR and x is aligned for them)
    __device__ __forceinline__ void xload(const WideParams<T>& P, int32_t c, T (&v)[NR]) const {
        const T* p = P.x + (size_t)c * P.nrhs;
        if constexpr (NR >= 2 && sizeof(T) == 8) {
            if (P.nrhs == NR && aligned16(P.x)) {
#pragma unroll
                for (int j = 0; j < NR; j += 2) {
                    const double2 d = __ldcg(reinterpret_cast<const double2*>(p + j));
                    v[j] = d.x;
                    v[j + 1] = d.y;
                }
                return;
            }
        } else if constexpr (NR >= 4 && sizeof(T) == 4) {
            if (P.nrhs == NR && aligned16(P.x)) {
#pragma unroll
                for (int j = 0; j < NR; j += 4) {
                    const float4 d = __ldcg(reinterpret_cast<const float4*>(p + j));
                    v[j] = d.x;
                    v[j + 1] = d.y;
                    v[j + 2] = d.z;
                    v[j + 3] = d.w;
                }
                return;
            }
        }
#pragma unroll
        for (int j = 0; j < NR; ++j) v[j] = j < P.nrhs ? __ldcg(p + j) : T(0);
    }
    __device__ __forceinline__ void row(const WideParams<T>& P, const RowPre<T>& R0) const {
        T acc[NR];
#pragma unroll
        for (int j = 0; j < NR; ++j) acc[j] = T(0);
        T v[kPreEntries][NR];
#pragma unroll
        for (int u = 0; u < kPreEntries; ++u) {
            if (R0.s + lane + (int64_t)u * 32 < R0.e) {
                xload(P, R0.c[u], v[u]);
            } else {
#pragma unroll
                for (int j = 0; j < NR; ++j) v[u][j] = T(0);
            }
        }
#pragma unroll
        for (int u = 0; u < kPreEntries; ++u)
#pragma unroll
            for (int j = 0; j < NR; ++j) acc[j] += R0.y[u] * v[u][j];
        for (int64_t q = R0.s + lane + (int64_t)kPreEntries * 32; q < R0.e; q += 4 * 32) {
            int32_t c[4];
            T y[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool ok = q + u * 32 < R0.e;
                c[u] = ok ? P.col[q + u * 32] : 0;
                y[u] = ok ? P.val[q + u * 32] : T(0);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                // padding slots past the row's end read nothing: x of column 0
                // may still be unset (0 * NaN would poison the sum)
                if (q + u * 32 < R0.e) {
                    T w[NR];
                    xload(P, c[u], w);
#pragma unroll
                    for (int j = 0; j < NR; ++j) acc[j] += y[u] * w[j];
                }
            }
        }
        const T sum = warp_sums_spread<T, NR>(acc);
        constexpr int span = 32 / NR;
        const int j = lane / span;
        if (lane % span == 0 && j < P.nrhs) {
            __stcg(P.x + (size_t)R0.row * P.nrhs + j, P.rhs[(size_t)R0.row * P.nrhs + j] - sum);
        }
    }
};

// The row type of a wide or cluster run: lane groups of NR * ES lanes, or
// vector rows when ES == 0.
template <typename T, int NR, int ES>
struct RowSel {
    using type = RowGroup<T, NR, ES>;
};
template <typename T, int NR>
struct RowSel<T, NR, 0> {
    using type = RowVec<T, NR>;
};
template <int NR, int ES>
constexpr int group_lanes() {
    return ES == 0 ? 32 : NR * ES;
}

// The levels of a run over `ngroups` row groups numbered from gid, with a
// barrier between levels.  Returns false if a barrier gave up.
template <typename T, typename Group, typename Barrier>
__device__ __forceinline__ bool run_levels(const WideParams<T>& P, int64_t gid, int64_t ngroups, const Group& g,
                                           Barrier barrier) {
    RowPre<T> pre[2];
    auto prefetch = [&](int32_t l, RowPre<T>& R0) {
        R0.row = -1;
        if (l < P.lev_end) {
            const int64_t pos = P.lptr[l] + gid;
            if (pos < P.lptr[l + 1]) g.load(P, P.order[pos], R0);
        }
    };
    prefetch(P.lev_begin, pre[0]);
    prefetch(P.lev_begin + 1, pre[1]);
    for (int32_t l = P.lev_begin; l < P.lev_end; ++l) {
        const RowPre<T> cur = pre[0];
        pre[0] = pre[1];
        prefetch(l + 2, pre[1]);  // in flight during this level and the next
        if (cur.row >= 0) {
            g.row(P, cur);
            const int64_t le = P.lptr[l + 1];
            for (int64_t pos = P.lptr[l] + gid + ngroups; pos < le; pos += ngroups) {
                RowPre<T> more;
                g.load(P, P.order[pos], more);
                g.row(P, more);
            }
        }
        if (l + 1 < P.lev_end && !barrier()) return false;
    }
    return true;
}

// Wide run: the whole co-resident grid, a software grid barrier between levels.
constexpr int kWideThreads = 512;  // one block per SM: fewer arrivals per grid barrier

template <typename T, int NR, int ES>
__global__ void __launch_bounds__(kWideThreads, 1) k_wide(const WideParams<T> P) {
    using Group = typename RowSel<T, NR, ES>::type;
    const Group g((int)lane_id(), P.nrhs);
    constexpr int R = Group::R;
    const int64_t gid = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * R + lane_id() / (32 / R);
    const int64_t ngroups = (((int64_t)gridDim.x * blockDim.x) >> 5) * R;
    unsigned epoch = 0;
    run_levels<T>(P, gid, ngroups, g, [&]() { return grid_barrier(P.bar, ++epoch, P.st); });
}

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cluster_size() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}

// Cluster run: one thread-block cluster (launched as the whole grid); the
// hardware cluster barrier with release / acquire semantics orders each
// level's x stores before the next level's loads (both through L2).  It waits
// only for the CTAs of the cluster, which the hardware schedules together.
template <typename T, int NR, int ES>
__global__ void __launch_bounds__(1024, 1) k_cluster(const WideParams<T> P) {
    using Group = typename RowSel<T, NR, ES>::type;
    const Group g((int)lane_id(), P.nrhs);
    constexpr int R = Group::R;
    const int64_t warps = blockDim.x >> 5;
    const int64_t gid = ((int64_t)cluster_rank() * warps + (threadIdx.x >> 5)) * R + lane_id() / (32 / R);
    const int64_t ngroups = (int64_t)cluster_size() * warps * R;
    run_levels<T>(P, gid, ngroups, g, []() {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        return true;
    });
}

// ---------------------------------------------------------------------------
// Rows of a wide stretch (all rows with solve_mode 1): one cooperative launch.
// x starts as the "pending" marker; warp w takes the rows at positions w,
// w + W, ... of the stretch; a row loads all its dependencies at once and
// publishes its value with one relaxed store.  Rows are taken in level order
// and all warps are co-resident, so the lowest unfinished position can always
// proceed.  A row that finds values pending waits (bounded) for the one on its
// highest level first and then loads the pending ones again: with every lane
// polling its own values the polls of the thousands of waiting warps filled the
// L2 (61x64x67 grid of 124 levels: 0.97 -> 0.54 ms per application).  Each warp
// loads the structure of its next two rows while it waits.
// ---------------------------------------------------------------------------
template <typename T>
struct RowParams {
    int64_t n;
    const SolveRow* __restrict__ rows;
    const int32_t* __restrict__ col;
    const T* __restrict__ val;
    const T* __restrict__ rhs;
    T* x;
    int nrhs;
    DevStatus* st;
};

template <typename T>
__device__ __forceinline__ SolveRow row_at(const RowParams<T>& P, int64_t i) {
    return i < P.n ? P.rows[i] : SolveRow{0, 0, -1, -1, 0};
}

// Column and value of entry q of a row.
template <typename T>
__device__ __forceinline__ void row_entry(const RowParams<T>& P, const SolveRow& d, int q, int32_t& c, T& y) {
    const bool ok = q < d.cnt;
    c = ok ? P.col[d.start + q] : 0;
    y = ok ? P.val[d.start + q] : T(0);
}

// Lane groups: lane (es, j) owns right-hand side j and entries es, es + ES, ...
template <typename T, int NR>
__global__ void __launch_bounds__(512, sizeof(T) == 4 ? 2 : 1) k_rows(const RowParams<T> P) {
    constexpr int ES = 32 / NR;
    constexpr int U = kPreEntries;
    const int lane = (int)lane_id();
    const int j = lane % NR, es = lane / NR;
    const bool jok = j < P.nrhs;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const unsigned spin_limit = P.st->spin_limit;
    // polls back off after the first few so that waiting warps leave L2
    // bandwidth to the rows being computed
    auto wait_value = [&](const T* src, T v) -> T {
        unsigned spins = 0;
        while (is_pending(v)) {
            if (wait_gives_up(spins, spin_limit, &P.st->timeout)) return T(0);
            if (spins > 4) __nanosleep(64);
            v = ld_relaxed(src);
        }
        return v;
    };
    struct Pre {
        SolveRow d;
        int32_t c[U];
        T y[U];
        T b;
    };
    auto load = [&](const SolveRow& d, Pre& R) {
        R.d = d;
#pragma unroll
        for (int u = 0; u < U; ++u) row_entry(P, d, es + u * ES, R.c[u], R.y[u]);
        R.b = es == 0 && jok && d.row >= 0 ? P.rhs[(size_t)d.row * P.nrhs + j] : T(0);
    };
    Pre pre[2];
    load(row_at(P, gw), pre[0]);
    load(row_at(P, gw + nw), pre[1]);
    SolveRow after = row_at(P, gw + 2 * nw);
    for (int64_t pos = gw; pos < P.n; pos += nw) {
        const Pre cur = pre[0];
        pre[0] = pre[1];
        load(after, pre[1]);
        after = row_at(P, pos + 3 * nw);
        const int nr = P.nrhs, cnt = cur.d.cnt;
        const T* const src = P.x;
        T v[U];
        bool pend = false;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            v[u] = (jok && es + u * ES < cnt) ? ld_relaxed(src + (size_t)cur.c[u] * nr + j) : T(0);
            pend |= is_pending(v[u]);
        }
        if (cur.d.last >= 0 && __any_sync(kFull, pend)) {
            const T* const p = src + (size_t)cur.d.last * nr + (jok ? j : 0);
            wait_value(p, ld_relaxed(p));
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (is_pending(v[u])) v[u] = ld_relaxed(src + (size_t)cur.c[u] * nr + j);
        }
        T acc = T(0);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (jok && es + u * ES < cnt) v[u] = wait_value(src + (size_t)cur.c[u] * nr + j, v[u]);
            acc += cur.y[u] * v[u];
        }
        for (int base = U * ES; base < cnt; base += U * ES) {
            int32_t c[U];
            T y[U], w[U];
#pragma unroll
            for (int u = 0; u < U; ++u) row_entry(P, cur.d, base + es + u * ES, c[u], y[u]);
#pragma unroll
            for (int u = 0; u < U; ++u)
                w[u] = (jok && base + es + u * ES < cnt) ? ld_relaxed(src + (size_t)c[u] * nr + j) : T(0);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (jok && base + es + u * ES < cnt) w[u] = wait_value(src + (size_t)c[u] * nr + j, w[u]);
                acc += y[u] * w[u];
            }
        }
#pragma unroll
        for (int o = NR; o < 32; o <<= 1) acc += __shfl_xor_sync(kFull, acc, o);
        if (es == 0 && jok && cur.d.row >= 0) st_relaxed(P.x + (size_t)cur.d.row * nr + j, cur.b - acc);
    }
}

// Vector entries (rw_options.wide_slices = -1): lane l owns entries l, l + 32,
// ... and reads all right-hand sides of an entry in one relaxed vector load, so
// 4 entries per lane held ahead cover rows of up to 128 entries and a long row
// on the critical path costs one round of loads, not one per few entries.
template <typename T, int NR>
__device__ __forceinline__ void xload_relaxed(const T* x, int nrhs, int32_t c, T (&v)[NR]) {
    const T* p = x + (size_t)c * nrhs;
    if constexpr (NR >= 2 && sizeof(T) == 8) {
        if (nrhs == NR && aligned16(x)) {
#pragma unroll
            for (int j = 0; j < NR; j += 2) ld_relaxed_v2(reinterpret_cast<const double*>(p + j), v[j], v[j + 1]);
            return;
        }
    } else if constexpr (NR >= 4 && sizeof(T) == 4) {
        if (nrhs == NR && aligned16(x)) {
#pragma unroll
            for (int j = 0; j < NR; j += 4)
                ld_relaxed_v4(reinterpret_cast<const float*>(p + j), v[j], v[j + 1], v[j + 2], v[j + 3]);
            return;
        }
    }
#pragma unroll
    for (int j = 0; j < NR; ++j) v[j] = j < nrhs ? ld_relaxed(p + j) : T(0);
}

template <typename T, int NR>
__device__ __forceinline__ bool any_pending(const T (&v)[NR], int nrhs) {
    bool pend = false;
#pragma unroll
    for (int j = 0; j < NR; ++j) pend |= (j < nrhs) && is_pending(v[j]);
    return pend;
}

// MINB = 2 caps the registers so that two 512-thread blocks share an SM:
// twice the rows in flight, at the cost of some spilled prefetch state.
template <typename T, int NR, int MINB>
__global__ void __launch_bounds__(512, MINB) k_rows_vec(const RowParams<T> P) {
    constexpr int U = kPreEntries;
    const int lane = (int)lane_id();
    constexpr int span = 32 / NR;
    const int jo = lane / span;  // the right-hand side this lane stores
    const bool owner = (lane % span) == 0 && jo < P.nrhs;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const unsigned spin_limit = P.st->spin_limit;
    // re-polls (bounded, backing off) while any of the vector is pending
    auto wait_vec = [&](const T* src, int32_t c, T (&v)[NR]) {
        unsigned spins = 0;
        while (any_pending<T, NR>(v, P.nrhs)) {
            if (wait_gives_up(spins, spin_limit, &P.st->timeout)) {
#pragma unroll
                for (int j = 0; j < NR; ++j) v[j] = T(0);
                return;
            }
            if (spins > 4) __nanosleep(32);
            xload_relaxed<T, NR>(src, P.nrhs, c, v);
        }
    };
    struct Pre {
        SolveRow d;
        int32_t c[U];
        T y[U];
        T b;
    };
    auto load = [&](const SolveRow& d, Pre& R) {
        R.d = d;
#pragma unroll
        for (int u = 0; u < U; ++u) row_entry(P, d, lane + u * 32, R.c[u], R.y[u]);
        R.b = owner && d.row >= 0 ? P.rhs[(size_t)d.row * P.nrhs + jo] : T(0);
    };
    Pre pre[2];
    load(row_at(P, gw), pre[0]);
    load(row_at(P, gw + nw), pre[1]);
    SolveRow after = row_at(P, gw + 2 * nw);
    for (int64_t pos = gw; pos < P.n; pos += nw) {
        const Pre cur = pre[0];
        pre[0] = pre[1];
        load(after, pre[1]);
        after = row_at(P, pos + 3 * nw);
        const int cnt = cur.d.cnt;
        const T* const src = P.x;
        T acc[NR];
#pragma unroll
        for (int j = 0; j < NR; ++j) acc[j] = T(0);
        int32_t c[U];
        T y[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            c[u] = cur.c[u];
            y[u] = cur.y[u];
        }
        bool first = cur.d.last >= 0;
        for (int base = 0; base < cnt; base += U * 32) {
            if (base > 0) {
#pragma unroll
                for (int u = 0; u < U; ++u) row_entry(P, cur.d, base + lane + u * 32, c[u], y[u]);
            }
            T v[U][NR];
            bool pend = false;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (base + lane + u * 32 < cnt) {
                    xload_relaxed<T, NR>(src, P.nrhs, c[u], v[u]);
                    pend |= any_pending<T, NR>(v[u], P.nrhs);
                } else {
#pragma unroll
                    for (int j = 0; j < NR; ++j) v[u][j] = T(0);
                }
            }
            if (first && __any_sync(kFull, pend)) {
                T w[NR];
                xload_relaxed<T, NR>(src, P.nrhs, cur.d.last, w);
                wait_vec(src, cur.d.last, w);
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (base + lane + u * 32 < cnt && any_pending<T, NR>(v[u], P.nrhs)) {
                        if (NR == 1 && c[u] == cur.d.last) v[u][0] = w[0];
                        else xload_relaxed<T, NR>(src, P.nrhs, c[u], v[u]);
                    }
                first = false;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (base + u * 32 < cnt) {  // (FP64 instructions only for the slots the row uses)
                    if (base + lane + u * 32 < cnt) wait_vec(src, c[u], v[u]);
#pragma unroll
                    for (int j = 0; j < NR; ++j) acc[j] += y[u] * v[u][j];
                }
            }
        }
        const T sum = warp_sums_spread<T, NR>(acc);
        if (owner && cur.d.row >= 0) st_relaxed(P.x + (size_t)cur.d.row * P.nrhs + jo, cur.b - sum);
    }
}

// Rows of the widest levels (at least kWideRows, more rows than warps), one
// right-hand side: a warp takes four rows of one level, eight lanes each, so
// that every FP64 instruction serves four rows and a level takes a quarter of
// the rounds.  The rows array pads the levels of such a stretch to whole groups
// of four; rows of different levels never share a warp (one could wait for
// another).  Latency of the loads bounds it.  61x64x67 asymmetric grid, FP64:
// these levels and the rest 219 us per application with a row per warp, 204 us
// packed (227 us with two thread blocks per SM, more polls than work); 10^6
// nodes, FP32: 25.4 ms of a PCG solve, 24.4 packed, 23.9 with two per SM.  With
// four right-hand sides it was the slower one (64^3 7-point grid: 17.99 ->
// 18.52 ms of PCG): the vector loads of k_rows_vec fill the lanes.
template <typename T>
__global__ void __launch_bounds__(512, sizeof(T) == 4 ? 2 : 1) k_rows_pack(const RowParams<T> P) {
    constexpr int U = kPreEntries, L = kPackLanes, R = kPackRows;
    const int lane = (int)lane_id(), l = lane % L;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t step = (((int64_t)gridDim.x * blockDim.x) >> 5) * R;
    const unsigned spin_limit = P.st->spin_limit;
    auto wait_value = [&](int32_t c, T v) -> T {
        unsigned spins = 0;
        while (is_pending(v)) {
            if (wait_gives_up(spins, spin_limit, &P.st->timeout)) return T(0);
            if (spins > 4) __nanosleep(32);
            v = ld_relaxed(P.x + c);
        }
        return v;
    };
    struct Pre {
        SolveRow d;
        int32_t c[U];
        T y[U];
        T b;
    };
    auto load = [&](const SolveRow& d, Pre& A) {
        A.d = d;
#pragma unroll
        for (int u = 0; u < U; ++u) row_entry(P, d, l + u * L, A.c[u], A.y[u]);
        A.b = l == 0 && d.row >= 0 ? P.rhs[d.row] : T(0);
    };
    const int64_t first = gw * R + lane / L;
    Pre pre[2];
    load(row_at(P, first), pre[0]);
    load(row_at(P, first + step), pre[1]);
    SolveRow after = row_at(P, first + 2 * step);
    for (int64_t pos = first; pos - lane / L < P.n; pos += step) {  // (warp-uniform)
        const Pre cur = pre[0];
        pre[0] = pre[1];
        load(after, pre[1]);
        after = row_at(P, pos + 3 * step);
        const int cnt = cur.d.cnt;
        T acc = T(0);
        int32_t c[U];
        T y[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            c[u] = cur.c[u];
            y[u] = cur.y[u];
        }
        const int most = __reduce_max_sync(kFull, cnt);
        for (int base = 0; base < most; base += U * L) {
            if (base > 0) {
#pragma unroll
                for (int u = 0; u < U; ++u) row_entry(P, cur.d, base + l + u * L, c[u], y[u]);
            }
            T v[U];
            bool pend = false;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                v[u] = base + l + u * L < cnt ? ld_relaxed(P.x + c[u]) : T(0);
                pend |= is_pending(v[u]);
            }
            if (__any_sync(kFull, pend)) {
                if (cur.d.last >= 0) wait_value(cur.d.last, ld_relaxed(P.x + cur.d.last));
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (is_pending(v[u])) v[u] = ld_relaxed(P.x + c[u]);
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (base + u * L < most) acc += y[u] * wait_value(c[u], v[u]);
        }
#pragma unroll
        for (int o = L / 2; o >= 1; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
        if (l == 0 && cur.d.row >= 0) st_relaxed(P.x + cur.d.row, cur.b - acc);
    }
}

template <typename T, int NR, bool VEC>
static rw_status launch_rows(rw_context* ctx, const RowParams<T>& P, bool pack) {
    int which = VEC && ctx->opt.solve_blocks_per_sm >= 2 ? 1 : 0;
    const void* kern;
    if constexpr (VEC) {
        kern = which ? (const void*)k_rows_vec<T, NR, 2> : (const void*)k_rows_vec<T, NR, 1>;
        if constexpr (NR == 1) {
            if (pack) {
                which = 2;
                kern = (const void*)k_rows_pack<T>;
            }
        }
    } else {
        kern = (const void*)k_rows<T, NR>;
    }
    static int per_sm_of[3] = {-1, -1, -1};
    int& per_sm = per_sm_of[which];
    if (per_sm < 0) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 512, 0);
        if (per_sm < 1) per_sm = 1;
    }
    int64_t blocks = (int64_t)std::min(per_sm, which == 2 && sizeof(T) == 8 ? 1 : 2) * ctx->num_sms;
    const int64_t need = (P.n + 15) / 16;
    if (blocks > need) blocks = need;
    if (blocks < 1) blocks = 1;
    void* args[] = {(void*)&P};
    RW_COUNT_LAUNCH();
    return check_cuda(cudaLaunchCooperativeKernel(kern, dim3((unsigned)blocks), dim3(512), args, 0, ctx->stream),
                      "row solve");
}

// ---------------------------------------------------------------------------
// Narrow stretch: its blocks one after the other, over a co-resident grid of
// one 256-thread block per SM.  The first kMainBlocks of them solve: in step b
// 256 of their warps take one slot of block b each,
//   gather: t_s = p_s - (entries in block b - 1), p_s being the right-hand side
//           minus the earlier entries;
//   a barrier among the solving blocks;
//   solve:  x_s = sum_{u <= s} (L_BB^-1)_su t_u;
//   a barrier of the whole grid.
// The other blocks prepare p of block b + 1 meanwhile: everything up to block
// b - 1 is final.  Entries from before the stretch, most of the thousands that
// the long rows of Y^T hold, are summed by the whole chip before it
// (k_stretch_begin).  The chain per block is then two barriers and two rounds
// of loads.
// ---------------------------------------------------------------------------
static_assert(kBlockRows % kMainBlocks == 0 && kBlockRows / kMainBlocks <= 8, "a warp of a solving block per slot");
constexpr int kLongGather = 512;

template <typename T>
struct BlockSums {
    const int64_t* __restrict__ ptr;
    const int32_t* __restrict__ idx;
    const T* __restrict__ val;
};

template <typename T>
struct BlockParams {
    const SolveBlock* __restrict__ blocks;
    int32_t block0, nblocks;
    const int32_t* __restrict__ trow;
    BlockSums<T> prev, older;
    bool from_rhs;           // the stretch starts the order: t has not been set
    const T* __restrict__ inv;
    const T* __restrict__ rhs;
    T* x;
    T* t;
    int nrhs;
    unsigned* bar;           // [0] grid barrier, [1] barrier of the solving blocks
    unsigned epoch0, mid0;   // barriers passed by earlier launches of this solve
    DevStatus* st;
};

// Barrier of the thread blocks that arrive at *count (see grid_barrier): passed
// when it reaches target.  Returns false when a wait gave up.
__device__ __forceinline__ bool blocks_barrier(unsigned* count, unsigned target, DevStatus* st) {
    __shared__ int give_up;
    __syncthreads();
    if (threadIdx.x == 0) {
        give_up = 0;
        const unsigned limit = st->spin_limit;
        atom_add_release(count, 1u);
        unsigned spins = 0;
        while ((int)(ld_acquire_u32(count) - target) < 0) {
            if (wait_gives_up(spins, limit, &st->timeout)) {
                give_up = 1;
                break;
            }
        }
    }
    __syncthreads();
    return give_up == 0;
}

// The nrhs values at node c (vector loads when nrhs == NR and x is aligned for
// them: a caller's vector need not be), from L2.
template <typename T, int NR>
__device__ __forceinline__ void xload_cg(const T* x, int nrhs, int64_t c, T (&v)[NR]) {
    const T* p = x + c * nrhs;
    if constexpr (NR >= 2 && sizeof(T) == 8) {
        if (nrhs == NR && aligned16(x)) {
#pragma unroll
            for (int j = 0; j < NR; j += 2) {
                const double2 d = __ldcg(reinterpret_cast<const double2*>(p + j));
                v[j] = d.x;
                v[j + 1] = d.y;
            }
            return;
        }
    } else if constexpr (NR >= 4 && sizeof(T) == 4) {
        if (nrhs == NR && aligned16(x)) {
#pragma unroll
            for (int j = 0; j < NR; j += 4) {
                const float4 d = __ldcg(reinterpret_cast<const float4*>(p + j));
                v[j] = d.x;
                v[j + 1] = d.y;
                v[j + 2] = d.z;
                v[j + 3] = d.w;
            }
            return;
        }
    }
#pragma unroll
    for (int j = 0; j < NR; ++j) v[j] = j < nrhs ? __ldcg(p + j) : T(0);
}

// acc += sum of val[q] * x[idx[q]] over q = q0, q0 + step, ... < q1
template <typename T, int NR>
__device__ __forceinline__ void gather(const BlockSums<T>& B, const T* x, int nrhs, int64_t q0, int64_t q1, int step,
                                       T (&acc)[NR]) {
    constexpr int U = NR >= 16 ? 1 : NR >= 8 ? 2 : 4;
    for (int64_t q = q0; q < q1; q += (int64_t)U * step) {
        int32_t c[U];
        T y[U], v[U][NR];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool ok = q + u * step < q1;
            c[u] = ok ? B.idx[q + u * step] : -1;
            y[u] = ok ? B.val[q + u * step] : T(0);
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (c[u] >= 0) xload_cg<T, NR>(x, nrhs, c[u], v[u]);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (c[u] >= 0) {
#pragma unroll
                for (int j = 0; j < NR; ++j) acc[j] += y[u] * v[u][j];
            }
    }
}

// t of `count` <= 8 slots from t0 on, less their rows' sums over B: a warp per
// slot, the whole thread block for a row of more than kLongGather entries.
// from_rhs: t starts as the right-hand side (otherwise as what it holds).
template <typename T, int NR>
__device__ __forceinline__ void gather_slots(const BlockSums<T>& B, const T* x, const T* rhs, bool from_rhs,
                                             const int32_t* trow, T* t, int nr, int64_t t0, int count,
                                             T (&part)[8][NR]) {
    constexpr int span = 32 / NR;
    const int lane = (int)lane_id(), warp = (int)threadIdx.x >> 5;
    const int jo = lane / span;
    const bool owner = (lane % span) == 0 && jo < nr;
    for (int i = 0; i < count; ++i) {
        const int64_t q0 = B.ptr[t0 + i], q1 = B.ptr[t0 + i + 1];
        const bool whole = q1 - q0 > kLongGather;
        if (!whole && warp != i) continue;
        T acc[NR];
#pragma unroll
        for (int j = 0; j < NR; ++j) acc[j] = T(0);
        if (whole) gather<T, NR>(B, x, nr, q0 + threadIdx.x, q1, 256, acc);
        else gather<T, NR>(B, x, nr, q0 + lane, q1, 32, acc);
        T sum = warp_sums_spread<T, NR>(acc);
        if (whole) {
            __syncthreads();
            if ((lane % span) == 0) part[warp][jo] = sum;
            __syncthreads();
            if (warp != i) continue;
            sum = T(0);
            for (int w = 0; w < 8; ++w) sum += part[w][jo];
        }
        if (owner) {
            T* to = t + (t0 + i) * nr + jo;
            __stcg(to, (from_rhs ? rhs[(size_t)trow[t0 + i] * nr + jo] : __ldcg(to)) - sum);
        }
    }
}

// The right-hand sides of a stretch's slots less their rows' entries from
// before the stretch.
template <typename T, int NR>
__global__ void __launch_bounds__(256) k_stretch_begin(int64_t t0, int64_t t1, const SolveBlock* __restrict__ blocks,
                                                       const BlockSums<T> B, const T* x, const T* __restrict__ rhs,
                                                       const int32_t* __restrict__ trow, T* t, int nr) {
    __shared__ T part[8][NR];
    for (int64_t s = t0 + (int64_t)blockIdx.x * 8; s < t1; s += (int64_t)gridDim.x * 8) {
        const int rows = blocks[s / kBlockRows].rows - (int)(s % kBlockRows);
        if (rows > 0) gather_slots<T, NR>(B, x, rhs, true, trow, t, nr, s, min(8, rows), part);
    }
}

template <typename T, int NR>
__global__ void __launch_bounds__(256, 1) k_blocks(const BlockParams<T> P) {
    constexpr int span = 32 / NR;
    constexpr int U = 4;                    // entries per lane of the block before read ahead
    constexpr int V = kBlockRows / 32;      // entries per lane of the inverse's row
    __shared__ T part[8][NR];
    const int lane = (int)lane_id(), warp = (int)threadIdx.x >> 5;
    const int jo = lane / span;  // the right-hand side this lane stores
    const bool owner = (lane % span) == 0 && jo < P.nrhs;
    const bool solves = (int)blockIdx.x < kMainBlocks;
    const int nr = P.nrhs;
    const int slot = warp * kMainBlocks + (int)blockIdx.x;  // rows of all lengths on every SM

    // what step b reads that does not depend on x, loaded before the barrier that starts it
    bool mine = false;
    int32_t row = 0, c[U];
    int64_t q1 = 0, q0 = 0;
    T y[U], iv[V];
    auto fetch = [&](int64_t b) {
        mine = slot < P.blocks[b].rows;
        const int64_t t = b * kBlockRows + slot;
        q0 = q1 = 0;
        if (mine) {
            row = P.trow[t];
            q0 = P.prev.ptr[t] + lane;
            q1 = P.prev.ptr[t + 1];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool ok = q0 + 32 * u < q1;
            c[u] = ok ? P.prev.idx[q0 + 32 * u] : -1;
            y[u] = ok ? P.prev.val[q0 + 32 * u] : T(0);
        }
        const T* inv = P.inv + (b - P.block0) * tri(kBlockRows) + tri(slot);  // (every block before is full)
#pragma unroll
        for (int k = 0; k < V; ++k) iv[k] = mine && lane + 32 * k <= slot ? inv[lane + 32 * k] : T(0);
    };

    unsigned epoch = P.epoch0, mid = P.mid0;
    if (solves && slot < kBlockRows) fetch(P.block0);
    for (int i = 0; i < P.nblocks; ++i) {
        const int64_t b = P.block0 + i, t = b * kBlockRows + slot;
        if (solves) {
            if (mine) {
                // (the stretch's first block has no earlier entries in it)
                const T p = !owner                 ? T(0)
                            : P.from_rhs && i == 0 ? P.rhs[(size_t)row * nr + jo]
                                                   : __ldcg(P.t + t * nr + jo);
                T acc[NR];
#pragma unroll
                for (int j = 0; j < NR; ++j) acc[j] = T(0);
                constexpr int W = NR >= 16 ? 1 : NR >= 8 ? 2 : U;  // loads in flight
#pragma unroll
                for (int u0 = 0; u0 < U; u0 += W) {
                    T v[W][NR];
#pragma unroll
                    for (int u = 0; u < W; ++u)
                        if (c[u0 + u] >= 0) xload_cg<T, NR>(P.x, nr, c[u0 + u], v[u]);
#pragma unroll
                    for (int u = 0; u < W; ++u)
                        if (c[u0 + u] >= 0) {
#pragma unroll
                            for (int j = 0; j < NR; ++j) acc[j] += y[u0 + u] * v[u][j];
                        }
                }
                gather<T, NR>(P.prev, P.x, nr, q0 + 32 * U, q1, 32, acc);
                const T sum = warp_sums_spread<T, NR>(acc);
                if (owner) __stcg(P.t + t * nr + jo, p - sum);
            }
            if (!blocks_barrier(P.bar + 1, ++mid * (unsigned)kMainBlocks, P.st)) return;
            if (mine) {
                T acc[NR];
#pragma unroll
                for (int j = 0; j < NR; ++j) acc[j] = T(0);
                constexpr int W = NR >= 8 ? 1 : 16 / NR >= V ? V : 16 / NR;  // loads in flight
#pragma unroll
                for (int k0 = 0; k0 < V; k0 += W) {
                    T v[W][NR];
#pragma unroll
                    for (int k = 0; k < W; ++k)
                        if (lane + 32 * (k0 + k) <= slot)
                            xload_cg<T, NR>(P.t, nr, b * kBlockRows + lane + 32 * (k0 + k), v[k]);
#pragma unroll
                    for (int k = 0; k < W; ++k)
                        if (32 * (k0 + k) <= slot) {  // (FP64 instructions only for what the row holds)
                            // (the loads above do not wait for the inverse)
#pragma unroll
                            for (int j = 0; j < NR; ++j)
                                acc[j] += nonzero(iv[k0 + k]) ? iv[k0 + k] * v[k][j] : T(0);
                        }
                }
                const T sum = warp_sums_spread<T, NR>(acc);
                if (owner) __stcg(P.x + (size_t)row * nr + jo, sum);
            }
            if (i + 1 < P.nblocks && slot < kBlockRows) fetch(b + 1);
        } else if (i + 1 < P.nblocks) {
            // p of the next block's slots, eight at a time
            const int rows = P.blocks[b + 1].rows, others = (int)gridDim.x - kMainBlocks;
            for (int s0 = ((int)blockIdx.x - kMainBlocks) * 8; s0 < rows; s0 += others * 8)
                gather_slots<T, NR>(P.older, P.x, P.rhs, P.from_rhs, P.trow, P.t, nr, (b + 1) * kBlockRows + s0,
                                    min(8, rows - s0), part);
        }
        if (i + 1 < P.nblocks && !blocks_barrier(P.bar, ++epoch * gridDim.x, P.st)) return;
    }
}

template <typename T, int NR>
static rw_status launch_blocks(rw_context* ctx, const BlockParams<T>& P) {
    void* args[] = {(void*)&P};
    RW_COUNT_LAUNCH();
    return check_cuda(cudaLaunchCooperativeKernel((const void*)k_blocks<T, NR>, dim3((unsigned)ctx->num_sms),
                                                  dim3(256), args, 0, ctx->stream),
                      "block solve");
}

// Before a solve: x marked pending (solve modes 1 and 2), the barrier words of
// its block launches cleared, and in the forward solve w <- w / d row by row (the
// D^-1 step between the two solves: one FP64 division instruction serves 32 rows
// here, one row inside the solve).
template <typename T>
__global__ void k_solve_begin(T* x, int64_t cnt, T* w, const T* __restrict__ d, int nrhs, unsigned* bar) {
    const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    if (i0 < 2) bar[i0] = 0u;
    for (int64_t i = i0; i < cnt; i += step) {
        if (x) x[i] = pending_value(T(0));
        if (w) w[i] = w[i] / d[i / nrhs];
    }
}

// ---------------------------------------------------------------------------
// Host dispatch
// ---------------------------------------------------------------------------
// Entry slices of the lane groups: an explicit option, else 32 / NR (one
// row per warp), as a power of two with NR * ES <= 32.
static int lane_slices(int opt, int NR) {
    if (opt < 0) return 0;  // vector rows
    const int es = opt > 0 ? opt : 32 / NR;
    int p = 1;
    while (p * 2 <= es && p * 2 * NR <= 32) p *= 2;
    return p;
}

template <typename T, int NR, int ES>
static rw_status launch_wide(rw_context* ctx, const SolveSchedule& S, int32_t lev_begin, int32_t lev_end,
                             const int64_t* rp, const int32_t* col, const T* val, const T* rhs,
                             T* x, int nrhs, unsigned* bar) {
    if constexpr (NR * ES > 32) {
        return RW_ERR_ARG;
    } else {
        cudaStream_t s = ctx->stream;
        static int per_sm = -1;
        if (per_sm < 0) {
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_wide<T, NR, ES>, kWideThreads, 0);
            if (per_sm < 1) per_sm = 1;
        }
        rw_status rc;
        if ((rc = check_cuda(cudaMemsetAsync(bar, 0, 2 * sizeof(unsigned), s), "memset"))) return rc;
        const int bps = ctx->opt.solve_blocks_per_sm > 0 ? ctx->opt.solve_blocks_per_sm : 1;
        int64_t blocks = (int64_t)std::min(per_sm, bps) * ctx->num_sms;
        int64_t maxw = 0;
        for (int32_t l = lev_begin; l < lev_end; ++l) maxw = std::max(maxw, S.lptr_h[l + 1] - S.lptr_h[l]);
        constexpr int64_t rows_per_block = (kWideThreads / 32) * (32 / group_lanes<NR, ES>());
        const int64_t need = (maxw + rows_per_block - 1) / rows_per_block;
        if (blocks > need) blocks = need;
        if (blocks < 1) blocks = 1;
        WideParams<T> P{lev_begin, lev_end, S.lptr, S.order, rp, col, val, rhs, x, nrhs, bar, ctx->d_status};
        void* args[] = {(void*)&P};
        RW_COUNT_LAUNCH();
        return check_cuda(cudaLaunchCooperativeKernel((const void*)k_wide<T, NR, ES>, dim3((unsigned)blocks),
                                                      dim3(kWideThreads), args, 0, s),
                          "wide-run solve");
    }
}

template <typename T, int NR, int ES>
static rw_status launch_cluster(rw_context* ctx, const SolveSchedule& S, int32_t lev_begin, int32_t lev_end,
                                const int64_t* rp, const int32_t* col, const T* val, const T* rhs,
                                T* x, int nrhs, unsigned* bar, int csize) {
    if constexpr (NR * ES > 32) {
        return RW_ERR_ARG;
    } else {
        rw_status arc = set_kernel_attr_once(ctx->device, (const void*)k_cluster<T, NR, ES>,
                                             cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (arc) return arc;
        WideParams<T> P{lev_begin, lev_end, S.lptr, S.order, rp, col, val, rhs, x, nrhs, bar, ctx->d_status};
        cudaLaunchConfig_t cfg = {};
        cfg.blockDim = dim3(NR >= 8 ? 512u : 1024u);
        cfg.dynamicSmemBytes = 0;
        cfg.stream = ctx->stream;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        // the largest size up to csize that the device can place (once per size)
        static int placeable[17] = {};
        if (csize < 1 || csize > 16) csize = 16;
        while (csize > 1) {
            if (placeable[csize] == 0) {
                cfg.gridDim = dim3((unsigned)csize);
                at[0].val.clusterDim.x = (unsigned)csize;
                int nc = 0;
                placeable[csize] =
                    (cudaOccupancyMaxActiveClusters(&nc, k_cluster<T, NR, ES>, &cfg) == cudaSuccess && nc >= 1) ? 1 : -1;
                cudaGetLastError();
            }
            if (placeable[csize] > 0) break;
            csize >>= 1;
        }
        cfg.gridDim = dim3((unsigned)csize);
        at[0].val.clusterDim.x = (unsigned)csize;
        RW_COUNT_LAUNCH();
        return check_cuda(cudaLaunchKernelEx(&cfg, k_cluster<T, NR, ES>, P), "cluster-run solve");
    }
}

// Levels [l, end) one after another: consecutive levels up to the cluster width
// go to one cluster, the rest to the whole grid.
template <typename T, int NR, int ES>
static rw_status launch_levels(rw_context* ctx, const SolveSchedule& S, int32_t l, int32_t end, const int64_t* rp,
                               const int32_t* col, const T* val, const T* rhs, T* x, int nrhs, unsigned* bar) {
    const int64_t cw = ctx->opt.cluster_width > 0 ? ctx->opt.cluster_width : 0;
    const int csize = ctx->opt.cluster_size > 0 ? ctx->opt.cluster_size : 16;
    while (l < end) {
        const bool narrow = cw > 0 && S.lptr_h[l + 1] - S.lptr_h[l] <= cw;
        int32_t e = l + 1;
        while (e < end && (cw > 0 && S.lptr_h[e + 1] - S.lptr_h[e] <= cw) == narrow) ++e;
        // cluster runs (1024-thread blocks, 64 registers) keep lane groups
        constexpr int CES = ES == 0 ? 32 / NR : ES;
        rw_status rc = narrow ? launch_cluster<T, NR, CES>(ctx, S, l, e, rp, col, val, rhs, x, nrhs, bar, csize)
                              : launch_wide<T, NR, ES>(ctx, S, l, e, rp, col, val, rhs, x, nrhs, bar);
        if (rc) return rc;
        l = e;
    }
    return RW_OK;
}

template <typename T>
static const T* schedule_values(const double* v, const float* v32) {
    if constexpr (sizeof(T) == 8) return v;
    else return v32;
}

template <typename T>
static BlockSums<T> block_sums(const SolveEntries& E) {
    return BlockSums<T>{E.ptr, E.idx, schedule_values<T>(E.val, E.val32)};
}

template <typename T, int NR>
static rw_status solve_runs_nr(rw_context* ctx, const SolveSchedule& S, const int64_t* rp,
                               const int32_t* col, const T* val, const T* rhs, T* x, int nrhs, unsigned* bar, int mode,
                               bool backward, T* w, const T* d, void* t) {
    cudaStream_t s = ctx->stream;
    rw_status rc;
    const bool rows = mode == 1 || mode == 2;
    const int64_t cnt = (int64_t)S.n * nrhs;
    if (rows || w) {
        RW_COUNT_LAUNCH();
        k_solve_begin<T><<<grid_for(cnt, 256, ctx->num_sms * 8), 256, 0, s>>>(rows ? x : nullptr, cnt, w, d, nrhs, bar);
        if ((rc = check_launch("solve begin"))) return rc;
    }
    // the rows in slots [slot0, slot1); vector entries while one entry's
    // right-hand sides fit in 32 bytes of registers
    auto solve_rows = [&](int64_t slot0, int64_t slot1, bool pack) -> rw_status {
        const RowParams<T> P{slot1 - slot0, S.rows + slot0, col, val, rhs, x, nrhs, ctx->d_status};
        if constexpr (NR * sizeof(T) <= 32) {
            // One FP32 right-hand side backward, blocks per SM left to the library: the entries of the long rows of
            // Y^T over lane groups, two thread blocks per SM (k_rows), 3.8 -> 3.2 ms per solve of 10^6 nodes with
            // long-range edges, 1.19 -> 1.12 ms on a 56^3 27-point grid; forward the same costs 2.4 -> 2.9 ms.
            const bool groups = sizeof(T) * NR == 4 && backward && !pack && ctx->opt.solve_blocks_per_sm <= 0;
            if (ctx->opt.wide_slices < 0 && !groups) return launch_rows<T, NR, true>(ctx, P, pack);
        }
        return launch_rows<T, NR, false>(ctx, P, false);
    };
    if (mode == 1) return solve_rows(0, S.nrows, false);
    // the levels [l, end) one after another
    auto solve_levels = [&](int32_t l, int32_t end) -> rw_status {
        switch (lane_slices(ctx->opt.wide_slices, NR)) {
            case 0: {
                // vector rows while one entry's right-hand sides fit in 64 bytes of registers
                constexpr int ES = NR * sizeof(T) <= 64 ? 0 : 32 / NR;
                return launch_levels<T, NR, ES>(ctx, S, l, end, rp, col, val, rhs, x, nrhs, bar);
            }
            case 1: return launch_levels<T, NR, 1>(ctx, S, l, end, rp, col, val, rhs, x, nrhs, bar);
            case 2: return launch_levels<T, NR, 2>(ctx, S, l, end, rp, col, val, rhs, x, nrhs, bar);
            case 4: return launch_levels<T, NR, 4>(ctx, S, l, end, rp, col, val, rhs, x, nrhs, bar);
            case 8: return launch_levels<T, NR, 8>(ctx, S, l, end, rp, col, val, rhs, x, nrhs, bar);
            case 16: return launch_levels<T, NR, 16>(ctx, S, l, end, rp, col, val, rhs, x, nrhs, bar);
            default: return launch_levels<T, NR, 32>(ctx, S, l, end, rp, col, val, rhs, x, nrhs, bar);
        }
    };
    unsigned epoch = 0, mid = 0;
    bool clear = rows || w;  // the barrier words hold the epochs
    const bool packs = rows && NR == 1 && ctx->opt.wide_slices < 0;
    for (size_t i = 0; i < S.stretches.size(); ++i) {
        const SolveStretch& st = S.stretches[i];
        if (st.nblocks == 0) {
            const bool pack = packs && st.pack;
            size_t e = i;  // unpacked neighbours in one launch
            while (!pack && e + 1 < S.stretches.size() && S.stretches[e + 1].nblocks == 0 &&
                   !(packs && S.stretches[e + 1].pack))
                ++e;
            i = e;
            if (rows) {
                rc = solve_rows(st.slot0, S.stretches[e].slot1, pack);
            } else {
                rc = solve_levels(st.lev0, S.stretches[e].lev1);
                clear = false;
            }
            if (rc) return rc;
            continue;
        }
        if (!clear) {
            if ((rc = check_cuda(cudaMemsetAsync(bar, 0, 2 * sizeof(unsigned), s), "memset"))) return rc;
            epoch = mid = 0;
            clear = true;
        }
        BlockParams<T> P{};
        P.blocks = S.blocks;
        P.block0 = st.block0;
        P.nblocks = st.nblocks;
        P.trow = S.trow;
        P.prev = block_sums<T>(S.ext[0]);
        P.older = block_sums<T>(S.ext[1]);
        P.from_rhs = st.pos0 == 0;
        P.inv = schedule_values<T>(S.inv, S.inv32) + st.inv0;
        P.rhs = rhs;
        P.x = x;
        P.t = static_cast<T*>(t ? t : S.t);
        P.nrhs = nrhs;
        P.bar = bar;
        P.epoch0 = epoch;
        P.mid0 = mid;
        P.st = ctx->d_status;
        if (st.pos0 > 0) {
            const int64_t t0 = (int64_t)st.block0 * kBlockRows, t1 = t0 + (int64_t)st.nblocks * kBlockRows;
            RW_COUNT_LAUNCH();
            k_stretch_begin<T, NR><<<grid_for((t1 - t0) / 8, 1, ctx->num_sms * 8), 256, 0, s>>>(
                t0, t1, S.blocks, block_sums<T>(S.ext[2]), x, rhs, S.trow, P.t, nrhs);
            if ((rc = check_launch("stretch begin"))) return rc;
        }
        if ((rc = launch_blocks<T, NR>(ctx, P))) return rc;
        epoch += (unsigned)st.nblocks - 1;
        mid += (unsigned)st.nblocks;
    }
    return RW_OK;
}

template <typename T>
rw_status solve_runs(rw_context* ctx, const SolveSchedule& S, const int64_t* rp, const int32_t* col,
                     const T* val, const T* rhs, T* x, int nrhs, unsigned* bar, bool backward, T* w, const T* d,
                     void* t) {
    NvtxRange nvtx_range(backward ? "rw_solve_bwd" : "rw_solve_fwd");
    if (S.n == 0) return RW_OK;
    const int mode = backward && ctx->opt.solve_mode_bwd >= 0 ? ctx->opt.solve_mode_bwd : ctx->opt.solve_mode;
    int nr = 1;
    while (nr < nrhs) nr <<= 1;
    switch (nr) {
        case 1: return solve_runs_nr<T, 1>(ctx, S, rp, col, val, rhs, x, nrhs, bar, mode, backward, w, d, t);
        case 2: return solve_runs_nr<T, 2>(ctx, S, rp, col, val, rhs, x, nrhs, bar, mode, backward, w, d, t);
        case 4: return solve_runs_nr<T, 4>(ctx, S, rp, col, val, rhs, x, nrhs, bar, mode, backward, w, d, t);
        case 8: return solve_runs_nr<T, 8>(ctx, S, rp, col, val, rhs, x, nrhs, bar, mode, backward, w, d, t);
        default: return solve_runs_nr<T, 16>(ctx, S, rp, col, val, rhs, x, nrhs, bar, mode, backward, w, d, t);
    }
}

template rw_status solve_runs<double>(rw_context*, const SolveSchedule&, const int64_t*, const int32_t*,
                                      const double*, const double*, double*, int, unsigned*, bool, double*,
                                      const double*, void*);
template rw_status solve_runs<float>(rw_context*, const SolveSchedule&, const int64_t*, const int32_t*,
                                     const float*, const float*, float*, int, unsigned*, bool, float*, const float*,
                                     void*);

}  // namespace rw
