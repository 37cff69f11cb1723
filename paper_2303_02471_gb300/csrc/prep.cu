// Preprocessing kernels of the column-wise SpGEMM (arXiv 2303.02471):
// input validation, row compaction, the operation count Op_j with binning (Section 3.1's
// "Sorting" pre-pass, done as a bucket pass), per-bin column lists, and the
// int64 scan that turns per-column counts into C's column pointers.
#include <cstring>

#include "kernels.cuh"

namespace spg {

// CSC well-formedness of A (Section 2.1: colptr[0] = 0, colptr[n] = nnz,
// colptr non-decreasing, rows in [0, nrows)), its columns' lengths as 32-bit
// integers for the Op count's gathers, and a mark per row that holds an entry,
// in one pass over A.  A mark is a plain store of eight bytes: stores to one
// L2 sector from many SMs take turns, so narrow marks lose (bytes took 133 us
// for the 4.7M entries of the very sparse product and 370 us for the skewed
// rows of R-MAT 2^18, bits set by atomics 46 and 25 us, so 30 and 42 us).
constexpr int kCheckUnroll = 4;

__global__ void __launch_bounds__(256) k_check_rows(const int64_t *__restrict__ cp, const int32_t *__restrict__ row,
                                                   int64_t nrows, int64_t ncols, int64_t nnz, int validate,
                                                   int64_t *__restrict__ mark, uint32_t *__restrict__ zlen,
                                                   Ctrl *ctrl) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t j = tid; j <= ncols; j += stride) {
        const int64_t c = cp[j], c1 = j < ncols ? cp[j + 1] : c;
        if (j < ncols) zlen[j] = (uint32_t)(c1 - c);
        if (validate && ((j == 0 && c != 0) || (j == ncols && c != nnz) || c1 < c || c < 0))
            set_error(ctrl, SPG_ERR_INVALID, 0, j);
    }
    for (int64_t e0 = tid; e0 < nnz; e0 += kCheckUnroll * stride) {
        int32_t r[kCheckUnroll];
#pragma unroll
        for (int u = 0; u < kCheckUnroll; ++u) r[u] = e0 + u * stride < nnz ? row[e0 + u * stride] : 0;
#pragma unroll
        for (int u = 0; u < kCheckUnroll; ++u) {
            if (e0 + u * stride >= nnz) continue;
            if (r[u] >= 0 && (int64_t)r[u] < nrows) mark[r[u]] = 1;
            else if (validate) set_error(ctrl, SPG_ERR_INVALID, 1, e0 + u * stride);
        }
    }
}

// Rows with entries numbered in ascending order, where compaction applies
// (row_rule): map[r] = compact row or -1, inv[compact] = r.  ctrl->mrows =
// their count.  A CTA takes a tile of kRowTile rows; the rows of the other
// tiles are counted from the marks themselves up to kRowRecount tiles (which
// saves a launch), up to kRowDirect tiles (8.4M rows) from the tiles' counts,
// which every CTA then adds up (64 MB of L2 reads at the limit, growing with
// the square of the tiles: 4.4 TB at 2^31 rows), else from their prefix
// sums, a launch more.  The marks are padded with zeros to whole tiles.
constexpr int kRowTile = 2048;
constexpr int kRowThreads = 256;
constexpr int kRowRecount = 8;
constexpr int64_t kRowDirect = 4096;
constexpr int kRowPer = kRowTile / kRowThreads;  // consecutive rows of a thread

// The marks of thread threadIdx.x in tile `tile`, as bits.
__device__ __forceinline__ uint32_t row_bits(const ulonglong2 *__restrict__ marks, int64_t tile) {
    uint32_t b = 0;
#pragma unroll
    for (int i = 0; i < kRowPer / 2; ++i) {
        const ulonglong2 v = marks[(tile * kRowThreads + threadIdx.x) * (kRowPer / 2) + i];
        b |= ((uint32_t)v.x | ((uint32_t)v.y << 1)) << (2 * i);
    }
    return b;
}

__global__ void __launch_bounds__(kRowThreads) k_row_counts(const ulonglong2 *__restrict__ marks,
                                                           int32_t *__restrict__ counts) {
    __shared__ int s_n;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    const int w = __reduce_add_sync(0xffffffffu, __popc(row_bits(marks, blockIdx.x)));
    if ((threadIdx.x & 31) == 0) atomicAdd(&s_n, w);
    __syncthreads();
    if (threadIdx.x == 0) counts[blockIdx.x] = s_n;
}

// One CTA: the counts of `tiles` tiles into their exclusive prefix sums, the
// total at counts[tiles] (at most the rows, so below 2^31).  kRowSumItems
// consecutive counts a thread and step.
constexpr int kRowSumThreads = 1024;
constexpr int kRowSumItems = 8;

__global__ void __launch_bounds__(kRowSumThreads) k_row_sums(int32_t *counts, int64_t tiles) {
    __shared__ int s_warp[kRowSumThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int carry = 0;
    for (int64_t base = 0; base < tiles; base += kRowSumThreads * kRowSumItems) {
        const int64_t i0 = base + (int64_t)threadIdx.x * kRowSumItems;
        int v[kRowSumItems];
        int sum = 0;
#pragma unroll
        for (int u = 0; u < kRowSumItems; ++u) {
            v[u] = i0 + u < tiles ? counts[i0 + u] : 0;
            sum += v[u];
        }
        int incl = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += o;
        }
        if (lane == 31) s_warp[warp] = incl;
        __syncthreads();
        int w = s_warp[lane];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, w, d);
            if (lane >= d) w += o;
        }
        const int total = __shfl_sync(0xffffffffu, w, 31);
        const int before = __shfl_sync(0xffffffffu, w, warp > 0 ? warp - 1 : 0);
        int run = carry + (warp > 0 ? before : 0) + incl - sum;
#pragma unroll
        for (int u = 0; u < kRowSumItems; ++u) {
            if (i0 + u < tiles) counts[i0 + u] = run;
            run += v[u];
        }
        carry += total;
        __syncthreads();
    }
    if (threadIdx.x == 0) counts[tiles] = carry;
}

// counts: the tiles' counts, or (summed) their prefix sums and the total;
// null: the tiles are counted here.
__global__ void __launch_bounds__(kRowThreads) k_row_index(const ulonglong2 *__restrict__ marks, int64_t m,
                                                          const int32_t *__restrict__ counts, int summed,
                                                          int32_t *__restrict__ map, int32_t *__restrict__ inv,
                                                          Ctrl *ctrl) {
    __shared__ int s_warp[kRowThreads / 32];
    __shared__ int s_before, s_all;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_before = s_all = 0;
    __syncthreads();
    // rows with entries before the tile, and of all tiles
    int before = 0, all = 0;
    if (summed) {
        if (threadIdx.x == 0) {
            before = counts[blockIdx.x];
            all = counts[gridDim.x];
        }
    } else if (counts) {
        for (int64_t i = threadIdx.x; i < gridDim.x; i += kRowThreads) {
            const int n = counts[i];
            all += n;
            if (i < blockIdx.x) before += n;
        }
    } else {
        for (int64_t t = 0; t < gridDim.x; ++t) {
            const int n = __popc(row_bits(marks, t));
            all += n;
            if (t < blockIdx.x) before += n;
        }
    }
    before = __reduce_add_sync(0xffffffffu, before);
    all = __reduce_add_sync(0xffffffffu, all);
    if (lane == 0) {
        atomicAdd(&s_before, before);
        atomicAdd(&s_all, all);
    }
    const uint32_t bits = row_bits(marks, blockIdx.x);
    const int c = __popc(bits);
    int incl = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += o;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x == 0) ctrl->mrows = (unsigned long long)s_all;
    if (!row_rule(s_all, m).compact) return;
    int at = s_before + incl - c;
    for (int i = 0; i < warp; ++i) at += s_warp[i];
    const int64_t r0 = (int64_t)blockIdx.x * kRowTile + kRowPer * threadIdx.x;
#pragma unroll
    for (int i = 0; i < kRowPer; ++i) {
        if (r0 + i >= m) break;
        const bool in = (bits >> i) & 1u;
        map[r0 + i] = in ? at : -1;
        if (in) inv[at++] = (int32_t)(r0 + i);
    }
}

size_t row_mark_bytes(int64_t m) { return (size_t)ceil_div(m, kRowTile) * kRowTile * sizeof(int64_t); }
int64_t row_tile_count(int64_t m) { return ceil_div(m, kRowTile) + 1; }

cudaError_t launch_row_index(const int64_t *mark, int64_t m, int32_t *counts, int32_t *map, int32_t *inv,
                             Ctrl *ctrl, int *launches, cudaStream_t s) {
    const int64_t tiles = ceil_div(m, kRowTile);
    if (tiles <= 0) return cudaSuccess;
    const ulonglong2 *marks = reinterpret_cast<const ulonglong2 *>(mark);
    const bool direct = tiles <= kRowRecount, summed = tiles > kRowDirect;
    if (!direct) k_row_counts<<<(unsigned)tiles, kRowThreads, 0, s>>>(marks, counts);
    if (summed) k_row_sums<<<1, kRowSumThreads, 0, s>>>(counts, tiles);
    k_row_index<<<(unsigned)tiles, kRowThreads, 0, s>>>(marks, m, direct ? nullptr : counts, summed ? 1 : 0, map, inv,
                                                        ctrl);
    *launches += direct ? 1 : summed ? 3 : 2;
    return cudaGetLastError();
}

// A's rows through the compaction map when it is used (grid-stride part of
// the kernel that calls it); a row that held no entry when the map was made
// is reported.
__device__ __forceinline__ void remap_rows(const int32_t *Arow, int64_t nnz, const int32_t *map, int64_t m, int32_t *out,
                                           Ctrl *ctrl) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nnz; i += stride) {
        const int32_t r = Arow[i];
        int32_t c = r >= 0 && r < m ? map[r] : -1;
        if (c < 0) {
            set_error(ctrl, SPG_ERR_INVALID, kDetailRowMap, i);
            c = 0;
        }
        out[i] = c;
    }
}

__global__ void k_row_remap(const int32_t *Arow, int64_t nnz, const int32_t *map, int64_t m, int32_t *out,
                            Ctrl *ctrl) {
    remap_rows(Arow, nnz, map, m, out, ctrl);
}

// Op_j = sum over stored B_kj of Z^A_k (Section 3.1), its bin, the bin
// histogram and the total product count, with B's well-formedness checked on
// the way (a bad pointer or row is reported and not followed) and A's rows
// renumbered first where compaction applies.  Empty columns get nnz 0 here.
//
// A warp takes up to 32 columns, one per lane: runs of kDealRun neighbouring
// columns (their pointers, Op and row entries share sectors), dealt through a
// permutation of the runs (index times `mult` modulo their number, mult
// coprime to it) so that the heavy columns of a skewed matrix, which sit
// together (or, in R-MAT, at indices with few one bits), spread over the
// CTAs.  A lane sums the Z^A_k of its own column up to kCountShort entries,
// kCountUnroll gathers in flight; the longer columns of the CTA's eight warps
// go on a list that the warps share, a warp per column.  A product of few
// columns gives its warps fewer of them (`cols`), so that the gathers'
// latency is spread over the chip.  Z^A_k is one 4-byte gather (a pair of
// 8-byte column pointers kept L1's tag stage busy).  Dealing single columns,
// flattening them 32 entries at a time with 64-bit warp scans and a 64-bit
// division per column took 78 us for the very sparse product of 2^20 columns,
// 47 us for R-MAT 2^18 and 28 us for 15013 columns of 23 entries; 48, 44
// (53 with the renumbering of A) and 16 us so.
constexpr int kCountThreads = 256;
constexpr int kCountShort = 24;
constexpr int kCountUnroll = 4;
constexpr int kCountLong = 8;
constexpr int kDealRun = 4;

// x mod n for x < n^2 < 2^62, with inv = floor(2^64 / n) (n > 1): the quotient
// from the high product is at most one short.
__device__ __forceinline__ int64_t mod_by(unsigned long long x, unsigned long long n, unsigned long long inv) {
    unsigned long long r = x - __umul64hi(x, inv) * n;
    if (r >= n) r -= n;
    return (int64_t)r;
}

// floor(log2(op)) of a column with products.
__device__ __forceinline__ int op_class(int64_t op) { return op >> 31 ? 31 : 31 - __clz((int)op); }

__global__ void __launch_bounds__(kCountThreads) k_count_bin(CountArgs a, Ctrl *ctrl) {
    __shared__ unsigned long long s_hist[NBINS];
    __shared__ unsigned long long s_max[NBINS];
    __shared__ unsigned long long s_binprod[NBINS];
    __shared__ unsigned long long s_binb[NBINS];
    __shared__ unsigned long long s_prod, s_cap;
    __shared__ unsigned s_cls[32];
    __shared__ int64_t s_op[kCountThreads];    // Op of the CTA's columns
    __shared__ int s_long[kCountThreads];      // columns (thread indices) of more than kCountShort entries
    __shared__ int64_t s_lp[kCountThreads];    // their first entry
    __shared__ int32_t s_ln[kCountThreads];    // and number of entries
    __shared__ int s_nlong;
    // what the row pass found: nothing here follows a malformed A.  Other CTAs
    // of this kernel report a malformed B in the same word meanwhile, so one
    // thread reads it for the whole CTA.
    if (__syncthreads_or(threadIdx.x == 0 && ctrl->err != 0)) return;
    if (threadIdx.x < NBINS) {
        s_hist[threadIdx.x] = 0;
        s_max[threadIdx.x] = 0;
        s_binprod[threadIdx.x] = 0;
        s_binb[threadIdx.x] = 0;
    }
    if (threadIdx.x < 32) s_cls[threadIdx.x] = 0;
    if (threadIdx.x == 0) s_prod = s_cap = 0;
    const RowRule rows = row_rule((int64_t)ctrl->mrows, a.mA);
    const int64_t t = effective_t(a.t, a.hmax, rows.m);
    if (rows.compact) remap_rows(a.Arow, a.nnzA, a.rmap, a.mA, a.arow, ctrl);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long mine = 0, cap = 0;
    const int64_t runs = (a.nB + kDealRun - 1) / kDealRun;
    // runs per warp and CTA: a.cols / kDealRun, a power of two up to 8
    const int rw = a.cols / kDealRun, rcta = rw * (kCountThreads / 32);
    for (int64_t g0 = (int64_t)blockIdx.x * rcta; g0 < runs; g0 += (int64_t)gridDim.x * rcta) {
        __syncthreads();
        if (threadIdx.x == 0) s_nlong = 0;
        __syncthreads();
        const int64_t g = lane < a.cols ? g0 + warp * rw + lane / kDealRun : runs;
        const int64_t j = g < runs ? mod_by((unsigned long long)g * (unsigned long long)a.mult,
                                            (unsigned long long)runs, a.inv) * kDealRun + lane % kDealRun
                                   : a.nB;
        const bool on = j < a.nB;
        int64_t p0 = 0;
        int nb = 0;
        if (on) {
            p0 = a.Bcp[j];
            const int64_t p1 = a.Bcp[j + 1];
            if (a.validate && (p0 < 0 || p1 < p0 || p1 > a.nnzB || (j == 0 && p0 != 0) ||
                               (j + 1 == a.nB && p1 != a.nnzB))) {
                set_error(ctrl, SPG_ERR_INVALID, 2, j);
                p0 = 0;
            } else {
                nb = (int)(p1 - p0);  // a column holds at most 2^31 - 1 distinct rows
            }
        }
        if (nb > kCountShort) {
            const int i = atomicAdd(&s_nlong, 1);
            s_long[i] = threadIdx.x;
            s_lp[i] = p0;
            s_ln[i] = nb;
        }
        const int ns = nb > kCountShort ? 0 : nb;
        int64_t s = 0;
        for (int q0 = 0; q0 < ns; q0 += kCountUnroll) {
            int32_t k[kCountUnroll];
#pragma unroll
            for (int u = 0; u < kCountUnroll; ++u) k[u] = q0 + u < ns ? a.Brow[p0 + q0 + u] : -1;
#pragma unroll
            for (int u = 0; u < kCountUnroll; ++u) {
                if (q0 + u >= ns) continue;
                if (a.validate && (k[u] < 0 || (int64_t)k[u] >= a.nA))
                    set_error(ctrl, SPG_ERR_INVALID, 3, p0 + q0 + u);
                else
                    s += a.zlen[k[u]];
            }
        }
        s_op[threadIdx.x] = s;
        __syncthreads();
        // long columns: one warp each, shared by the CTA's warps
        const int nl = s_nlong;
        for (int i = warp; i < nl; i += kCountThreads / 32) {
            const int64_t pc = s_lp[i];
            const int nc = s_ln[i];
            int64_t sz = 0;
            for (int q0 = lane; q0 < nc; q0 += 32 * kCountLong) {
                int32_t k[kCountLong];
#pragma unroll
                for (int u = 0; u < kCountLong; ++u) {
                    const int q = q0 + 32 * u;
                    k[u] = q < nc ? a.Brow[pc + q] : -1;
                    if (a.validate && q < nc && (k[u] < 0 || (int64_t)k[u] >= a.nA)) {
                        set_error(ctrl, SPG_ERR_INVALID, 3, pc + q);
                        k[u] = -1;
                    }
                }
#pragma unroll
                for (int u = 0; u < kCountLong; ++u)
                    if (k[u] >= 0) sz += a.zlen[k[u]];
            }
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) sz += __shfl_xor_sync(0xffffffffu, sz, d);
            if (lane == 0) s_op[s_long[i]] = sz;
        }
        __syncthreads();
        s = s_op[threadIdx.x];
        int b = -1;
        if (on) {
            a.op[j] = s;
            mine += (unsigned long long)s;
            cap += (unsigned long long)(s < rows.m ? s : rows.m);
            b = bin_of(s, t, a.hmax, a.promote);
            if (b == BIN_EMPTY) a.Ccp[j + 1] = 0;
            if (b == BIN_DENSE) atomicAdd(&s_cls[op_class(s)], 1u);
        }
        // per-bin statistics, one group of lanes per bin present; sums of 32
        // values below 2^26 fit 32 bits (else 64-bit butterflies)
        const bool small = __all_sync(0xffffffffu, s < (1 << 26) && nb < (1 << 26));
        unsigned pending = __ballot_sync(0xffffffffu, on);
        while (pending) {
            const int leader = __ffs(pending) - 1;
            const int bb = __shfl_sync(0xffffffffu, b, leader);
            const unsigned m = __ballot_sync(0xffffffffu, on && b == bb);
            const bool in = (m >> lane) & 1u;
            unsigned long long sm, mx, nbs;
            if (small) {
                sm = __reduce_add_sync(0xffffffffu, in ? (unsigned)s : 0u);
                mx = __reduce_max_sync(0xffffffffu, in ? (unsigned)s : 0u);
                nbs = __reduce_add_sync(0xffffffffu, in ? (unsigned)nb : 0u);
            } else {
                sm = mx = in ? (unsigned long long)s : 0ull;
                nbs = in ? (unsigned long long)nb : 0ull;
#pragma unroll
                for (int d = 16; d > 0; d >>= 1) {
                    sm += __shfl_xor_sync(0xffffffffu, sm, d);
                    nbs += __shfl_xor_sync(0xffffffffu, nbs, d);
                    const unsigned long long o = __shfl_xor_sync(0xffffffffu, mx, d);
                    if (o > mx) mx = o;
                }
            }
            if (lane == leader) {
                atomicAdd(&s_hist[bb], (unsigned long long)__popc(m));
                atomicMax(&s_max[bb], mx);
                if (sm) atomicAdd(&s_binprod[bb], sm);
                if (nbs) atomicAdd(&s_binb[bb], nbs);
            }
            pending &= ~m;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.Ccp[0] = 0;
        if (a.validate && a.nB == 0 && (a.Bcp[0] != 0 || a.nnzB != 0)) set_error(ctrl, SPG_ERR_INVALID, 2, 0);
    }
    for (int d = 16; d > 0; d >>= 1) {
        mine += __shfl_xor_sync(0xffffffffu, mine, d);
        cap += __shfl_xor_sync(0xffffffffu, cap, d);
    }
    if (lane == 0) {
        atomicAdd(&s_prod, mine);
        atomicAdd(&s_cap, cap);
    }
    __syncthreads();
    if (threadIdx.x < NBINS && s_hist[threadIdx.x]) {
        atomicAdd(&ctrl->hist[threadIdx.x], s_hist[threadIdx.x]);
        atomicMax(&ctrl->maxop[threadIdx.x], s_max[threadIdx.x]);
        atomicAdd(&ctrl->binprod[threadIdx.x], s_binprod[threadIdx.x]);
        atomicAdd(&ctrl->binnnzb[threadIdx.x], s_binb[threadIdx.x]);
    }
    if (threadIdx.x < 32 && s_cls[threadIdx.x])
        atomicAdd(&ctrl->cls[threadIdx.x], (unsigned long long)s_cls[threadIdx.x]);
    if (threadIdx.x == 0) {
        atomicAdd(&ctrl->products, s_prod);
        atomicAdd(&ctrl->capsum, s_cap);
    }
}

cudaError_t launch_count_bin(const CountArgs &args, int sms, Ctrl *ctrl, cudaStream_t s) {
    CountArgs a = args;
    const int64_t runs = ceil_div(a.nB, kDealRun);
    a.mult = column_deal_mult(runs);
    // floor(2^64 / runs); one run only ever asks for 0 mod 1
    a.inv = runs > 1 ? (unsigned long long)(((unsigned __int128)1 << 64) / (unsigned __int128)runs) : 0;
    // eight warps a CTA; at least four CTAs per SM before a warp takes more
    a.cols = kDealRun;
    while (a.cols < 32 && ceil_div(a.nB, 8 * a.cols) > 4 * (int64_t)sms) a.cols *= 2;
    const int g = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(a.nB, 8 * a.cols), 16 * (int64_t)sms));
    k_count_bin<<<g, kCountThreads, 0, s>>>(a, ctrl);
    return cudaGetLastError();
}

int64_t column_deal_mult(int64_t n) {
    if (n <= 2) return 1;
    auto gcd = [](int64_t a, int64_t b) {
        while (b) {
            const int64_t r = a % b;
            a = b;
            b = r;
        }
        return a;
    };
    int64_t m = (int64_t)((double)n * 0.6180339887498949);
    if (m < 1) m = 1;
    while (gcd(m, n) != 1) ++m;
    return m % n == 0 ? 1 : m;
}

// Single pass: slot capacity min(Op_j, rows) of every column, written to
// caps[j] (caps = the slot offsets + 1, scanned afterwards).
__global__ void k_slot_caps(const int64_t *__restrict__ op, int64_t nB, int64_t mrows, int64_t *__restrict__ caps) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < nB; j += (int64_t)gridDim.x * blockDim.x) {
        const int64_t v = op[j];
        caps[j] = v < mrows ? v : mrows;
    }
}

// Single pass: every entry of C from its column's slot to its place in C.
// The positions of C are cut into tiles of kCopyTile entries, each copied by
// one CTA with coalesced stores, so a column of any length is spread over
// as many CTAs as its tiles (a warp per column left the longest columns of
// a power-law matrix to single warps).  k_tile_cols records the column
// holding each tile's first position; k_tile_copy then takes the tile's
// columns 256 at a time (their first positions and slot offsets staged in
// shared memory), and every thread finds its positions' columns by a binary
// search there.
constexpr int64_t kCopyTile = 4096;
constexpr int kCopyThreads = 256;

__global__ void k_tile_cols(int64_t nB, const int64_t *__restrict__ Ccp, int32_t *__restrict__ tile_col) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < nB; j += (int64_t)gridDim.x * blockDim.x) {
        const int64_t c0 = Ccp[j], c1 = Ccp[j + 1];
        for (int64_t k = (c0 + kCopyTile - 1) / kCopyTile; k * kCopyTile < c1; ++k) tile_col[k] = (int32_t)j;
    }
}

template <typename W>
__global__ void __launch_bounds__(kCopyThreads) k_tile_copy(int64_t nB, int64_t nnzC, const int64_t *__restrict__ Ccp,
                                                           const int64_t *__restrict__ soff,
                                                           const int32_t *__restrict__ tile_col,
                                                           const int32_t *__restrict__ srow,
                                                           const W *__restrict__ sval, int32_t *__restrict__ Crow,
                                                           W *__restrict__ Cval) {
    __shared__ int64_t s_c[kCopyThreads + 1];  // first positions in C of the group's columns, then its end
    __shared__ int64_t s_s[kCopyThreads + 1];  // their slot offsets (slot of column i: [s_s[i], s_s[i + 1]))
    for (int64_t k = blockIdx.x; k * kCopyTile < nnzC; k += gridDim.x) {
        const int64_t p_lo = k * kCopyTile;
        const int64_t p_hi = p_lo + kCopyTile < nnzC ? p_lo + kCopyTile : nnzC;
        int64_t jg = tile_col[k];
        for (;;) {
            const int G = (int)(nB - jg < kCopyThreads ? nB - jg : kCopyThreads);
            if (threadIdx.x < G) {
                s_c[threadIdx.x] = Ccp[jg + threadIdx.x];
                s_s[threadIdx.x] = soff[jg + threadIdx.x];
            }
            if (threadIdx.x == 0) {  // the group's end (jg + G <= nB)
                s_c[G] = Ccp[jg + G];
                s_s[G] = soff[jg + G];
            }
            __syncthreads();
            const int64_t g_lo = p_lo > s_c[0] ? p_lo : s_c[0];
            const int64_t g_hi = p_hi < s_c[G] ? p_hi : s_c[G];
            // every position of the tile in the group's first column (a long
            // column): no search
            const bool one = G == 1 || s_c[1] >= g_hi;
            for (int64_t p0 = g_lo; p0 < g_hi; p0 += 4 * kCopyThreads) {
                int32_t r[4];
                W v[4];
                int64_t dst[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int64_t p = p0 + u * kCopyThreads + threadIdx.x;
                    dst[u] = -1;
                    if (p < g_hi) {
                        // the last column starting at or before p (s_c[0] <= p < s_c[G]): it holds p
                        int lo = 0, hi = one ? 0 : G - 1;
                        while (lo < hi) {
                            const int mid = (lo + hi + 1) >> 1;
                            if (s_c[mid] <= p) lo = mid; else hi = mid - 1;
                        }
                        const int64_t off = p - s_c[lo];
                        // a count never exceeds its slot; reads stay inside the slots
                        if (off < s_s[lo + 1] - s_s[lo]) {
                            r[u] = srow[s_s[lo] + off];
                            v[u] = sval[s_s[lo] + off];
                            dst[u] = p;
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (dst[u] >= 0) {
                        Crow[dst[u]] = r[u];
                        Cval[dst[u]] = v[u];
                    }
            }
            const bool more = s_c[G] < p_hi;  // uniform over the CTA
            __syncthreads();
            if (!more) break;
            jg += G;
        }
    }
}

cudaError_t launch_slot_copy(int64_t nB, int64_t nnzC, const int64_t *Ccp, const int64_t *soff, int32_t *tile_col,
                             const int32_t *srow, const void *sval, int32_t *Crow, void *Cval, int w, int sms,
                             cudaStream_t s) {
    if (nB <= 0 || nnzC <= 0) return cudaSuccess;
    const int gc = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(nB, 256), 8 * (int64_t)sms));
    k_tile_cols<<<gc, 256, 0, s>>>(nB, Ccp, tile_col);
    const int g = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(nnzC, kCopyTile), 8 * (int64_t)sms));
    if (w == 8)
        k_tile_copy<uint64_t><<<g, kCopyThreads, 0, s>>>(nB, nnzC, Ccp, soff, tile_col, srow,
                                                         static_cast<const uint64_t *>(sval), Crow,
                                                         static_cast<uint64_t *>(Cval));
    else
        k_tile_copy<uint32_t><<<g, kCopyThreads, 0, s>>>(nB, nnzC, Ccp, soff, tile_col, srow,
                                                         static_cast<const uint32_t *>(sval), Crow,
                                                         static_cast<uint32_t *>(Cval));
    return cudaGetLastError();
}

int64_t copy_tile_count(int64_t n) { return n / kCopyTile + 2; }

// Column ids into per-bin lists, the dense bin's by class (see next_dense).  A
// block lists its columns in ascending order and reserves its slots with one
// global atomic per list, so a list ascends within a block's tile and roughly
// over them.  The lists start at the running sums of their counts, taken from
// the control block, so nothing of it waits for the host; block 0 then writes
// the control block to the host's mirror (the host reads its counts and
// errors, not the scatter cursors this kernel moves).
constexpr int kScatterThreads = 256;
constexpr int kScatterItems = 4;  // columns per thread: fewer blocks on the lists' cursors
constexpr int kScatterLists = NBINS + 32;  // a bin, or NBINS + a class of the dense bin
constexpr int kScatterParts = kScatterItems * kScatterThreads / 32;

__global__ void __launch_bounds__(kScatterThreads) k_bin_scatter(const int64_t *__restrict__ op, int64_t nB,
                                                                int64_t tcfg, int64_t hmax, int promote, int64_t mA,
                                                                int32_t *__restrict__ bin_cols, Ctrl *ctrl,
                                                                unsigned char *host) {
    // columns of each list in the warps' parts of the tile, then before them
    __shared__ unsigned int s_cnt[kScatterParts][kScatterLists];
    __shared__ unsigned long long s_base[kScatterLists];
    if (host && blockIdx.x == 0)
        for (int i = threadIdx.x; i < (int)(sizeof(Ctrl) / 8); i += kScatterThreads)
            reinterpret_cast<unsigned long long *>(host)[i] = reinterpret_cast<const unsigned long long *>(ctrl)[i];
    if (ctrl->err || !bin_cols) return;  // Op is not there for a malformed product
    for (int i = threadIdx.x; i < kScatterParts * kScatterLists; i += kScatterThreads) (&s_cnt[0][0])[i] = 0u;
    __syncthreads();
    const int64_t t = effective_t(tcfg, hmax, row_rule((int64_t)ctrl->mrows, mA).m);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t j0 = (int64_t)blockIdx.x * (kScatterThreads * kScatterItems) + threadIdx.x;
    int b[kScatterItems];
    unsigned r[kScatterItems];
#pragma unroll
    for (int u = 0; u < kScatterItems; ++u) {
        const int64_t j = j0 + u * kScatterThreads;
        const int64_t o = j < nB ? op[j] : 0;
        b[u] = bin_of(o, t, hmax, promote);
        if (b[u] == BIN_DENSE) b[u] = NBINS + op_class(o);
        r[u] = 0;
    }
#pragma unroll
    for (int u = 0; u < kScatterItems; ++u) {
        unsigned pending = __ballot_sync(0xffffffffu, b[u] != BIN_EMPTY);
        while (pending) {
            const int bb = __shfl_sync(0xffffffffu, b[u], __ffs(pending) - 1);
            const unsigned m = __ballot_sync(0xffffffffu, b[u] == bb);
            if (b[u] == bb) r[u] = __popc(m & ((1u << lane) - 1u));
            if (lane == 0) s_cnt[u * (kScatterThreads / 32) + warp][bb] = __popc(m);
            pending &= ~m;
        }
    }
    __syncthreads();
    if (threadIdx.x < kScatterLists) {
        const int l = threadIdx.x;
        unsigned n = 0;
        for (int p = 0; p < kScatterParts; ++p) {
            const unsigned c = s_cnt[p][l];
            s_cnt[p][l] = n;
            n += c;
        }
        if (n) {
            // the lists of the bins before, and of the heavier classes
            unsigned long long off = 0;
            for (int i = BIN_EMPTY + 1; i < (l < NBINS ? l : BIN_DENSE); ++i) off += ctrl->hist[i];
            for (int c = 31; l >= NBINS && c > l - NBINS; --c) off += ctrl->cls[c];
            unsigned long long *fill = l < NBINS ? &ctrl->fill[l] : &ctrl->clsfill[l - NBINS];
            s_base[l] = off + atomicAdd(fill, (unsigned long long)n);
        }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kScatterItems; ++u)
        if (b[u] != BIN_EMPTY)
            bin_cols[s_base[b[u]] + s_cnt[u * (kScatterThreads / 32) + warp][b[u]] + r[u]] =
                (int32_t)(j0 + u * kScatterThreads);
}

cudaError_t launch_bin_scatter(const CountArgs &a, int32_t *bin_cols, Ctrl *ctrl, unsigned char *host,
                               cudaStream_t s) {
    static_assert(sizeof(Ctrl) % 8 == 0, "the control block is copied in 8-byte words");
    const int64_t g = bin_cols ? std::max<int64_t>(1, ceil_div(a.nB, kScatterThreads * kScatterItems)) : 1;
    k_bin_scatter<<<(unsigned)g, kScatterThreads, 0, s>>>(a.op, a.nB, a.t, a.hmax, a.promote, a.mA, bin_cols,
                                                          ctrl, host);
    return cudaGetLastError();
}

// ----------------------------------------------------------- int64 scan
// Inclusive scan of x[0..n) in place, in three passes over tiles of
// kScanTile elements: tile sums, a scan of the tile sums, the tiles.
constexpr int kScanThreads = 512;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ __forceinline__ int64_t block_incl_scan_i64(int64_t v, int64_t *s_warp, int64_t &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        int64_t o = __shfl_up_sync(0xffffffffu, v, d);
        if (lane >= d) v += o;
    }
    if (lane == 31) s_warp[warp] = v;
    __syncthreads();
    if (warp == 0) {
        int64_t w = lane < nw ? s_warp[lane] : 0;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            int64_t o = __shfl_up_sync(0xffffffffu, w, d);
            if (lane >= d) w += o;
        }
        if (lane < nw) s_warp[lane] = w;
    }
    __syncthreads();
    total = s_warp[nw - 1];
    int64_t r = v + (warp > 0 ? s_warp[warp - 1] : 0);
    __syncthreads();
    return r;
}

__global__ void k_scan_tiles(const int64_t *__restrict__ x, int64_t n, int64_t *__restrict__ sums) {
    __shared__ int64_t s_warp[32];
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    int64_t s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        int64_t e = base + (int64_t)i * kScanThreads + threadIdx.x;
        if (e < n) s += x[e];
    }
    int64_t total;
    block_incl_scan_i64(s, s_warp, total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__global__ void k_scan_sums(int64_t *sums, int64_t ntiles) {
    __shared__ int64_t s_warp[32];
    int64_t carry = 0;
    for (int64_t base = 0; base < ntiles; base += blockDim.x) {
        int64_t e = base + threadIdx.x;
        int64_t v = e < ntiles ? sums[e] : 0;
        int64_t total;
        int64_t incl = block_incl_scan_i64(v, s_warp, total);
        if (e < ntiles) sums[e] = carry + incl - v;  // exclusive
        carry += total;
    }
}

// summed: sums holds the exclusive prefix of the tiles' sums, else the sums
// themselves, which the CTA adds up to its own tile (one launch fewer, for as
// many tiles as kScanDirect).  With `host`, the last tile's CTA writes the
// scan's last value and the control block to the host's mirror.
constexpr int64_t kScanDirect = 4096;

__global__ void __launch_bounds__(kScanThreads) k_scan_apply(int64_t *__restrict__ x, int64_t n,
                                                            const int64_t *__restrict__ sums, int summed,
                                                            const Ctrl *ctrl, unsigned char *host) {
    __shared__ int64_t s_warp[32];
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    int64_t v[kScanItems];
    int64_t s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        int64_t e = base + i;
        v[i] = e < n ? x[e] : 0;
        s += v[i];
    }
    int64_t before = 0;
    if (summed) {
        before = sums[blockIdx.x];
    } else if (blockIdx.x > 0) {  // uniform over the CTA
        int64_t part = 0;
        for (int64_t i = threadIdx.x; i < blockIdx.x; i += kScanThreads) part += sums[i];
        block_incl_scan_i64(part, s_warp, before);
    }
    int64_t total;
    int64_t incl = block_incl_scan_i64(s, s_warp, total);
    int64_t run = before + incl - s;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        int64_t e = base + i;
        run += v[i];
        if (e < n) x[e] = run;
    }
    if (host && blockIdx.x + 1 == gridDim.x) {
        if (threadIdx.x == 0) *reinterpret_cast<int64_t *>(host) = before + total;
        for (int i = threadIdx.x; i < (int)(sizeof(Ctrl) / 8); i += kScanThreads)
            reinterpret_cast<unsigned long long *>(host)[1 + i] = reinterpret_cast<const unsigned long long *>(ctrl)[i];
    }
}

int scan_launches(int64_t n) {
    const int64_t ntiles = scan_tile_count(n);
    return n <= 0 ? 0 : ntiles == 1 ? 1 : ntiles <= kScanDirect ? 2 : 3;
}

cudaError_t launch_inclusive_scan(int64_t *x, int64_t n, int64_t *tile_sums, cudaStream_t s, const Ctrl *ctrl,
                                  unsigned char *host) {
    if (n <= 0) return cudaSuccess;
    const int64_t ntiles = ceil_div(n, kScanTile);
    const bool summed = ntiles > kScanDirect;
    if (ntiles > 1) k_scan_tiles<<<(unsigned)ntiles, kScanThreads, 0, s>>>(x, n, tile_sums);
    if (summed) k_scan_sums<<<1, 1024, 0, s>>>(tile_sums, ntiles);
    k_scan_apply<<<(unsigned)ntiles, kScanThreads, 0, s>>>(x, n, tile_sums, summed ? 1 : 0, ctrl, host);
    return cudaGetLastError();
}

int64_t scan_tile_count(int64_t n) { return n <= 0 ? 1 : ceil_div(n, kScanTile); }

// ------------------------------------------------------------ readback
namespace {

__global__ void k_readback(const unsigned char *s0, size_t n0, const unsigned char *s1, size_t n1,
                           unsigned char *dst, size_t off1) {
    for (size_t i = threadIdx.x; i < n0; i += blockDim.x) dst[i] = s0[i];
    for (size_t i = threadIdx.x; i < n1; i += blockDim.x) dst[off1 + i] = s1[i];
}

constexpr int kMaxDevices = 64;
thread_local Mirror t_mirror[kMaxDevices];

}  // namespace

Mirror *thread_mirror() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
    return &t_mirror[dev];
}

Mirror::~Mirror() {
    if (host) cudaFreeHost(host);
}

cudaError_t Mirror::reserve(size_t need) {
    if (cap >= need) return cudaSuccess;
    if (host) cudaFreeHost(host);
    host = dev = nullptr;
    cap = 0;
    const size_t want = need > (size_t(64) << 10) ? need : (size_t(64) << 10);
    cudaError_t e = cudaHostAlloc(&host, want, cudaHostAllocMapped);
    if (e != cudaSuccess) {
        host = nullptr;
        return e;
    }
    if ((e = cudaHostGetDevicePointer(&dev, host, 0)) != cudaSuccess) return e;
    cap = want;
    return cudaSuccess;
}

cudaError_t readback(Mirror *mp, void *dst0, const void *src0, size_t n0, void *dst1, const void *src1, size_t n1,
                     cudaStream_t s) {
    cudaError_t e;
    if (!mp && !(mp = thread_mirror())) return cudaErrorInvalidDevice;
    Mirror &m = *mp;
    const size_t off1 = (n0 + 15) & ~size_t(15);
    if ((e = m.reserve(off1 + n1)) != cudaSuccess) return e;
    k_readback<<<1, 256, 0, s>>>(static_cast<const unsigned char *>(src0), n0,
                                 static_cast<const unsigned char *>(src1), n1,
                                 static_cast<unsigned char *>(m.dev), off1);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
    if (n0) std::memcpy(dst0, m.host, n0);
    if (n1) std::memcpy(dst1, static_cast<unsigned char *>(m.host) + off1, n1);
    return cudaSuccess;
}

}  // namespace spg
