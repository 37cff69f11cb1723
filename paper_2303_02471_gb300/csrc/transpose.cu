// CSC transpose: row k of M (m x n) becomes column k of M^T (n x m).  Data
// movement only; the Galerkin product P^T (A P) needs P^T as a CSC operand.
//
// Steps: count the entries of every row (atomics), scan into T's column
// pointers, scatter every entry (e, row r, column j) to a slot of column r
// claimed with an atomic cursor, then sort each output column by j so the
// result is deterministic (registers of a lane up to 8 entries, of a warp up
// to 256, CTA bitonic sort in shared memory up to 16384, in place in global
// memory beyond), and finally gather the values through the permutation.
#include "kernels.cuh"

namespace spg {

namespace {

constexpr int kTrSmemSort = 16384;

// Rows outside [0, m) are skipped by both the count and the scatter.
__global__ void k_tr_count(const int32_t *__restrict__ row, int64_t nnz, int64_t m, unsigned long long *cnt) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz; e += stride) {
        const int32_t r = row[e];
        if (r >= 0 && r < m) atomicAdd(&cnt[r], 1ULL);
    }
}

// kScatterLanes lanes per column, so that a column of a few dozen entries is
// a few rounds of independent atomics instead of a serial chain of them.
constexpr int kScatterLanes = 8;

__global__ void k_tr_scatter(const int64_t *__restrict__ cp, const int32_t *__restrict__ row, int64_t ncols,
                             int64_t m, unsigned long long *cursor, int32_t *__restrict__ Trow,
                             int64_t *__restrict__ Tperm) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x / kScatterLanes;
    const int sl = threadIdx.x & (kScatterLanes - 1);
    for (int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / kScatterLanes; j < ncols; j += stride) {
        const int64_t end = cp[j + 1];
        for (int64_t e = cp[j] + sl; e < end; e += kScatterLanes) {
            const int32_t r = row[e];
            if (r < 0 || r >= m) continue;
            const int64_t pos = (int64_t)atomicAdd(&cursor[r], 1ULL);
            Trow[pos] = (int32_t)j;
            Tperm[pos] = e;
        }
    }
}

// Output columns of at most 256 entries, `per` of them per warp.  A lane sorts
// its own column of up to kLaneSort entries with a sorting network in registers
// (of the smallest size that fits the warp's columns); the whole warp then
// sorts the longer ones one after another.  Grid columns and stencils have
// only columns of a few entries, and a warp per column spent a 256-entry
// network on each: 226 us for the 64000 rows of a 40^3 prolongation.
constexpr int kLaneSort = 8;

template <int N>
__device__ __forceinline__ void lane_sort(int64_t b, int L, int32_t *Trow, int64_t *Tperm) {
    int32_t key[N];
    int64_t val[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        key[i] = i < L ? Trow[b + i] : 0x7fffffff;
        val[i] = i < L ? Tperm[b + i] : 0;
    }
    // odd-even merge sort (Batcher)
#pragma unroll
    for (int p = 1; p < N; p <<= 1)
#pragma unroll
        for (int k = p; k >= 1; k >>= 1)
#pragma unroll
            for (int i = k % p; i + k < N; i += 2 * k)
#pragma unroll
                for (int q = 0; q < k; ++q)
                    if (i + q + k < N && (i + q) / (2 * p) == (i + q + k) / (2 * p))
                        cas_pair(key[i + q], val[i + q], key[i + q + k], val[i + q + k], true);
#pragma unroll
    for (int i = 0; i < N; ++i)
        if (i < L) {
            Trow[b + i] = key[i];
            Tperm[b + i] = val[i];
        }
}

template <int R>
__device__ __forceinline__ void warp_sort(int64_t b, int L, int32_t *Trow, int64_t *Tperm) {
    const int lane = threadIdx.x & 31;
    int32_t key[R];
    int64_t val[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int e = r * 32 + lane;
        key[r] = e < L ? Trow[b + e] : 0x7fffffff;
        val[r] = e < L ? Tperm[b + e] : 0;
    }
    group_bitonic_sort<32, R, int64_t>(0xffffffffu, key, val);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int e = r * 32 + lane;
        if (e < L) {
            Trow[b + e] = key[r];
            Tperm[b + e] = val[r];
        }
    }
}

__global__ void __launch_bounds__(256) k_tr_sort_warp(const int64_t *__restrict__ Tcp, int64_t ncolsT, int per,
                                                     int32_t *Trow, int64_t *Tperm) {
    const int lane = threadIdx.x & 31;
    const int64_t c = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * per + lane;
    int64_t b = 0, len = 0;
    if (lane < per && c < ncolsT) {
        b = Tcp[c];
        len = Tcp[c + 1] - b;
    }
    const int L = len <= 256 ? (int)len : 0;  // longer columns: k_tr_sort_cta
    const int own = L <= kLaneSort ? L : 0;
    const unsigned most = __reduce_max_sync(0xffffffffu, (unsigned)own);
    if (most > 4) lane_sort<8>(b, own, Trow, Tperm);
    else if (most > 2) lane_sort<4>(b, own, Trow, Tperm);
    else if (most > 1) lane_sort<2>(b, own, Trow, Tperm);
    unsigned todo = __ballot_sync(0xffffffffu, L > kLaneSort);
    while (todo) {
        const int s = __ffs(todo) - 1;
        todo &= todo - 1u;
        const int64_t sb = __shfl_sync(0xffffffffu, b, s);
        const int sL = __shfl_sync(0xffffffffu, L, s);
        if (sL <= 32) warp_sort<1>(sb, sL, Trow, Tperm);
        else if (sL <= 64) warp_sort<2>(sb, sL, Trow, Tperm);
        else warp_sort<8>(sb, sL, Trow, Tperm);
    }
}

// One CTA per output column of more than 256 entries: bitonic sort over the
// next power of two, in shared memory when it fits, else in place in `tmp`.
// A CTA looks through blockDim columns at a time, one per thread, dealt over
// the CTAs by index so that neighbouring long columns go to different CTAs;
// where there are none (the common case) one round of loads is all it does.
// Its grid (sort_cta_grid): a CTA per 64 columns, which keeps that round
// short, or a CTA per column that can be long (at most nnz / 257 are) where
// that is more, up to four CTAs per SM, whose share of the long columns is
// even enough (64 rows of 10000 entries: 0.74 ms, one of them alone 0.53,
// all 64 in one CTA 29.8).
__global__ void __launch_bounds__(512) k_tr_sort_cta(const int64_t *__restrict__ Tcp, int64_t ncolsT, int32_t *Trow,
                                                    int64_t *Tperm, int32_t *gkey, int64_t *gval) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int64_t s_col[512];
    __shared__ int s_n;
    for (int64_t c0 = blockIdx.x; c0 < ncolsT; c0 += (int64_t)gridDim.x * blockDim.x) {
        if (threadIdx.x == 0) s_n = 0;
        __syncthreads();
        const int64_t mine = c0 + (int64_t)threadIdx.x * gridDim.x;
        if (mine < ncolsT && Tcp[mine + 1] - Tcp[mine] > 256) s_col[atomicAdd(&s_n, 1)] = mine;
        __syncthreads();
        const int n = s_n;
        for (int at = 0; at < n; ++at) {
            const int64_t c = s_col[at];
            const int64_t b = Tcp[c], L = Tcp[c + 1] - b;
            int64_t N = 1;
            while (N < L) N <<= 1;
            const bool in_smem = N <= kTrSmemSort;
            // beyond shared memory, sort a padded copy in the scratch: column c
            // owns [2 b, 2 b + N) there, inside [2 b, 2 (b + L)) since N < 2 L
            int32_t *key = in_smem ? reinterpret_cast<int32_t *>(smem) : gkey + 2 * b;
            int64_t *val = in_smem ? reinterpret_cast<int64_t *>(smem + (size_t)kTrSmemSort * 4) : gval + 2 * b;
            for (int64_t e = threadIdx.x; e < N; e += blockDim.x) {
                key[e] = e < L ? Trow[b + e] : 0x7fffffff;
                val[e] = e < L ? Tperm[b + e] : 0;
            }
            __syncthreads();
            for (int64_t k = 2; k <= N; k <<= 1) {
                for (int64_t jj = k >> 1; jj > 0; jj >>= 1) {
                    for (int64_t i = threadIdx.x; i < N; i += blockDim.x) {
                        const int64_t l = i ^ jj;
                        if (l > i) {
                            const bool up = (i & k) == 0;
                            const int32_t ki = key[i], kl = key[l];
                            if (up ? ki > kl : ki < kl) {
                                key[i] = kl;
                                key[l] = ki;
                                const int64_t t = val[i];
                                val[i] = val[l];
                                val[l] = t;
                            }
                        }
                    }
                    __syncthreads();
                }
            }
            for (int64_t e = threadIdx.x; e < L; e += blockDim.x) {
                Trow[b + e] = key[e];
                Tperm[b + e] = val[e];
            }
            __syncthreads();
        }
        __syncthreads();
    }
}

// Columns per warp of k_tr_sort_warp: 32 where that gives every warp slot of
// the chip a warp (kSortWarps per SM), else fewer, so that longer columns are
// not left to the few warps of a matrix with few columns.  Whole transposes:
// 64 rows of 200 entries 1018 us with 32 columns per warp, 92 so; 100000 rows
// of 100 1405 and 1184, R-MAT 2^16 773 and 384; the 40^3 prolongation 77 and
// 80, 200000 rows of 3 entries with one of 200 in 64 191 and 219 (a warp per
// column: 1467).
constexpr int kSortWarps = 64;

int sort_warp_columns(int64_t m, int sms) {
    int per = 32;
    while (per > 1 && ceil_div(m, per) < kSortWarps * (int64_t)sms) per >>= 1;
    return per;
}

int sort_cta_grid(int64_t m, int64_t nnz, int sms) {
    const int64_t longest = std::min<int64_t>(m, nnz / 257);
    return (int)std::max<int64_t>(1, std::min<int64_t>(std::max<int64_t>(ceil_div(m, 64), longest), 4 * (int64_t)sms));
}

// T's values through the permutation, for the entries T actually holds.
template <typename VT>
__global__ void k_tr_gather(const int64_t *__restrict__ perm, const int64_t *__restrict__ Tcp, int64_t m,
                            const VT *__restrict__ src, VT *__restrict__ dst) {
    const int64_t n = Tcp[m];
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += stride) dst[e] = src[perm[e]];
}

// dst[i] = src[idx[i]] (gather) or dst[idx[i]] = src[i] (scatter).
template <typename VT>
__global__ void k_permute(const VT *__restrict__ src, const int64_t *__restrict__ idx, VT *__restrict__ dst,
                          int64_t n, int scatter) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        if (scatter) dst[idx[i]] = src[i];
        else dst[i] = src[idx[i]];
    }
}

struct TrLayout {
    size_t cnt = 0, tiles = 0, perm = 0, key = 0, val = 0, total = 0;
};

size_t al256(size_t v) { return (v + 255) & ~size_t(255); }

TrLayout tr_layout(const spg_csc *M) {
    TrLayout L;
    size_t off = 0;
    L.cnt = off; off = al256(off + (size_t)(M->nrows + 1) * 8);
    L.tiles = off; off = al256(off + (size_t)scan_tile_count(M->nrows) * 8);
    L.perm = off; off = al256(off + (size_t)M->nnz * 8);       // permutation when the caller passes none
    L.key = off; off = al256(off + (size_t)M->nnz * 2 * 4 + 64);  // padded sort copies of long columns
    L.val = off; off = al256(off + (size_t)M->nnz * 2 * 8 + 64);
    L.total = off;
    return L;
}

}  // namespace

}  // namespace spg

using namespace spg;

extern "C" {

spg_status spg_transpose_workspace_size(const spg_csc *M, size_t *bytes) {
    if (!M || !bytes || M->nrows < 0 || M->ncols < 0 || M->nnz < 0) return SPG_ERR_INVALID;
    *bytes = tr_layout(M).total;
    return SPG_OK;
}

spg_status spg_csc_transpose(const spg_csc *M, int64_t *T_colptr, int32_t *T_rowidx, void *T_values, int64_t *perm,
                             void *workspace, size_t ws_bytes, spg_stream stream) {
    if (!M || !T_colptr || M->nrows < 0 || M->ncols < 0 || M->nnz < 0 || !M->colptr) return SPG_ERR_INVALID;
    if (M->nrows > INT32_MAX || M->ncols > INT32_MAX) return SPG_ERR_INDEX_OVERFLOW;
    if (M->nnz > 0 && (!M->rowidx || !T_rowidx || (T_values && !M->values))) return SPG_ERR_INVALID;
    if (M->dtype != SPG_F64 && M->dtype != SPG_F32) return SPG_ERR_INVALID;
    const TrLayout L = tr_layout(M);
    if (!workspace || ws_bytes < L.total || (reinterpret_cast<uintptr_t>(workspace) & 255)) return SPG_ERR_WORKSPACE;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    unsigned char *ws = static_cast<unsigned char *>(workspace);
    unsigned long long *cnt = reinterpret_cast<unsigned long long *>(ws + L.cnt);
    int64_t *pm = perm ? perm : reinterpret_cast<int64_t *>(ws + L.perm);
    const int64_t m = M->nrows, nnz = M->nnz;
    if (cudaMemsetAsync(cnt, 0, (size_t)(m + 1) * 8, s) != cudaSuccess) return SPG_ERR_CUDA;
    if (cudaMemsetAsync(T_colptr, 0, sizeof(int64_t), s) != cudaSuccess) return SPG_ERR_CUDA;
    if (nnz > 0) {
        const int g = (int)std::min<int64_t>(ceil_div(nnz, 256), 4096);
        k_tr_count<<<g, 256, 0, s>>>(M->rowidx, nnz, m, cnt);
    }
    if (m > 0) {
        if (cudaMemcpyAsync(T_colptr + 1, cnt, (size_t)m * 8, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
            return SPG_ERR_CUDA;
        if (launch_inclusive_scan(T_colptr + 1, m, reinterpret_cast<int64_t *>(ws + L.tiles), s) != cudaSuccess)
            return SPG_ERR_CUDA;
        // cursors start at the column starts
        if (cudaMemcpyAsync(cnt, T_colptr, (size_t)m * 8, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
            return SPG_ERR_CUDA;
    }
    if (nnz > 0) {
        const int gc = (int)std::min<int64_t>(ceil_div(M->ncols * kScatterLanes, 256), 4096);
        k_tr_scatter<<<gc, 256, 0, s>>>(M->colptr, M->rowidx, M->ncols, m, cnt, T_rowidx, pm);
        int dev = 0, sms = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return SPG_ERR_CUDA;
        const int per = sort_warp_columns(m, sms);
        k_tr_sort_warp<<<(unsigned)ceil_div(m, 8 * per), 256, 0, s>>>(T_colptr, m, per, T_rowidx, pm);
        const size_t smem = (size_t)kTrSmemSort * 12;
        cudaFuncSetAttribute(k_tr_sort_cta, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        k_tr_sort_cta<<<(unsigned)sort_cta_grid(m, nnz, sms), 512, smem, s>>>(
            T_colptr, m, T_rowidx, pm, reinterpret_cast<int32_t *>(ws + L.key),
            reinterpret_cast<int64_t *>(ws + L.val));
        if (T_values) {
            const int gg = (int)std::min<int64_t>(ceil_div(nnz, 256), 4096);
            if (M->dtype == SPG_F64)
                k_tr_gather<double><<<gg, 256, 0, s>>>(pm, T_colptr, m, static_cast<const double *>(M->values),
                                                       static_cast<double *>(T_values));
            else
                k_tr_gather<float><<<gg, 256, 0, s>>>(pm, T_colptr, m, static_cast<const float *>(M->values),
                                                      static_cast<float *>(T_values));
        }
    }
    return cudaGetLastError() == cudaSuccess ? SPG_OK : SPG_ERR_CUDA;
}

spg_status spg_permute_values(const void *src, const int64_t *idx, void *dst, int64_t n, int32_t dtype,
                              int32_t scatter, spg_stream stream) {
    if (n < 0 || (dtype != SPG_F64 && dtype != SPG_F32)) return SPG_ERR_INVALID;
    if (n == 0) return SPG_OK;
    if (!src || !idx || !dst) return SPG_ERR_INVALID;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int g = (int)std::min<int64_t>(ceil_div(n, 256), 8192);
    if (dtype == SPG_F64)
        k_permute<double><<<g, 256, 0, s>>>(static_cast<const double *>(src), idx, static_cast<double *>(dst), n,
                                            scatter);
    else
        k_permute<float><<<g, 256, 0, s>>>(static_cast<const float *>(src), idx, static_cast<float *>(dst), n,
                                           scatter);
    return cudaGetLastError() == cudaSuccess ? SPG_OK : SPG_ERR_CUDA;
}

}  // extern "C"
