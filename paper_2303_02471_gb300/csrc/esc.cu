// ESC accumulator (Expand, Sort, Compress; Section 4) for the light columns
// of C = A x B: the lane-group bins, Op_j <= 256.
//
// G lanes (G = min(32, the bin's largest Op_j)) hold a column's products in
// registers, R = opmax / G of them per lane, so a warp works 32 / G columns at
// a time:
//   Expand    lane l loads the column's B entry l and the place of its A
//             column; product q of the column is gathered by lane q mod G,
//             whose owner entry comes from an OR-reduced mask of the entries'
//             first products;
//   Sort      a bitonic network over the G R keys (row, q): each is one word,
//             distinct, and in the order a stable sort of the rows gives, and
//             only the word moves (one shuffle and one min or max per lane and
//             stage).  The network's mirrored form needs no directions;
//   Compress  equal rows are neighbours: the first of each run writes one
//             entry of C at its column's pointer plus its rank among the
//             column's runs, with the run's sum.  Where a warp's columns repeat
//             no row (the common case of very sparse products) the sorted
//             products are the column.
// The sums do not depend on timing (no atomics on values).
//
// What bounds it: instruction issue.  The form before this one expanded tiles
// of 256 products into shared memory and counted each product's place among
// its column's keys there (bins of <= 64) or radix sorted the tile: 13.8 warp
// instructions per product; for the very sparse product of 2^20 columns (21 M
// products, double) it took 0.50 ms for the values and 0.26 ms to count, this
// one 0.44 and 0.23 ms (10.8 warp instructions per product), and 6 instead of
// 14 us for a bin of a few columns.  The gathers'
// latency comes next: it is covered by the warps in flight and by loading the
// next columns' entries and products while the present ones are sorted.
//
// Modes: with values and no count output it is the numeric phase (C's
// column pointers come from the symbolic phase; a column whose run count
// differs is reported); without values it counts the runs of each column
// into cnt_out[j + 1] (the symbolic phase); with values and a count output it
// writes each column at base[j] and its count into cnt_out[j + 1] (the
// single-pass form, where base holds slots sized by Op_j).
//
// Keys are 32-bit words where (row, place in the column) fits (2^24 rows in
// the bin of 256 products, 2^29 in that of 8) and A and B have fewer than 2^31
// entries, else 64-bit.
#include "columns.cuh"
#include "esc.cuh"

namespace spg {

// A warp takes up to esc_steps steps of 32 / G columns at a time from the
// bin's list (a tile; at least kEscAhead steps where it takes several tiles,
// as the loads run that far ahead).
constexpr int kEscAhead = 3;
template <int N>
constexpr int esc_steps() {
    return N <= 32 ? 8 : 4;
}

constexpr int esc_log2(int n) { return n <= 1 ? 0 : 1 + esc_log2(n / 2); }

template <typename KT>
__device__ __forceinline__ KT esc_min(KT a, KT b) { return min(a, b); }
template <typename KT>
__device__ __forceinline__ KT esc_max(KT a, KT b) { return max(a, b); }
template <typename KT>
__device__ __forceinline__ KT esc_pick(KT a, KT b, bool upper) {
    return (a < b) != upper ? a : b;
}

// The index type that goes with a key type: 32-bit keys are used with 32-bit
// positions in A and B (fewer shuffles, address words and registers).
template <typename KT>
struct EscIndex {
    using type = int64_t;
};
template <>
struct EscIndex<uint32_t> {
    using type = int32_t;
};
// Value i of an int64 pointer array, known to fit IT.
template <typename IT>
__device__ __forceinline__ IT esc_ptr(const int64_t *cp, int64_t i) {
    if constexpr (sizeof(IT) == 4) return reinterpret_cast<const int32_t *>(cp)[2 * i];  // little-endian low word
    else return cp[i];
}

// Ascending sort of G * R distinct keys, element r * G + (lane of the group)
// in key[r].  Bitonic network in mirrored form: merging runs of k / 2 starts
// by comparing element e with e ^ (k - 1), then e with e ^ j; the lower
// element always keeps the smaller key.
template <int G, int R, typename KT>
__device__ __forceinline__ void esc_sort(KT (&key)[R]) {
    const int lane = threadIdx.x & 31;
    auto exchange = [&](int x, bool upper) {  // with the lane ^ x, in place
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const KT o = __shfl_xor_sync(0xffffffffu, key[r], x);
            key[r] = esc_pick(key[r], o, upper);
        }
    };
#pragma unroll
    for (int k = 2; k <= G * R; k <<= 1) {
        if (k <= G) {
            exchange(k - 1, (lane & (k >> 1)) != 0);
        } else {  // mirrored over registers and lanes
            const int rm = k / G - 1;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if ((r ^ rm) < r) continue;
                const KT lo = key[r], hi = key[r ^ rm];
                key[r] = esc_min(lo, __shfl_xor_sync(0xffffffffu, hi, G - 1));
                key[r ^ rm] = esc_max(hi, __shfl_xor_sync(0xffffffffu, lo, G - 1));
            }
        }
#pragma unroll
        for (int j = k >> 2; j > 0; j >>= 1) {
            if (j >= G) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    if (r & (j / G)) continue;
                    const KT lo = key[r], hi = key[r | (j / G)];
                    key[r] = esc_min(lo, hi);
                    key[r | (j / G)] = esc_max(lo, hi);
                }
            } else {
                exchange(j, (lane & j) != 0);
            }
        }
    }
}

// Shared memory of a warp with more than one product per lane: the values by
// place, and the sorted keys when rows repeat.
template <int N, typename VT, typename KT>
struct EscWarp {
    VT val[N];
    KT key[N];
};

// Counting uses a filter of hashed rows in the bins of up to 64 products (see
// the kernel): 2^13 bits a warp, so that 38 distinct rows, the average of the
// bin of 64 in a very sparse product, collide in one column of eleven.
constexpr int kEscFilterBits = 13;
template <int N, bool VALS>
constexpr bool esc_filter() {
    return !VALS && N <= 64;
}

template <int N, bool VALS, typename VT, typename KT>
__host__ __device__ constexpr size_t esc_warp_bytes() {
    return VALS && N > 32         ? (sizeof(EscWarp<N, VT, KT>) + 15) & ~size_t(15)
           : esc_filter<N, VALS>() ? size_t(1) << (kEscFilterBits - 3)
                                   : 0;
}

// CTAs per SM the kernels are built for (registers).
template <int N, bool VALS, typename VT, typename KT>
constexpr int esc_min_blocks() {
    return sizeof(KT) == 8 || (N == 256 && VALS && sizeof(VT) == 8) ? 3 : VALS || N >= 64 ? 4 : N == 32 ? 5 : 6;
}

template <int N, bool VALS, typename VT, typename KT>
__global__ void __launch_bounds__(kEscWarps * 32, (esc_min_blocks<N, VALS, VT, KT>()))
    k_esc(BinTask t, Operands o, const int64_t *base, int64_t *cnt_out, int32_t *Crow, VT *Cval, int steps) {
    using IT = typename EscIndex<KT>::type;
    constexpr int G = N < 32 ? N : 32, R = N / G, S = 32 / G, L = esc_log2(N);
    // the next step's products are gathered while a step is sorted (more
    // products per lane keep enough loads in flight by themselves)
    constexpr bool AHEAD = R <= 2;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned long long s_max, s_sum;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gl = lane & (G - 1), gb = lane & ~(G - 1);
    const unsigned gm = G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u) << gb;
    const unsigned upto = gm & (lane == 31 ? 0xffffffffu : (2u << lane) - 1u);
    const unsigned below = gm & ((1u << lane) - 1u);
    [[maybe_unused]] EscWarp<N, VT, KT> *W =
        reinterpret_cast<EscWarp<N, VT, KT> *>(smem + warp * esc_warp_bytes<N, VALS, VT, KT>());
    if (threadIdx.x == 0) s_max = s_sum = 0;
    __syncthreads();
    const TOps<VT> ops = typed<VT>(o);
    const uint64_t pol = keep_policy();
    int my_max = 0;  // of a column's runs; their sum
    unsigned long long my_sum = 0;
    constexpr bool FILTER = esc_filter<N, VALS>();
    [[maybe_unused]] uint32_t *filter = reinterpret_cast<uint32_t *>(smem) + warp * (1 << (kEscFilterBits - 5));
    [[maybe_unused]] bool repeated = false;
    if constexpr (FILTER) {
        for (int i = lane; i < 1 << (kEscFilterBits - 5); i += 32) filter[i] = 0u;
        __syncwarp();
    }
    const int ct = S * steps;
    const int64_t ntiles = ceil_div(t.count, (int64_t)ct);
    const int64_t tstride = (int64_t)gridDim.x * kEscWarps;
    int64_t tile = (int64_t)blockIdx.x * kEscWarps + warp;

    // a tile's columns, one per lane: B's entries and C's place
    struct Tile {
        int32_t j;
        IT p0;
        int nb;
        int ccap;  // entries the column's place holds
        int64_t cb;
    };
    auto fetch = [&](int64_t tl) -> Tile {
        Tile x{0, 0, 0, 0, 0};
        const int64_t f = tl * ct + lane;
        if (tl < ntiles && lane < ct && f < t.count) {
            x.j = t.cols[f];
            x.p0 = esc_ptr<IT>(ops.Bcp, x.j);
            x.nb = (int)(esc_ptr<IT>(ops.Bcp, x.j + 1) - x.p0);
            if (VALS) {
                x.cb = base[x.j];
                x.ccap = (int)(base[x.j + 1] - x.cb);
            }
        }
        return x;
    };
    Tile cur = fetch(tile), nxt = fetch(tile + tstride);
    // A step's loads, each made a step before the next one needs it: a lane's
    // B entry (its row, hence A's column), that column's place and length and
    // B_kj, the products.  Steps from `steps` on are the next tile's.
    struct Row {
        int32_t k;
        IT p;
        int nb;
    };
    struct Entry {
        IT a0;
        int z, nb;
        VT b;
    };
    struct Products {
        int32_t row[R];
        VT a[R], b[R];
        int n;
    };
    auto row_of = [&](int s) -> Row {
        const bool now = s < steps;
        const int c = ((now ? s : s - steps) * S + lane / G) & 31;
        const IT p = __shfl_sync(0xffffffffu, now ? cur.p0 : nxt.p0, c) + gl;
        const int nb = __shfl_sync(0xffffffffu, now ? cur.nb : nxt.nb, c);
        return Row{gl < nb ? ops.Brow[p] : -1, p, nb};
    };
    auto entry_of = [&](const Row &r) -> Entry {
        Entry e{0, 0, r.nb, VT(0)};
        if (r.k >= 0) {
            e.a0 = esc_ptr<IT>(ops.Acp, r.k);
            // more than the bin holds (the pattern changed since planning)
            // is enough to fail the count
            const IT z = esc_ptr<IT>(ops.Acp, (int64_t)r.k + 1) - e.a0;
            e.z = z <= N ? (int)z : N + 1;
            if (VALS) e.b = ops.Bval[r.p];
        }
        return e;
    };
    auto products_of = [&](int s, Entry ent) -> Products {
        Products x;
        const int nb = ent.nb;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            x.row[r] = 0;
            x.a[r] = x.b[r] = VT(0);
        }
        x.n = 0;  // the column's products so far
        for (int e0 = 0;; e0 += G) {
            const int z = ent.z;
            int zi = z;
#pragma unroll
            for (int d = 1; d < G; d <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, zi, d, G);
                if (gl >= d) zi += v;
            }
            const int total = __shfl_sync(0xffffffffu, zi, G - 1, G);
            const int start = x.n + zi - z;  // the entry's first product
            const IT ab = ent.a0 - start;    // product q is A's entry ab + q
            // entries without products break the count of the masks' bits
            const bool plain = __all_sync(0xffffffffu, z > 0 || e0 + gl >= nb);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                // windows of R > 1 that the chunk does not reach (uniform)
                if (R > 1 && !(x.n < (r + 1) * G && x.n + total > r * G)) continue;
                const int q = r * G + gl;
                int own;
                if (plain) {
                    const int at = start - r * G;
                    const unsigned bits =
                        __reduce_or_sync(0xffffffffu, z > 0 && at >= 0 && at < G ? 1u << (gb + at) : 0u);
                    own = gb + __popc(bits & upto) - 1;
                    if (R > 1) own += __popc(__ballot_sync(0xffffffffu, z > 0 && at < 0));
                } else {  // the group's last entry starting at or before q
                    own = gb;
#pragma unroll
                    for (int step = G / 2; step > 0; step >>= 1)
                        if (__shfl_sync(0xffffffffu, start, (own + step) & 31) <= q) own += step;
                }
                const IT qa = __shfl_sync(0xffffffffu, ab, own & 31) + q;
                VT b = VT(0);
                if (VALS) b = __shfl_sync(0xffffffffu, ent.b, own & 31);
                if (q >= x.n && q < x.n + total) {
                    x.row[r] = ld_keep(ops.Arow + qa, pol);
                    if (VALS) {
                        x.a[r] = ld_keep(ops.Aval + qa, pol);
                        x.b[r] = b;
                    }
                }
            }
            x.n = x.n + total <= N ? x.n + total : N + 1;
            if (!__any_sync(0xffffffffu, e0 + G < nb)) break;
            const bool now = s < steps;
            const int c = ((now ? s : s - steps) * S + lane / G) & 31;
            const int en = e0 + G + gl;
            const IT p = __shfl_sync(0xffffffffu, now ? cur.p0 : nxt.p0, c) + en;
            ent = entry_of(Row{en < nb ? ops.Brow[p] : -1, p, nb});
        }
        return x;
    };

    Row rn = row_of(0);
    Entry en = entry_of(rn);
    rn = row_of(1);
    Products pr;
    if constexpr (AHEAD) {
        pr = products_of(0, en);
        en = entry_of(rn);
        rn = row_of(2);
    }
    for (; tile < ntiles; tile += tstride) {
        const int64_t first = tile * ct;
        const int nc = (int)(t.count - first < ct ? t.count - first : ct);
        for (int s = 0; s < steps; ++s) {
            // ---- expand
            Products now;
            if constexpr (AHEAD) {
                now = pr;
                pr = products_of(s + 1, en);
                en = entry_of(rn);
                rn = row_of(s + 3);
            } else {
                now = products_of(s, en);
                en = entry_of(rn);
                rn = row_of(s + 2);
            }
            const int c = s * S + lane / G;
            const int n = now.n;
            // more products than the bin holds (the pattern changed since
            // planning) fail the count below
            const int nn = n < N ? n : N;
            int runs = 0;
            // Counting columns whose rows all differ needs no sort: the rows'
            // hashed bits are set in the warp's filter, and where no bit was
            // set before, no row repeats.  Not tried after a step that did
            // repeat rows (a structured matrix repeats them in every column).
            bool sorted = true;
            if constexpr (FILTER) {
                if (!repeated) {  // uniform over the warp
                    bool hit = false;
                    unsigned h[R];
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const int q = r * G + gl;
                        h[r] = (((unsigned)now.row[r] * S + (unsigned)(lane / G)) * 2654435761u) >> (32 - kEscFilterBits);
                        const unsigned bit = 1u << (h[r] & 31);
                        if (q < nn) hit |= (atomicOr(&filter[h[r] >> 5], bit) & bit) != 0;
                    }
                    sorted = __any_sync(0xffffffffu, hit);
#pragma unroll
                    for (int r = 0; r < R; ++r)
                        if (r * G + gl < nn) filter[h[r] >> 5] = 0u;
                    __syncwarp();
                    runs = nn;
                }
            }
            if (sorted) {
                runs = 0;
                KT key[R];
                VT val[R];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int q = r * G + gl;
                    key[r] = q < n ? ((KT)(uint32_t)now.row[r] << L) | (KT)q : ~KT(0);
                    val[r] = VALS ? now.a[r] * now.b[r] : VT(0);
                }
                if constexpr (VALS && R > 1) {
                    __syncwarp();  // the last step's reads are done
#pragma unroll
                    for (int r = 0; r < R; ++r) W->val[r * G + lane] = val[r];
                    __syncwarp();
                }
                // ---- sort
                esc_sort<G, R, KT>(key);
                // ---- compress: the first element of each run of equal rows
                unsigned heads[R];
                bool head[R];
                bool again = false;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int e = r * G + gl;
                    KT prev = __shfl_up_sync(0xffffffffu, key[r], 1, G);
                    if (R > 1 && r > 0) {
                        const KT last = __shfl_sync(0xffffffffu, key[r - 1], G - 1);
                        if (gl == 0) prev = last;
                    }
                    head[r] = e < nn && (e == 0 || (prev >> L) != (key[r] >> L));
                    heads[r] = __ballot_sync(0xffffffffu, head[r]);
                    again |= e < nn && !head[r];
                    runs += __popc(heads[r] & gm);
                }
                if constexpr (FILTER) repeated = __any_sync(0xffffffffu, again);
                if constexpr (VALS) {
                    const int64_t cbase = __shfl_sync(0xffffffffu, cur.cb, c);
                    const int cap = __shfl_sync(0xffffffffu, cur.ccap, c);
                    const bool repeats = __any_sync(0xffffffffu, again);
                    VT sum[R];
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const int src = (int)(key[r] & (KT)(N - 1));
                        if constexpr (R == 1) sum[r] = __shfl_sync(0xffffffffu, val[r], gb + src);
                        else sum[r] = W->val[src];
                    }
                    if (repeats) {
                        if constexpr (R == 1) {
                            // the rest of the run one after another, in sorted order
                            const VT own = sum[0];
                            for (int d = 1; d < G; ++d) {
                                const VT v = __shfl_down_sync(0xffffffffu, own, d, G);
                                const KT k = __shfl_down_sync(0xffffffffu, key[0], d, G);
                                const bool on = gl + d < nn && (k >> L) == (key[0] >> L);
                                if (!__any_sync(0xffffffffu, on)) break;
                                if (on) sum[0] += v;
                            }
                        } else {
#pragma unroll
                            for (int r = 0; r < R; ++r) W->key[r * G + lane] = key[r];
                            __syncwarp();
#pragma unroll
                            for (int r = 0; r < R; ++r)
                                if (head[r])
                                    for (int e = r * G + lane + 1; e < nn && (W->key[e] >> L) == (key[r] >> L); ++e)
                                        sum[r] += W->val[(int)(W->key[e] & (KT)(N - 1))];
                        }
                    }
                    int rank = 0;
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const int at = rank + __popc(heads[r] & below);
                        // a column with more runs than its place holds is reported
                        // below and not written past its place
                        if (head[r] && at < cap) {
                            Crow[cbase + at] = ops.crow((int32_t)(key[r] >> L));
                            Cval[cbase + at] = sum[r];
                        }
                        rank += __popc(heads[r] & gm);
                    }
                    if (!cnt_out && c < nc && gl == 0 && (runs != cap || n > N))
                        set_error(t.ctrl, SPG_ERR_INVALID, kDetailCountMismatch + t.bin, first + c);
                }
            }
            if (cnt_out) {
                const int32_t jc = __shfl_sync(0xffffffffu, cur.j, c);
                if (c < nc && gl == 0) {
                    if (n > N) set_error(t.ctrl, SPG_ERR_INVALID, kDetailCountMismatch + t.bin, jc);
                    cnt_out[jc + 1] = runs;
                    my_max = max(my_max, runs);
                    my_sum += (unsigned long long)runs;
                }
            }
        }
        cur = nxt;
        nxt = fetch(tile + 2 * tstride);
    }
    if (cnt_out) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            my_sum += __shfl_xor_sync(0xffffffffu, my_sum, d);
            my_max = max(my_max, __shfl_xor_sync(0xffffffffu, my_max, d));
        }
        if (lane == 0 && my_sum) {
            atomicMax(&s_max, (unsigned long long)my_max);
            atomicAdd(&s_sum, my_sum);
        }
        __syncthreads();
        if (threadIdx.x == 0 && s_max) {
            atomicMax(&t.ctrl->maxnnz[t.bin], s_max);
            atomicAdd(&t.ctrl->binnnz[t.bin], s_sum);
        }
    }
}

// ------------------------------------------------------------- launches
template <int N, bool VALS, typename VT, typename KT>
static cudaError_t launch_esc_n(const BinTask &t, const Operands &o, const int64_t *base, int64_t *cnt_out,
                                int32_t *Crow, VT *Cval, int sms, cudaStream_t s) {
    auto k = k_esc<N, VALS, VT, KT>;
    const size_t smem = (size_t)kEscWarps * esc_warp_bytes<N, VALS, VT, KT>();
    if (smem > 48 * 1024) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, kEscWarps * 32, smem) != cudaSuccess || occ < 1)
        occ = 1;
    // few columns: as few steps per warp as the warps that fit the chip allow,
    // a tile each
    constexpr int S = 32 / (N < 32 ? N : 32);
    static_assert(esc_steps<N>() >= kEscAhead, "loads run kEscAhead steps ahead, at most into the next tile");
    const int64_t warps = (int64_t)occ * sms * kEscWarps;
    const int steps = (int)std::min<int64_t>(esc_steps<N>(), ceil_div(t.count, S * warps));
    const int64_t ntiles = ceil_div(t.count, (int64_t)S * steps);
    const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(ceil_div(ntiles, kEscWarps), (int64_t)occ * sms));
    k<<<(unsigned)grid, kEscWarps * 32, smem, s>>>(t, o, base, cnt_out, Crow, Cval, steps);
    return cudaGetLastError();
}

template <bool VALS, typename VT, typename KT>
static cudaError_t launch_esc_k(const BinTask &t, const Operands &o, const int64_t *base, int64_t *cnt_out,
                                int32_t *Crow, VT *Cval, int sms, cudaStream_t s) {
    switch (t.bin - BIN_WARP0) {
#define ESC_CASE(b) \
    case b: return launch_esc_n<warp_bin_opmax(b), VALS, VT, KT>(t, o, base, cnt_out, Crow, Cval, sms, s);
        ESC_CASE(0) ESC_CASE(1) ESC_CASE(2) ESC_CASE(3) ESC_CASE(4) ESC_CASE(5)
#undef ESC_CASE
    }
    return cudaErrorInvalidValue;
}

template <bool VALS, typename VT>
static cudaError_t launch_esc_t(const BinTask &t, const Operands &o, const int64_t *base, int64_t *cnt_out,
                                int32_t *Crow, VT *Cval, int sms, cudaStream_t s) {
    if (t.count <= 0) return cudaSuccess;
    // rows below m and places below the bin's opmax in one 32-bit word, and
    // positions in A and B in 31 bits
    const bool narrow = t.m <= ((int64_t)1 << 32) / warp_bin_opmax(t.bin - BIN_WARP0) && o.nnz_max <= INT32_MAX - 32;
    return narrow ? launch_esc_k<VALS, VT, uint32_t>(t, o, base, cnt_out, Crow, Cval, sms, s)
                  : launch_esc_k<VALS, VT, uint64_t>(t, o, base, cnt_out, Crow, Cval, sms, s);
}

cudaError_t launch_esc_bin(const BinTask &t, const Operands &o, const int64_t *base, int64_t *cnt_out,
                           int32_t *Crow, void *Cval, bool values, int dtype, int sms, cudaStream_t s) {
    if (!values) return launch_esc_t<false, float>(t, o, base, cnt_out, nullptr, nullptr, sms, s);
    return dtype == SPG_F64
               ? launch_esc_t<true, double>(t, o, base, cnt_out, Crow, static_cast<double *>(Cval), sms, s)
               : launch_esc_t<true, float>(t, o, base, cnt_out, Crow, static_cast<float *>(Cval), sms, s);
}

}  // namespace spg
