// Construction of pruned quadtrees and forests (Sec. 6, Def. 6.1) in O(N log N) work:
// every structure comes from sorted packed box keys or, for forests of small problems,
// from counts on each problem's dense leaf grid - never from dense maps of a deep level.
//
// A box of problem p at coordinates (x, y) of its level packs into the 64-bit key
// (p << 2 kb) | (y << kb) | x, kb = bits of the deepest leaf level, so a sorted key array
// lists the boxes of each problem row by row.  The builder
//   1. picks the common leaf side (the largest power of two <= max_leaf_side at which no
//      leaf holds more than leaf_size sources or targets): on the problems' dense leaf
//      grids when their cells are few (occupancy counts), else from sorted leaf keys of
//      the points (a run of equal keys is one leaf);
//   2. puts the points in row-major leaf order per problem (a counting sort on the dense
//      grids, else the sorted keys), so the sources of a leaf row segment are one
//      contiguous range, and lists the occupied leaves with their first source and
//      target;
//   3. builds the boxes of every level at once, numbered level by level in parity-class
//      order (class, problem, (y >> 1, x >> 1) row by row: each class one contiguous range
//      of compact ids).  While a bit per cell of every level is affordable (grid_words_max),
//      the boxes are the set bits of grids laid out in that very order: a leaf sets its
//      ancestors' bits, one scan of the words' populations numbers the boxes, and parents,
//      children and interaction lists are bit tests and ranks.  Deeper trees of few points
//      keep sorted keys: each leaf emits its level-k key where it heads its level-k row
//      segment, one sort and one unique pass give every level's boxes, one stable partition
//      by (level, class) their numbers, and the links are binary searches;
//   4. lists the near-field strips (SW consecutive leaves of a row holding a target) and
//      the occupied leaves of each strip's three neighbour-row segments.
// The sorts are a stable least-significant-digit radix sort (8-bit digits, per-block
// digit counts, one exclusive scan, ranked scatter).  When targets equal sources (same
// offsets and coordinates) one order serves both.
#include <algorithm>
#include <climits>

#include "device_common.h"

namespace lfmm {

namespace {

constexpr int kT = 256;

int grid_of(int64_t n, int threads = kT, int cap = 152 * 16) {
    int64_t g = (n + threads - 1) / threads;
    return (int)std::max<int64_t>(1, std::min<int64_t>(g, cap));
}

// ------------------------------------------------------------------------- exclusive scan
constexpr int kScanBlock = 1024;

// POP: the items are the populations of the words in[i]
template <bool POP>
__device__ __forceinline__ int32_t scan_item(int32_t v) {
    return POP ? __popc((unsigned)v) : v;
}

template <bool POP>
__global__ void scan_reduce_kernel(const int32_t* __restrict__ in, int64_t n, int32_t* __restrict__ sums) {
    __shared__ int32_t w[kT / 32];
    const int64_t base = (int64_t)blockIdx.x * kScanBlock;
    int32_t v = 0;
    for (int i = threadIdx.x; i < kScanBlock; i += blockDim.x)
        if (base + i < n) v += scan_item<POP>(in[base + i]);
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    if ((threadIdx.x & 31) == 0) w[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        int32_t t = 0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += w[i];
        sums[blockIdx.x] = t;
    }
}

// exclusive scan of the block totals in place (one block); total to sums[nb]
__global__ void scan_sums_kernel(int32_t* __restrict__ sums, int nb) {
    __shared__ int32_t carry_s, w[1024 / 32];
    if (threadIdx.x == 0) carry_s = 0;
    __syncthreads();
    for (int base = 0; base < nb; base += blockDim.x) {
        const int i = base + threadIdx.x;
        const int32_t v = i < nb ? sums[i] : 0;
        int32_t x = v;
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(kFull, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) w[wid] = x;
        __syncthreads();
        if (wid == 0) {
            int32_t s = lane < (int)(blockDim.x >> 5) ? w[lane] : 0;
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t y = __shfl_up_sync(kFull, s, o);
                if (lane >= o) s += y;
            }
            w[lane] = s;
        }
        __syncthreads();
        const int32_t incl = x + (wid > 0 ? w[wid - 1] : 0);
        const int32_t carry = carry_s;
        if (i < nb) sums[i] = carry + incl - v;
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) carry_s = carry + incl;
        __syncthreads();
    }
    if (threadIdx.x == 0) sums[nb] = carry_s;
}

// TOTALS: sums holds the blocks' totals, else their prefix sums
template <bool POP, bool TOTALS>
__global__ void scan_apply_kernel(const int32_t* __restrict__ in, int64_t n, const int32_t* __restrict__ sums,
                                  int32_t* __restrict__ out) {
    __shared__ int32_t w[kT / 32], wb[kT / 32];
    if (TOTALS) {
        int32_t b = 0;
        for (int i = threadIdx.x; i < (int)blockIdx.x; i += kT) b += sums[i];
        for (int o = 16; o; o >>= 1) b += __shfl_xor_sync(kFull, b, o);
        if ((threadIdx.x & 31) == 0) wb[threadIdx.x >> 5] = b;
    }
    constexpr int PER = kScanBlock / kT;  // 4 consecutive items per thread
    const int64_t base = (int64_t)blockIdx.x * kScanBlock + (int64_t)threadIdx.x * PER;
    int32_t v[PER], t = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        v[j] = base + j < n ? scan_item<POP>(in[base + j]) : 0;
        t += v[j];
    }
    int32_t x = t;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) w[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int32_t s = lane < (int)(blockDim.x >> 5) ? w[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(kFull, s, o);
            if (lane >= o) s += y;
        }
        if (lane < kT / 32) w[lane] = s;
    }
    __syncthreads();
    int32_t before = 0;
    if (TOTALS) {
#pragma unroll
        for (int i = 0; i < kT / 32; ++i) before += wb[i];
    } else {
        before = sums[blockIdx.x];
    }
    int32_t run = before + x - t + (wid > 0 ? w[wid - 1] : 0);
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        if (base + j < n) out[base + j] = run;
        run += v[j];
    }
    const int64_t nblk = (n + kScanBlock - 1) / kScanBlock;
    if (blockIdx.x == nblk - 1 && threadIdx.x == blockDim.x - 1) out[n] = run;
}

int64_t scan_tmp_ints(int64_t n) { return (n + kScanBlock - 1) / kScanBlock + 1; }

// The scan of up to kScanSmall items in one block (16,384 items that way took 12 us, 65,536
// 41 us), and up to kScanTwo block totals without a launch of their own: every block adds the
// totals before it itself.  Two launches fewer, or one, on the host, which is what the
// building of small trees waits for.
constexpr int64_t kScanSmall = 4096;
constexpr int64_t kScanTwo = 2048;
template <bool POP>
__global__ void __launch_bounds__(1024) scan_small_kernel(const int32_t* __restrict__ in, int n,
                                                          int32_t* __restrict__ out) {
    __shared__ int32_t w[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, i0 = 4 * threadIdx.x;
    int32_t v[4], t = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        v[j] = i0 + j < n ? scan_item<POP>(in[i0 + j]) : 0;
        t += v[j];
    }
    int32_t x = t;
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) w[wid] = x;
    __syncthreads();
    int32_t s = w[lane];
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(kFull, s, o);
        if (lane >= o) s += y;
    }
    const int32_t before = __shfl_sync(kFull, s, max(wid - 1, 0));
    int32_t run = (wid > 0 ? before : 0) + x - t;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (i0 + j < n) out[i0 + j] = run;
        run += v[j];
    }
    if (threadIdx.x == 1023) out[n] = run;
}

// out[0..n] = exclusive prefix sums of in[0..n) (out[n] = total); sums: scan_tmp_ints(n)
template <bool POP = false>
cudaError_t exscan(const int32_t* in, int32_t* out, int64_t n, int32_t* sums, cudaStream_t s) {
    const int64_t nb = (n + kScanBlock - 1) / kScanBlock;
    if (nb == 0) return cudaMemsetAsync(out, 0, sizeof(int32_t), s);
    if (n <= kScanSmall) {
        scan_small_kernel<POP><<<1, 1024, 0, s>>>(in, (int)n, out);
        return cudaGetLastError();
    }
    scan_reduce_kernel<POP><<<(unsigned)nb, kT, 0, s>>>(in, n, sums);
    if (nb <= kScanTwo) {
        scan_apply_kernel<POP, true><<<(unsigned)nb, kT, 0, s>>>(in, n, sums, out);
        return cudaGetLastError();
    }
    scan_sums_kernel<<<1, 1024, 0, s>>>(sums, (int)nb);
    scan_apply_kernel<POP, false><<<(unsigned)nb, kT, 0, s>>>(in, n, sums, out);
    return cudaGetLastError();
}
int exscan_launches(int64_t n) {
    return n <= kScanSmall ? 1 : n <= kScanTwo * kScanBlock ? 2 : 3;
}

// ------------------------------------------------------------------------- radix sort
constexpr int kRadix = 256;
constexpr int kItems = 8;
constexpr int kTile = kT * kItems;  // keys per block

// hist[d * nblocks + b] = keys of tile b whose digit (bits shift .. shift + 7) is d
__global__ void radix_hist_kernel(const uint64_t* __restrict__ keys, int64_t n, int shift, int nblocks,
                                  int32_t* __restrict__ hist) {
    __shared__ int32_t h[kRadix];
    for (int d = threadIdx.x; d < kRadix; d += blockDim.x) h[d] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kTile;
    for (int i = threadIdx.x; i < kTile; i += blockDim.x)
        if (base + i < n) atomicAdd(&h[(int)((keys[base + i] >> shift) & (kRadix - 1))], 1);
    __syncthreads();
    for (int d = threadIdx.x; d < kRadix; d += blockDim.x) hist[(int64_t)d * nblocks + blockIdx.x] = h[d];
}

// Stable scatter of tile b: keys go to offs[d * nblocks + b] + (keys of digit d before them
// in the tile).  Warp w takes the tile's keys [w 256, w 256 + 256) in 8 rounds of 32; a
// key's rank among its warp's keys of the same digit comes from the lanes that share its
// digit in the round (match) and the warp's running count; warps are then offset by the
// counts of the warps before them.  The tile is put in order in shared memory first, so
// that consecutive threads store a digit's run of keys (8 on average) to consecutive
// places: storing each key from its own lane sent a 32-byte sector per key and value
// (4.2 M keys, four passes: 212 us, now 166).
__global__ void __launch_bounds__(kT) radix_scatter_kernel(const uint64_t* __restrict__ kin,
                                                           const uint32_t* __restrict__ vin,
                                                           uint64_t* __restrict__ kout, uint32_t* __restrict__ vout,
                                                           int64_t n, int shift, int nblocks,
                                                           const int32_t* __restrict__ offs) {
    static_assert(kT == kRadix, "one thread per digit");
    __shared__ int32_t wc[kT / 32][kRadix];
    __shared__ int32_t boff[kRadix];  // place in the output of the tile's key at position 0 of its order, per digit
    __shared__ int32_t wsum[kT / 32];
    __shared__ uint64_t sk[kTile];
    __shared__ uint32_t sv[kTile];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < (kT / 32) * kRadix; i += kT) (&wc[0][0])[i] = 0;
    const int off = offs[(int64_t)threadIdx.x * nblocks + blockIdx.x];
    const int64_t base = (int64_t)blockIdx.x * kTile + (int64_t)warp * (32 * kItems);
    uint64_t k[kItems];
    uint32_t v[kItems];
    int dg[kItems], rk[kItems];
#pragma unroll
    for (int it = 0; it < kItems; ++it) {
        const int64_t i = base + it * 32 + lane;
        k[it] = i < n ? kin[i] : 0ull;
        v[it] = (i < n && vin) ? vin[i] : 0u;
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kItems; ++it) {
        const bool ok = base + it * 32 + lane < n;
        const int d = ok ? (int)((k[it] >> shift) & (kRadix - 1)) : kRadix;  // kRadix: no key
        const unsigned peers = __match_any_sync(kFull, d);
        const int leader = __ffs(peers) - 1;
        int start = 0;
        if (lane == leader && ok) {
            start = wc[warp][d];
            wc[warp][d] = start + __popc(peers);
        }
        start = __shfl_sync(kFull, start, leader);
        dg[it] = d;
        rk[it] = start + __popc(peers & ((1u << lane) - 1u));
        __syncwarp();
    }
    __syncthreads();
    // thread d: the tile's keys of smaller digits, then of earlier warps
    int run = 0;
    for (int w = 0; w < kT / 32; ++w) run += wc[w][threadIdx.x];
    int inc = run;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    int first = inc - run;
    for (int w = 0; w < warp; ++w) first += wsum[w];
    boff[threadIdx.x] = off - first;
    for (int w = 0; w < kT / 32; ++w) {
        const int t = wc[w][threadIdx.x];
        wc[w][threadIdx.x] = first;
        first += t;
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kItems; ++it) {
        if (dg[it] < kRadix) {
            const int pos = wc[warp][dg[it]] + rk[it];
            sk[pos] = k[it];
            sv[pos] = v[it];
        }
    }
    __syncthreads();
    const int cnt = (int)min((int64_t)kTile, n - (int64_t)blockIdx.x * kTile);
    for (int i = threadIdx.x; i < cnt; i += kT) {
        const uint64_t key = sk[i];
        const int64_t pos = (int64_t)boff[(int)((key >> shift) & (kRadix - 1))] + i;
        kout[pos] = key;
        if (vout) vout[pos] = sv[i];
    }
}

// Device scratch of one sorting job: second key / value buffers and the digit counts.
struct SortBufs {
    uint64_t* k2 = nullptr;
    uint32_t* v2 = nullptr;
    int32_t* hist = nullptr;  // 256 nblocks + 1 ints
    int32_t* sums = nullptr;  // scan_tmp_ints(256 nblocks)
};

int64_t sort_hist_ints(int64_t n) { return (int64_t)kRadix * ((n + kTile - 1) / kTile) + 1; }

// One stable pass over the digit at `shift`: (ki, vi) -> (ko, vo); values optional.
cudaError_t radix_pass(const uint64_t* ki, const uint32_t* vi, uint64_t* ko, uint32_t* vo, int64_t n, int shift,
                       SortBufs& b, cudaStream_t s) {
    const int nblocks = (int)((n + kTile - 1) / kTile);
    radix_hist_kernel<<<nblocks, kT, 0, s>>>(ki, n, shift, nblocks, b.hist);
    cudaError_t e = exscan(b.hist, b.hist, (int64_t)kRadix * nblocks, b.sums, s);
    if (e != cudaSuccess) return e;
    radix_scatter_kernel<<<nblocks, kT, 0, s>>>(ki, vi, ko, vo, n, shift, nblocks, b.hist);
    return cudaGetLastError();
}

// Sorts n keys (and values, when v is set) by their low `bits` bits (bits <= 64; the
// keys hold no higher bits), stably, in place: the passes alternate between (k, v) and
// the scratch, and after an odd number of them one copy brings the result back.
cudaError_t radix_sort(uint64_t* k, uint32_t* v, int64_t n, int bits, SortBufs& b, cudaStream_t s) {
    if (n <= 1) return cudaSuccess;
    const int passes = std::max(1, (bits + 7) / 8);
    uint64_t *ki = k, *ko = b.k2;
    uint32_t *vi = v, *vo = v ? b.v2 : nullptr;
    for (int pass = 0; pass < passes; ++pass) {
        cudaError_t e = radix_pass(ki, vi, ko, vo, n, 8 * pass, b, s);
        if (e != cudaSuccess) return e;
        std::swap(ki, ko);
        std::swap(vi, vo);
    }
    if (passes & 1) {
        cudaError_t e = cudaMemcpyAsync(k, ki, (size_t)n * sizeof(uint64_t), cudaMemcpyDeviceToDevice, s);
        if (e == cudaSuccess && v) e = cudaMemcpyAsync(v, vi, (size_t)n * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s);
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

// ------------------------------------------------------------------------- keys and runs
__device__ __forceinline__ uint64_t pack_key(int p, int y, int x, int kb) {
    return ((uint64_t)p << (2 * kb)) | ((uint64_t)y << kb) | (uint64_t)x;
}
__device__ __forceinline__ void unpack_key(uint64_t key, int kb, int& p, int& y, int& x) {
    const uint64_t m = ((uint64_t)1 << kb) - 1;
    x = (int)(key & m);
    y = (int)((key >> kb) & m);
    p = (int)(key >> (2 * kb));
}
__device__ __forceinline__ int64_t lower_bound_key(const uint64_t* __restrict__ a, int64_t n, uint64_t v) {
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (a[mid] < v) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// [first, end) of every box row of A (level k, problem p, row y; its entry is
// row_off[k np + p] + y); rows without boxes keep {0, 0}
__global__ void row_range_kernel(const uint64_t* __restrict__ A, int64_t na, int kb, int kbits, int np,
                                 const int64_t* __restrict__ row_off, int2* __restrict__ rows) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < na; j += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t key = A[j], rk = key >> kb;
        const bool head = j == 0 || (A[j - 1] >> kb) != rk;
        const bool tail = j == na - 1 || (A[j + 1] >> kb) != rk;
        if (!head && !tail) continue;
        int p, y, x;
        unpack_key(key & (((uint64_t)1 << kbits) - 1), kb, p, y, x);
        const int64_t r = row_off[(key >> kbits) * np + p] + y;
        if (head) rows[r].x = (int)j;
        if (tail) rows[r].y = (int)(j + 1);
    }
}

// First entry of A at or after key v = (k, p, y, x) within its row (the row's end if none;
// `end` is set to the row's end), or, without a row table, within all of A.
__device__ __forceinline__ int64_t find_in_row(const uint64_t* __restrict__ A, int64_t na,
                                               const int2* __restrict__ rows, const int64_t* __restrict__ row_off,
                                               int np, int k, int p, int y, uint64_t v, int64_t& end) {
    int64_t lo = 0, hi = na;
    if (rows) {
        const int2 rr = rows[row_off[(int64_t)k * np + p] + y];
        lo = rr.x;
        hi = rr.y;
    }
    end = hi;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (A[mid] < v) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

__global__ void pid_kernel(const int64_t* __restrict__ off, int np, int32_t* __restrict__ pid) {
    for (int p = blockIdx.x; p < np; p += gridDim.x)
        for (int64_t i = off[p] + threadIdx.x; i < off[p + 1]; i += blockDim.x) pid[i] = p;
}

// bounding box of each problem's sources and targets, one block per problem
__global__ void bbox_forest_kernel(const int2* __restrict__ src, const int64_t* __restrict__ soff,
                                   const int2* __restrict__ tgt, const int64_t* __restrict__ toff, int np,
                                   int4* __restrict__ bb) {
    __shared__ int red[4][kT / 32];
    for (int p = blockIdx.x; p < np; p += gridDim.x) {
        int x0 = INT_MAX, y0 = INT_MAX, x1 = INT_MIN, y1 = INT_MIN;
        // four loads in flight per thread (a problem's points beyond its last repeat it); one
        // by one, 11.4 M points in 4,096 problems took 103 us, now 55
        auto sweep = [&](const int2* __restrict__ xy, int64_t a, int64_t b) {
            for (int64_t i = a + threadIdx.x; i < b; i += 4 * blockDim.x) {
                int2 v[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) v[q] = xy[min(i + (int64_t)q * blockDim.x, b - 1)];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    x0 = min(x0, v[q].x), y0 = min(y0, v[q].y), x1 = max(x1, v[q].x), y1 = max(y1, v[q].y);
            }
        };
        sweep(src, soff[p], soff[p + 1]);
        sweep(tgt, toff[p], toff[p + 1]);
        for (int o = 16; o; o >>= 1) {
            x0 = min(x0, __shfl_xor_sync(kFull, x0, o));
            y0 = min(y0, __shfl_xor_sync(kFull, y0, o));
            x1 = max(x1, __shfl_xor_sync(kFull, x1, o));
            y1 = max(y1, __shfl_xor_sync(kFull, y1, o));
        }
        const int w = threadIdx.x >> 5;
        if ((threadIdx.x & 31) == 0) red[0][w] = x0, red[1][w] = y0, red[2][w] = x1, red[3][w] = y1;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int i = 1; i < (int)(blockDim.x >> 5); ++i) {
                x0 = min(x0, red[0][i]), y0 = min(y0, red[1][i]);
                x1 = max(x1, red[2][i]), y1 = max(y1, red[3][i]);
            }
            bb[p] = make_int4(x0, y0, x1, y1);
        }
        __syncthreads();
    }
}

// leaf key of every point at leaf side 2^ls (value: the point's index)
__global__ void leaf_key_kernel(const int2* __restrict__ xy, int64_t n, const int32_t* __restrict__ pid,
                                const int32_t* __restrict__ x0, const int32_t* __restrict__ y0, int ls, int kb,
                                uint64_t* __restrict__ key, uint32_t* __restrict__ idx) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int p = pid ? pid[i] : 0;
        const int2 v = xy[i];
        const int bx = (int)(((int64_t)v.x - x0[p]) >> ls), by = (int)(((int64_t)v.y - y0[p]) >> ls);
        key[i] = pack_key(p, by, bx, kb);
        idx[i] = (uint32_t)i;
    }
}

// flag[i] = 1 where a run of equal keys starts (and key is not the skip value)
__global__ void run_start_kernel(const uint64_t* __restrict__ key, int64_t n, uint64_t skip,
                                 int32_t* __restrict__ flag) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        flag[i] = (key[i] != skip && (i == 0 || key[i] != key[i - 1])) ? 1 : 0;
}

// out[pos[i]] = key[i] and first[pos[i]] = i at run starts; first[m] = n (m runs)
__global__ void run_compact_kernel(const uint64_t* __restrict__ key, int64_t n, const int32_t* __restrict__ flag,
                                   const int32_t* __restrict__ pos, uint64_t* __restrict__ out,
                                   int32_t* __restrict__ first) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        if (flag[i]) {
            out[pos[i]] = key[i];
            if (first) first[pos[i]] = (int32_t)i;
        }
        if (i == 0 && first) first[pos[n]] = (int32_t)n;
    }
}

// *mx = longest run (first[j + 1] - first[j]) over j < m
__global__ void max_run_kernel(const int32_t* __restrict__ first, int64_t m, int* __restrict__ mx) {
    int best = 0;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x)
        best = max(best, first[j + 1] - first[j]);
    for (int o = 16; o; o >>= 1) best = max(best, __shfl_xor_sync(kFull, best, o));
    if ((threadIdx.x & 31) == 0) atomicMax(mx, best);
}

// sorted points: perm = the caller's index, loc = lx | ly << 16 inside the leaf
__global__ void point_order_kernel(const int2* __restrict__ xy, int64_t n, const uint32_t* __restrict__ idx,
                                   const int32_t* __restrict__ pid, const int32_t* __restrict__ x0,
                                   const int32_t* __restrict__ y0, int ls, int32_t* __restrict__ loc,
                                   int32_t* __restrict__ perm) {
    const int mask = (1 << ls) - 1;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t j = idx[i];
        const int p = pid ? pid[j] : 0;
        const int2 v = xy[j];
        const int lx = (int)(((int64_t)v.x - x0[p]) & mask), ly = (int)(((int64_t)v.y - y0[p]) & mask);
        loc[i] = lx | (ly << 16);
        perm[i] = (int32_t)j;
    }
}

// first sorted source / target of every occupied leaf (lower bound of its key); entry m
// holds the totals
__global__ void leaf_ranges_kernel(const uint64_t* __restrict__ leaves, int64_t m, const uint64_t* __restrict__ sk,
                                   int64_t ns, const uint64_t* __restrict__ tk, int64_t nt, int32_t* __restrict__ rs,
                                   int32_t* __restrict__ rt) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j <= m; j += (int64_t)gridDim.x * blockDim.x) {
        if (j == m) {
            rs[j] = (int32_t)ns;
            rt[j] = (int32_t)nt;
        } else {
            rs[j] = (int32_t)lower_bound_key(sk, ns, leaves[j]);
            rt[j] = (int32_t)lower_bound_key(tk, nt, leaves[j]);
        }
    }
}

// Boxes of every level from the occupied leaves.  A box of level k (k levels above the
// leaves) of problem p is the key (k << kbits) | (p, y >> k, x >> k) of any leaf below it;
// the levels of p are k = 1 .. L_p - 2 (levels >= 2 of its own tree).  Leaf j emits its
// level-k key only when it heads its level-k row segment (the previous leaf lies in
// another problem, row or level-k column), which leaves at most the 2^k leaf rows of a
// box to remove as duplicates.  Entry (k - 1) m + j.
__global__ void head_flag_kernel(const uint64_t* __restrict__ leaves, int64_t m, int kmax, const int32_t* __restrict__ L,
                                 int kb, int32_t* __restrict__ flag) {
    const int64_t n = m * kmax;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int k = (int)(i / m) + 1;
        const int64_t j = i - (int64_t)(k - 1) * m;
        int p, y, x;
        unpack_key(leaves[j], kb, p, y, x);
        bool head = L[p] - k >= 2;
        if (head && j > 0) {
            int pp, yy, xx;
            unpack_key(leaves[j - 1], kb, pp, yy, xx);
            head = !(pp == p && yy == y && (xx >> k) == (x >> k));
        }
        flag[i] = head ? 1 : 0;
    }
}

__global__ void head_key_kernel(const uint64_t* __restrict__ leaves, int64_t m, int kmax, int kb, int kbits,
                                const int32_t* __restrict__ flag, const int32_t* __restrict__ pos,
                                uint64_t* __restrict__ out) {
    const int64_t n = m * kmax;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        if (!flag[i]) continue;
        const int k = (int)(i / m) + 1;
        const int64_t j = i - (int64_t)(k - 1) * m;
        int p, y, x;
        unpack_key(leaves[j], kb, p, y, x);
        out[pos[i]] = ((uint64_t)k << kbits) | pack_key(p, y >> k, x >> k, kb);
    }
}

// Partition key 4 k + class of every box of every level (value: its position in the
// level-major row-major key array A).  A is ordered by (level, problem, row, column), so a
// stable partition by this one digit leaves every class in (problem, y >> 1, x >> 1) order:
// one radix pass instead of a sort by the whole (class, box) key (five passes at 14 levels;
// clustered_4m builds 1.3 M boxes).
__global__ void class_key_kernel(const uint64_t* __restrict__ A, int64_t n, int kb, int kbits,
                                 uint64_t* __restrict__ ck, uint32_t* __restrict__ idx) {
    const uint64_t low = ((uint64_t)1 << kbits) - 1;
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < n; g += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t key = A[g];
        const uint64_t k = key >> kbits;
        int p, y, x;
        unpack_key(key & low, kb, p, y, x);
        const uint64_t c = (uint64_t)((x & 1) | ((y & 1) << 1));
        ck[g] = (k << 2) | c;
        idx[g] = (uint32_t)g;
    }
}

// first class-major position of class c of level k (entry 4 k + c; entry 4 nk: all boxes)
__global__ void class_starts_kernel(const uint64_t* __restrict__ ck, int64_t n, int nk,
                                    int64_t* __restrict__ cstart) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t > 4 * nk) return;
    if (t == 4 * nk) {
        cstart[t] = n;
        return;
    }
    cstart[t] = lower_bound_key(ck, n, (uint64_t)t);
}

// Box b of the class-major order (all levels, level-major) <- its row-major entry cm[b]
// of A: problem, coordinates, the level-local compact id of each entry of A, and the
// row-major leaf index of each level-0 box.
__global__ void box_records_kernel(const uint64_t* __restrict__ A, const uint64_t* __restrict__ ck,
                                   const uint32_t* __restrict__ cm, int64_t n, const int64_t* __restrict__ cstart, int kb,
                                   int kbits, int32_t* __restrict__ bp, int32_t* __restrict__ bxy,
                                   int32_t* __restrict__ local_of, int32_t* __restrict__ leaf_rl) {
    const uint64_t low = ((uint64_t)1 << kbits) - 1;
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < n; b += (int64_t)gridDim.x * blockDim.x) {
        const int k = (int)(ck[b] >> 2);
        const uint32_t g = cm[b];
        int p, y, x;
        unpack_key(A[g] & low, kb, p, y, x);
        bp[b] = p;
        bxy[b] = x | (y << 16);
        const int64_t local = b - cstart[4 * k];
        local_of[g] = (int32_t)local;
        if (k == 0) leaf_rl[local] = (int32_t)g;
    }
}

// Parent, children and interaction list (Def. 6.1, slot order of the box's class) of
// every box, by search in A (sorted by level, problem, row, column).  A list's 27 boxes
// lie in the six rows y - 2 - (y & 1) .. y + 3 - (y & 1), six columns wide: one search
// per row, then a scan of at most six keys; s_slot maps an offset to its slot.
__global__ void links_kernel(int64_t n, const uint64_t* __restrict__ ck, const uint64_t* __restrict__ A, int64_t na,
                             const int32_t* __restrict__ local_of, const int32_t* __restrict__ bp,
                             const int32_t* __restrict__ bxy, const int32_t* __restrict__ L, int kb, int kbits, int kmax,
                             const int2* __restrict__ rows, const int64_t* __restrict__ row_off, int np,
                             int32_t* __restrict__ par, int32_t* __restrict__ ch, int32_t* __restrict__ il) {
    __shared__ signed char s_slot[4][36];
    for (int t = threadIdx.x; t < 4 * 36; t += blockDim.x) (&s_slot[0][0])[t] = -1;
    __syncthreads();
    for (int t = threadIdx.x; t < 4 * 27; t += blockDim.x) {
        const int c = t / 27, st = t % 27, px = c & 1, py = c >> 1;
        int dx, dy;
        interaction_slot(px, py, st, dx, dy);
        s_slot[c][(dy + 2 + py) * 6 + dx + 2 + px] = (signed char)st;
    }
    __syncthreads();
    const uint64_t cmask = ((uint64_t)1 << kb) - 1;
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < n; b += (int64_t)gridDim.x * blockDim.x) {
        const int k = (int)(ck[b] >> 2);
        const int p = bp[b];
        const int x = bxy[b] & 0xffff, y = bxy[b] >> 16;
        const int l = L[p] - k;
        const int nn = 1 << l;
        const int px = x & 1, py = y & 1, c = px | (py << 1);
        // parent at level k + 1 (a level >= 2 of the problem's tree)
        int pr = -1;
        if (k + 1 <= kmax && l - 1 >= 2) {
            const uint64_t v = ((uint64_t)(k + 1) << kbits) | pack_key(p, y >> 1, x >> 1, kb);
            int64_t e;
            const int64_t j = find_in_row(A, na, rows, row_off, np, k + 1, p, y >> 1, v, e);
            if (j < e && A[j] == v) pr = local_of[j];
        }
        par[b] = pr;
        // children at level k - 1, two per row
        if (k >= 1) {
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const uint64_t v = ((uint64_t)(k - 1) << kbits) | pack_key(p, 2 * y + r, 2 * x, kb);
                int64_t e;
                int64_t j = find_in_row(A, na, rows, row_off, np, k - 1, p, 2 * y + r, v, e);
                int c0 = -1, c1 = -1;
                if (j < e && A[j] == v) {
                    c0 = local_of[j];
                    ++j;
                }
                if (j < e && A[j] == v + 1) c1 = local_of[j];
                ch[b * 4 + 2 * r] = c0;
                ch[b * 4 + 2 * r + 1] = c1;
            }
        }
        // interaction list
        int32_t* out = il + b * 27;
        for (int st = 0; st < 27; ++st) out[st] = -1;
        const uint64_t lev = (uint64_t)k << kbits;
        const int xlo = max(x - 2 - px, 0), xhi = min(x + 3 - px, nn - 1);
        for (int dy = -2 - py; dy <= 3 - py; ++dy) {
            const int yy = y + dy;
            if (yy < 0 || yy >= nn) continue;
            const uint64_t vhi = lev | pack_key(p, yy, xhi, kb);
            int64_t e;
            for (int64_t j = find_in_row(A, na, rows, row_off, np, k, p, yy, lev | pack_key(p, yy, xlo, kb), e);
                 j < e && A[j] <= vhi; ++j) {
                const int dx = (int)(A[j] & cmask) - x;
                const int sl = s_slot[c][(dy + 2 + py) * 6 + dx + 2 + px];
                if (sl >= 0) out[sl] = local_of[j];
            }
        }
    }
}

// ------------------------------------------------------------------------- bit grids
// One bit per cell of every level: level k, class c, problem p is a grid of h x h bits, row
// by row from a word boundary, h = max(1, 2^(L_p - k) / 2), at word
// base[k] + c stride[k] + off[k np + p].  The words' order is the order of the compact ids,
// so a box's id is the number of set bits before its own (rank).
constexpr int kGridLevels = 21;
struct BitGrid {
    uint32_t base[kGridLevels], stride[kGridLevels];
    int nk, np, kmax;
    const uint32_t* off;  // null with one problem
    const int32_t* L;
    uint32_t* bits;
    const int32_t* before;  // set bits before each word
};
__device__ __forceinline__ uint32_t grid_word(const BitGrid& G, int k, int c, int p) {
    return G.base[k] + (uint32_t)c * G.stride[k] + (G.off ? G.off[k * G.np + p] : 0u);
}

// Every leaf's bit and those of its ancestors (levels >= 2 of its problem's tree).  A leaf
// that follows another of the same box in its row leaves that box's and all higher bits to
// the first one.
__global__ void grid_set_kernel(const BitGrid G, const uint64_t* __restrict__ leaves, const int32_t* __restrict__ m_d,
                                int kb) {
    const int64_t m = *m_d;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x) {
        int p, y, x, pp = -1, yy = 0, xx = 0;
        unpack_key(leaves[j], kb, p, y, x);
        if (j > 0) unpack_key(leaves[j - 1], kb, pp, yy, xx);
        const bool row = pp == p && yy == y;
        const int l = G.L[p];
        for (int k = 0; k < G.nk; ++k) {
            if (k > 0 && (l - k < 2 || (row && (xx >> k) == (x >> k)))) break;
            const int X = x >> k, Y = y >> k, h = max(1, (1 << (l - k)) >> 1);
            const uint32_t i = (uint32_t)(Y >> 1) * (uint32_t)h + (uint32_t)(X >> 1);
            atomicOr(G.bits + grid_word(G, k, (X & 1) | ((Y & 1) << 1), p) + (i >> 5), 1u << (i & 31));
        }
    }
}

// first id of every class of every level (entry 4 nk: all boxes), the level-local class
// starts, and what the host waits for: {M, class starts}
__global__ void grid_starts_kernel(const BitGrid G, int64_t words, const int32_t* __restrict__ m_d,
                                   int64_t* __restrict__ cstart, int64_t* __restrict__ dcls, int* __restrict__ out) {
    for (int t = threadIdx.x; t <= 4 * G.nk; t += blockDim.x) {
        auto start = [&](int i) -> int32_t {
            return G.before[i >= 4 * G.nk ? words : (int64_t)G.base[i >> 2] + (i & 3) * (int64_t)G.stride[i >> 2]];
        };
        const int32_t v = start(t);
        cstart[t] = v;
        out[1 + t] = v;
        if (t < 4 * G.nk) {
            dcls[5 * (t >> 2) + (t & 3)] = v - start(t & ~3);
            if ((t & 3) == 3) dcls[5 * (t >> 2) + 4] = start(t + 1) - start(t & ~3);
        }
    }
    if (threadIdx.x == 0) out[0] = *m_d;
}

// problem and coordinates of every box, word by word
__global__ void grid_records_kernel(const BitGrid G, int64_t words, int32_t* __restrict__ bp,
                                    int32_t* __restrict__ bxy) {
    for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < words; w += (int64_t)gridDim.x * blockDim.x) {
        uint32_t v = G.bits[w];
        if (!v) continue;
        int k = 0;
        while (k + 1 < G.nk && (uint32_t)w >= G.base[k + 1]) ++k;
        const uint32_t r = (uint32_t)w - G.base[k];
        const int c = (int)(r / G.stride[k]);
        const uint32_t in = r - (uint32_t)c * G.stride[k];
        int p = 0;
        if (G.off) {
            int lo = 0, hi = G.np;  // off[p] <= in < off[p + 1]
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (G.off[k * G.np + mid] <= in) lo = mid;
                else hi = mid;
            }
            p = lo;
        }
        const int lh = max(0, G.L[p] - k - 1);
        int id = G.before[w];
        const uint32_t i0 = (in - (G.off ? G.off[k * G.np + p] : 0u)) * 32;
        for (; v; v &= v - 1, ++id) {
            const uint32_t i = i0 + (uint32_t)__ffs(v) - 1;
            const int x = 2 * (int)(i & ((1u << lh) - 1)) + (c & 1), y = 2 * (int)(i >> lh) + (c >> 1);
            bp[id] = p;
            bxy[id] = x | (y << 16);
        }
    }
}

// the level-0 id of every leaf, and the leaf of every level-0 id
__global__ void grid_leaves_kernel(const BitGrid G, const uint64_t* __restrict__ leaves, int64_t m, int kb,
                                   int32_t* __restrict__ rl_id, int32_t* __restrict__ leaf_rl) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x) {
        int p, y, x;
        unpack_key(leaves[j], kb, p, y, x);
        const int h = max(1, (1 << G.L[p]) >> 1);
        const uint32_t i = (uint32_t)(y >> 1) * (uint32_t)h + (uint32_t)(x >> 1);
        const uint32_t w = grid_word(G, 0, (x & 1) | ((y & 1) << 1), p) + (i >> 5);
        const int id = G.before[w] + __popc(G.bits[w] & ((1u << (i & 31)) - 1));
        rl_id[j] = id;
        leaf_rl[id] = (int32_t)j;
    }
}

// Parent, children and interaction list of every box (as links_kernel): bit tests in the
// grids, ranks from the words' running counts.  The 27 candidates are, in each class, the
// 3 x 3 cells around the parent's: three bits in a row, in one word or two.  The lists are
// gathered in shared memory (27 words a box, an odd stride) and written in one piece.
__global__ void __launch_bounds__(kT) grid_links_kernel(const BitGrid G, int64_t n, const int64_t* __restrict__ cstart,
                                                        const int32_t* __restrict__ bp,
                                                        const int32_t* __restrict__ bxy, int32_t* __restrict__ par,
                                                        int32_t* __restrict__ ch, int32_t* __restrict__ il) {
    __shared__ signed char s_slot[4][36];
    __shared__ int s_start[kGridLevels + 1];
    __shared__ int32_t s_il[kT * 27];
    for (int t = threadIdx.x; t < 4 * 36; t += blockDim.x) (&s_slot[0][0])[t] = -1;
    for (int t = threadIdx.x; t <= G.nk; t += blockDim.x) s_start[t] = (int)cstart[4 * t];
    __syncthreads();
    for (int t = threadIdx.x; t < 4 * 27; t += blockDim.x) {
        const int c = t / 27, st = t % 27, px = c & 1, py = c >> 1;
        int dx, dy;
        interaction_slot(px, py, st, dx, dy);
        s_slot[c][(dy + 2 + py) * 6 + dx + 2 + px] = (signed char)st;
    }
    const int64_t tiles = (n + kT - 1) / kT;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int64_t b = tile * kT + threadIdx.x;
        int32_t* my = s_il + threadIdx.x * 27;
        __syncthreads();  // slots are set; the previous tile's lists are written
        for (int st = 0; st < 27; ++st) my[st] = -1;
        if (b < n) {
            int k = 0;
            while (b >= s_start[k + 1]) ++k;
            const int p = bp[b], x = bxy[b] & 0xffff, y = bxy[b] >> 16;
            const int l = G.L[p] - k, hn = 1 << l, h = max(1, hn >> 1);
            const int c = (x & 1) | ((y & 1) << 1), X = x >> 1, Y = y >> 1;
            int pr = -1;
            if (k + 1 <= G.kmax && l - 1 >= 2) {  // its parent is a box of level k + 1
                const uint32_t i = (uint32_t)(Y >> 1) * (uint32_t)(h >> 1) + (uint32_t)(X >> 1);
                const uint32_t w = grid_word(G, k + 1, (X & 1) | ((Y & 1) << 1), p) + (i >> 5);
                pr = G.before[w] + __popc(G.bits[w] & ((1u << (i & 31)) - 1)) - s_start[k + 1];
            }
            par[b] = pr;
            if (k >= 1) {
                const uint32_t i = (uint32_t)y * (uint32_t)hn + (uint32_t)x;  // the same cell of all four classes
                int cc[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t w = grid_word(G, k - 1, q, p) + (i >> 5), v = G.bits[w];
                    cc[q] = (v >> (i & 31)) & 1 ? G.before[w] + __popc(v & ((1u << (i & 31)) - 1)) - s_start[k - 1] : -1;
                }
                reinterpret_cast<int4*>(ch)[b] = make_int4(cc[0], cc[1], cc[2], cc[3]);
            }
            const int x0 = max(X - 1, 0), x1 = min(X + 1, h - 1);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t wq = grid_word(G, k, q, p);
#pragma unroll
                for (int dy = -1; dy <= 1; ++dy) {
                    const int yy = Y + dy;
                    if (yy < 0 || yy >= h) continue;
                    const uint32_t i0 = (uint32_t)yy * (uint32_t)h + (uint32_t)x0, i1 = i0 + (uint32_t)(x1 - x0);
                    const uint32_t w0 = wq + (i0 >> 5), w1 = wq + (i1 >> 5);
                    const uint32_t v0 = G.bits[w0], v1 = w1 == w0 ? v0 : G.bits[w1];
                    const uint64_t v = (uint64_t)v0 | (w1 == w0 ? 0ull : (uint64_t)v1 << 32);
                    const int sh = (int)(i0 & 31);
                    if (!((v >> sh) & ((1u << (x1 - x0 + 1)) - 1))) continue;
                    int id = G.before[w0] + __popcll(v & (((uint64_t)1 << sh) - 1)) - s_start[k];
                    for (int xx = x0; xx <= x1; ++xx)
                        if ((v >> (sh + xx - x0)) & 1) {
                            const int sl = s_slot[c][(2 * dy + (q >> 1) + 2) * 6 + 2 * (xx - X) + (q & 1) + 2];
                            if (sl >= 0) my[sl] = id;
                            ++id;
                        }
                }
            }
        }
        __syncthreads();
        const int64_t first = tile * kT * 27, count = min((int64_t)kT, n - tile * kT) * 27;
        for (int t = threadIdx.x; t < count; t += kT) il[first + t] = s_il[t];
    }
}

// Words of bit grids that are affordable: a few bytes per point, and at least what a leaf
// grid of 4,096 x 4,096 cells takes (clustered_4m: 11.2 M words for 8.4 M points).
int64_t grid_words_max(int64_t points) {
    return std::min<int64_t>(std::max<int64_t>((int64_t)1 << 20, 2 * points), (int64_t)1 << 30);
}

// leaf occupancy of every problem's dense leaf grid at side 2^ls (L: leaf levels at that
// side, cell_off: first cell of each problem)
__global__ void dense_count_kernel(const int2* __restrict__ xy, int64_t n, const int32_t* __restrict__ pid,
                                   const int32_t* __restrict__ x0, const int32_t* __restrict__ y0,
                                   const int32_t* __restrict__ L, const int64_t* __restrict__ cell_off, int ls,
                                   int32_t* __restrict__ cnt) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int p = pid ? pid[i] : 0;
        const int2 v = xy[i];
        const int64_t bx = ((int64_t)v.x - x0[p]) >> ls, by = ((int64_t)v.y - y0[p]) >> ls;
        atomicAdd(cnt + cell_off[p] + (by << L[p]) + bx, 1);
    }
}

// Counting sort on the dense leaf grids: each point takes the next slot of its leaf
// (cursor = the leaf's first slot, advanced atomically), so points come out row-major by
// leaf per problem, in arrival order inside a leaf; loc = lx | ly << 16, perm = the
// caller's index.
__global__ void dense_scatter_kernel(const int2* __restrict__ xy, int64_t n, const int32_t* __restrict__ pid,
                                     const int32_t* __restrict__ x0, const int32_t* __restrict__ y0,
                                     const int32_t* __restrict__ L, const int64_t* __restrict__ cell_off, int ls,
                                     int32_t* __restrict__ cursor, int32_t* __restrict__ loc,
                                     int32_t* __restrict__ perm) {
    const int mask = (1 << ls) - 1;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int p = pid ? pid[i] : 0;
        const int2 v = xy[i];
        const int64_t dx = (int64_t)v.x - x0[p], dy = (int64_t)v.y - y0[p];
        const int pos = atomicAdd(cursor + cell_off[p] + ((dy >> ls) << L[p]) + (dx >> ls), 1);
        loc[pos] = (int)(dx & mask) | ((int)(dy & mask) << 16);
        perm[pos] = (int32_t)i;
    }
}

// 1 where a dense leaf holds a source or a target
__global__ void occupied_flag_kernel(const int32_t* __restrict__ cs, const int32_t* __restrict__ ct, int64_t cells,
                                     int32_t* __restrict__ flag) {
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < cells; c += (int64_t)gridDim.x * blockDim.x)
        flag[c] = (cs[c] + (ct ? ct[c] : 0)) > 0 ? 1 : 0;
}

// occupied leaf j (dense cell c, pos[c] = j): key, first source and first target
__global__ void occupied_compact_kernel(const int32_t* __restrict__ flag, const int32_t* __restrict__ pos,
                                        int64_t cells, const int64_t* __restrict__ cell_off, int np,
                                        const int32_t* __restrict__ L, int kb, const int32_t* __restrict__ ss,
                                        const int32_t* __restrict__ ts, uint64_t* __restrict__ key,
                                        int32_t* __restrict__ rs, int32_t* __restrict__ rt) {
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < cells; c += (int64_t)gridDim.x * blockDim.x) {
        if (c == cells - 1) {  // the totals behind the last leaf
            const int m = pos[cells];
            rs[m] = ss[cells];
            rt[m] = ts[cells];
        }
        if (!flag[c]) continue;
        int lo = 0, hi = np;  // problem p: cell_off[p] <= c < cell_off[p + 1]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (cell_off[mid] <= c) lo = mid;
            else hi = mid;
        }
        const int64_t r = c - cell_off[lo];
        const int j = pos[c];
        key[j] = pack_key(lo, (int)(r >> L[lo]), (int)(r & (((int64_t)1 << L[lo]) - 1)), kb);
        rs[j] = ss[c];
        rt[j] = ts[c];
    }
}

// *mx = max(*mx, largest count)
__global__ void max_count_kernel(const int32_t* __restrict__ cnt, int64_t n, int* __restrict__ mx) {
    int best = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        best = max(best, cnt[i]);
    for (int o = 16; o; o >>= 1) best = max(best, __shfl_xor_sync(kFull, best, o));
    if ((threadIdx.x & 31) == 0) atomicMax(mx, best);
}

// *diff = 1 if the two point lists differ anywhere
__global__ void same_points_kernel(const int2* __restrict__ a, const int2* __restrict__ b, int64_t n,
                                   int* __restrict__ diff) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int2 u = a[i], v = b[i];
        if (u.x != v.x || u.y != v.y) *diff = 1;
    }
}

// Strip (problem, leaf row, column / SW) of each occupied leaf: 1 where the leaf is the
// strip's first one with a target.  Leaves are row-major, so a strip's leaves are
// consecutive and at most SW of them: the leaves before this one in its strip are looked
// at directly, and no sort has to bring the strips together.
__global__ void strip_flag_kernel(const uint64_t* __restrict__ leaves, const int32_t* __restrict__ rt, int64_t m,
                                  int kb, int SW, int32_t* __restrict__ flag) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x) {
        int p, y, x;
        unpack_key(leaves[j], kb, p, y, x);
        const uint64_t first = pack_key(p, y, x / SW * SW, kb);
        bool head = rt[j + 1] > rt[j];
        for (int64_t i = j - 1; head && i >= 0 && leaves[i] >= first; --i) head = rt[i + 1] == rt[i];
        flag[j] = head ? 1 : 0;
    }
}

// strip records (problem, leaf row, first column, 0), in the order of their first leaves
__global__ void strip_record_kernel(const uint64_t* __restrict__ leaves, const int32_t* __restrict__ flag,
                                    const int32_t* __restrict__ pos, int64_t m, int kb, int SW,
                                    int4* __restrict__ strips) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x) {
        if (!flag[j]) continue;
        int p, y, x;
        unpack_key(leaves[j], kb, p, y, x);
        strips[pos[j]] = make_int4(p, y, x / SW * SW, 0);
    }
}

// Leaves of the three row segments a strip's near field reads (rows by - 1 .. by + 1,
// columns max(bx0 - 1, 0) .. min(bx0 + SW, n - 1)): index ranges [j0, j1) in the sorted
// occupied-leaf keys, found by binary search.  The end key is column c_hi + 1 taken as a
// sum, so that one past the row's last column carries into the next row.
__global__ void strip_rows_kernel(const int4* __restrict__ strips, const int32_t* __restrict__ nstr_d,
                                  const uint64_t* __restrict__ leaves, int64_t m, const int32_t* __restrict__ L,
                                  int kb, int SW, int4* __restrict__ rows) {
    const int64_t nstr = *nstr_d;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nstr; i += (int64_t)gridDim.x * blockDim.x) {
        const int4 q = strips[i];
        const int p = q.x, by = q.y, bx0 = q.z;
        const int n = 1 << L[p];
        const int bx1 = min(bx0 + SW, n);
        const int c_lo = max(bx0 - 1, 0), c_hi = min(bx1, n - 1);
        int j[6];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const int yy = by + r - 1;
            if (yy >= 0 && yy < n) {
                const uint64_t row = ((uint64_t)p << (2 * kb)) + ((uint64_t)yy << kb);
                j[2 * r] = (int)lower_bound_key(leaves, m, row + (uint64_t)c_lo);
                j[2 * r + 1] = (int)lower_bound_key(leaves, m, row + (uint64_t)c_hi + 1);
            } else {
                j[2 * r] = j[2 * r + 1] = -1;
            }
        }
        rows[2 * i] = make_int4(j[0], j[1], j[2], j[3]);
        rows[2 * i + 1] = make_int4(j[4], j[5], 0, 0);
    }
}

int ceil_log2(int64_t v) {
    int k = 0;
    while (((int64_t)1 << k) < v) ++k;
    return k;
}

struct DevBuf {  // stream-ordered temporary freed on scope exit
    void* ptr = nullptr;
    cudaStream_t s = nullptr;
    ~DevBuf() {
        if (ptr) cudaFreeAsync(ptr, s);
    }
    int get(size_t bytes, cudaStream_t st) {
        s = st;
        const cudaError_t e = dev_malloc(&ptr, bytes ? bytes : 16, st);
        if (e != cudaSuccess) {
            cudaGetLastError();
            ptr = nullptr;
            return fail(LFMM_ENOMEM, "tree build: device allocation of " + std::to_string(bytes) + " bytes failed");
        }
        return LFMM_OK;
    }
};

int alloc(Forest& F, void** out, size_t n, cudaStream_t s) {
    *out = nullptr;
    const cudaError_t e = dev_malloc(out, n ? n : 16, s);
    if (e != cudaSuccess) {
        cudaGetLastError();
        *out = nullptr;
        return fail(LFMM_ENOMEM, "device allocation of " + std::to_string(n) + " bytes failed");
    }
    F.owned.push_back(*out);
    F.bytes += (int64_t)(n ? n : 16);
    return LFMM_OK;
}

// Unique keys of a sorted array (skipping `skip`): out[0..m), first[0..m] (first[m] = n),
// m on the host.  flag / pos: n + 1 ints of scratch; sums: scan_tmp_ints(n).
int unique_runs(const uint64_t* key, int64_t n, uint64_t skip, uint64_t* out, int32_t* first, int32_t* flag,
                int32_t* pos, int32_t* sums, int* m_host, cudaStream_t s) {
    if (n == 0) {
        *m_host = 0;
        if (first) LFMM_CUDA_TRY(cudaMemsetAsync(first, 0, sizeof(int32_t), s));
        return LFMM_OK;
    }
    run_start_kernel<<<grid_of(n), kT, 0, s>>>(key, n, skip, flag);
    LFMM_CUDA_TRY(exscan(flag, pos, n, sums, s));
    run_compact_kernel<<<grid_of(n), kT, 0, s>>>(key, n, flag, pos, out, first);
    LFMM_CUDA_TRY(cudaGetLastError());
    int32_t h = 0;
    LFMM_CUDA_TRY(cudaMemcpyAsync(&h, pos + n, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    LFMM_CUDA_TRY(cudaStreamSynchronize(s));
    *m_host = h;
    return LFMM_OK;
}

// the compact id of every sorted target's leaf, eight lanes per leaf
__global__ void target_leaf_kernel(const int32_t* __restrict__ rl_t, const int32_t* __restrict__ rl_id, int64_t m,
                                   int32_t* __restrict__ t_leaf) {
    const int64_t n8 = ((int64_t)gridDim.x * blockDim.x) >> 3;
    for (int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 3; j < m; j += n8) {
        const int id = rl_id[j];
        for (int v = rl_t[j] + (threadIdx.x & 7); v < rl_t[j + 1]; v += 8) t_leaf[v] = id;
    }
}

}  // namespace

cudaError_t launch_target_leaves(const Forest& F, int32_t* t_leaf, cudaStream_t s) {
    target_leaf_kernel<<<grid_of(8 * F.n_leaves), kT, 0, s>>>(F.rl_t, F.rl_id, F.n_leaves, t_leaf);
    return cudaGetLastError();
}

int forest_build(Forest& F, const int32_t* src, const int64_t* soff_h, int64_t ns, const int32_t* tgt,
                 const int64_t* toff_h, int64_t nt, int np, int leaf_size, int max_leaf_side, bool wide,
                 const ForestHint* hint, cudaStream_t s, PhaseTimer* timer) {
    int st;
    F.np = np;
    F.ns = ns;
    F.nt = nt;
    if (ns > INT32_MAX / 2 || nt > INT32_MAX / 2) return fail(LFMM_EINVAL, "forest too large");
    void* v;
    // targets = sources (same counts, offsets and coordinates): one sort serves both sides
    bool same = ns == nt && std::equal(soff_h, soff_h + np + 1, toff_h);
    // problem offsets and per-point problem ids (temporaries; none with one problem)
    DevBuf offs, pids;
    if ((st = offs.get((size_t)2 * (np + 1) * sizeof(int64_t) + 16, s))) return st;
    int64_t* soff = (int64_t*)offs.ptr;
    int64_t* toff = soff + (np + 1);
    int* word = (int*)(toff + (np + 1));  // the coordinate comparison's flag
    int32_t *spid = nullptr, *tpid = nullptr;
    std::vector<int4> hbb(np);
    const bool compare = same && src != tgt && !(hint && hint->same >= 0);
    if (hint && hint->same >= 0) same = same && hint->same == 1;
    if (compare) {
        LFMM_CUDA_TRY(cudaMemsetAsync(word, 0, sizeof(int), s));
        same_points_kernel<<<grid_of(ns), kT, 0, s>>>((const int2*)src, (const int2*)tgt, ns, word);
        timer->add_launches(1);
    }
    int* hw = readback_words();  // page-locked words for the readbacks, or ordinary ones
    std::vector<int> pageable;
    if (!hw) {
        pageable.resize(kReadbackWords);
        hw = pageable.data();
    }
    if (hint) {  // one problem, its box known
        hbb[0] = make_int4(hint->x0, hint->y0, hint->x1, hint->y1);
        if (compare) {
            LFMM_CUDA_TRY(cudaMemcpyAsync(hw, word, sizeof(int), cudaMemcpyDeviceToHost, s));
            LFMM_CUDA_TRY(cudaStreamSynchronize(s));
            same = hw[0] == 0;
        }
    } else {
        // bounding boxes first (int4: 16-byte aligned at the allocation's start), then the ids
        if ((st = pids.get((size_t)np * sizeof(int4) + (size_t)(np > 1 ? ns + nt : 0) * sizeof(int32_t), s))) return st;
        int4* bb = (int4*)pids.ptr;
        if (np == 1) {
            LFMM_CUDA_TRY(launch_set4((int*)bb, INT_MAX, INT_MAX, INT_MIN, INT_MIN, s));
            LFMM_CUDA_TRY(launch_bbox(src, ns, tgt, nt, (int*)bb, s));
        } else {
            LFMM_CUDA_TRY(cudaMemcpyAsync(soff, soff_h, (np + 1) * sizeof(int64_t), cudaMemcpyHostToDevice, s));
            LFMM_CUDA_TRY(cudaMemcpyAsync(toff, toff_h, (np + 1) * sizeof(int64_t), cudaMemcpyHostToDevice, s));
            spid = (int32_t*)(bb + np);
            tpid = spid + ns;
            pid_kernel<<<std::min(np, 152 * 8), kT, 0, s>>>(soff, np, spid);
            pid_kernel<<<std::min(np, 152 * 8), kT, 0, s>>>(toff, np, tpid);
            bbox_forest_kernel<<<std::min(np, 152 * 8), kT, 0, s>>>((const int2*)src, soff, (const int2*)tgt, toff, np,
                                                                   bb);
        }
        LFMM_CUDA_TRY(cudaGetLastError());
        timer->add_launches(np == 1 ? 2 : 3);
        LFMM_CUDA_TRY(cudaMemcpyAsync(hbb.data(), bb, np * sizeof(int4), cudaMemcpyDeviceToHost, s));
        if (compare) LFMM_CUDA_TRY(cudaMemcpyAsync(hw, word, sizeof(int), cudaMemcpyDeviceToHost, s));
        LFMM_CUDA_TRY(cudaStreamSynchronize(s));
        if (compare) same = hw[0] == 0;
    }
    F.x0.resize(np);
    F.y0.resize(np);
    F.K.resize(np);
    int Kmax = 0;
    for (int p = 0; p < np; ++p) {
        const int4 b = hbb[p];
        if (b.x > b.z) return fail(LFMM_EINVAL, "forest problem " + std::to_string(p) + " has no points");
        F.x0[p] = b.x;
        F.y0[p] = b.y;
        const int64_t ext = std::max((int64_t)b.z - b.x, (int64_t)b.w - b.y) + 1;
        if (ext > ((int64_t)1 << 30)) return fail(LFMM_EINVAL, "points span more than 2^30 lattice cells");
        F.K[p] = ceil_log2(ext);
        Kmax = std::max(Kmax, F.K[p]);
    }
    const int pbits = ceil_log2(std::max(np, 1));
    if ((st = alloc(F, &v, (size_t)3 * np * sizeof(int32_t), s))) return st;
    int32_t* dx0 = (int32_t*)v;
    int32_t* dy0 = dx0 + np;
    int32_t* dL = dy0 + np;
    F.d_L = dL;
    std::vector<int32_t> xyl((size_t)3 * np);  // x0, y0, L of every problem: one upload
    std::copy(F.x0.begin(), F.x0.end(), xyl.begin());
    std::copy(F.y0.begin(), F.y0.end(), xyl.begin() + np);

    // sorting scratch, sized for the largest sort of this phase (the union of source and
    // target leaves)
    const int64_t nmax = std::max<int64_t>({ns, nt, 1});
    const int64_t nsort = 2 * nmax;
    DevBuf kv, sb, runs;
    // sorted source keys / values, target keys / values, and one spare pair of 2 nmax
    if ((st = kv.get((size_t)4 * nmax * (sizeof(uint64_t) + sizeof(uint32_t)), s))) return st;
    uint64_t* sk = (uint64_t*)kv.ptr;      // source keys
    uint64_t* tk = sk + nmax;              // target keys
    uint64_t* kspare = sk + 2 * nmax;      // 2 nmax
    uint32_t* sv = (uint32_t*)(sk + 4 * nmax);
    uint32_t* tv = sv + nmax;
    SortBufs sbuf;
    const int64_t hist_ints = sort_hist_ints(nsort);
    if ((st = sb.get((size_t)(nsort * (sizeof(uint64_t) + sizeof(uint32_t))) +
                         (size_t)(hist_ints + scan_tmp_ints(hist_ints)) * sizeof(int32_t), s)))
        return st;
    sbuf.k2 = (uint64_t*)sb.ptr;
    sbuf.v2 = (uint32_t*)(sbuf.k2 + nsort);
    sbuf.hist = (int32_t*)(sbuf.v2 + nsort);
    sbuf.sums = sbuf.hist + hist_ints;
    // run scratch: flags, positions, firsts (n + 1 each), scan sums, two words, unique keys
    if ((st = runs.get((size_t)(3 * (nsort + 1) + scan_tmp_ints(nsort) + 2) * sizeof(int32_t) +
                           (size_t)(nsort + 1) * sizeof(uint64_t) + 16, s)))
        return st;
    int32_t* flag = (int32_t*)runs.ptr;
    int32_t* pos = flag + (nsort + 1);
    int32_t* first = pos + (nsort + 1);
    int32_t* ssum = first + (nsort + 1);
    int* mx = (int*)(ssum + scan_tmp_ints(nsort));
    uint64_t* ukeys = (uint64_t*)(((uintptr_t)(mx + 2) + 15) & ~(uintptr_t)15);  // unique keys

    // ---- 1. leaf side: the largest power of two <= max_leaf_side (and <= every root that
    // needs splitting) at which no leaf of any problem holds more than leaf_size points.
    // A candidate is checked on each problem's dense leaf grid when the grids are small,
    // else on sorted leaf keys (runs of equal keys are leaves), which then serve as the
    // point order.
    int ls = ceil_log2(max_leaf_side);
    if ((1 << ls) > max_leaf_side) --ls;
    ls = std::min(ls, Kmax);
    int maxs = 0, maxt = 0, kb = 1;
    bool dense = false;             // the final side was checked on dense grids (kept in cbk)
    DevBuf cbk;
    int64_t cells_k = 0;
    auto sort_side = [&](bool is_src, int bits, int* maxrun) -> int {
        const int64_t n = is_src ? ns : nt;
        uint64_t* k = is_src ? sk : tk;
        uint32_t* vv = is_src ? sv : tv;
        leaf_key_kernel<<<grid_of(n), kT, 0, s>>>((const int2*)(is_src ? src : tgt), n, is_src ? spid : tpid, dx0, dy0,
                                                  ls, kb, k, vv);
        LFMM_CUDA_TRY(cudaGetLastError());
        LFMM_CUDA_TRY(radix_sort(k, vv, n, bits, sbuf, s));
        timer->add_launches(1 + 5 * ((bits + 7) / 8));
        if (!maxrun) return LFMM_OK;
        int m = 0;
        int r;
        if ((r = unique_runs(k, n, ~0ull, ukeys, first, flag, pos, ssum, &m, s))) return r;
        LFMM_CUDA_TRY(cudaMemsetAsync(mx, 0, sizeof(int), s));
        max_run_kernel<<<grid_of(m), kT, 0, s>>>(first, m, mx);
        LFMM_CUDA_TRY(cudaMemcpyAsync(maxrun, mx, sizeof(int), cudaMemcpyDeviceToHost, s));
        LFMM_CUDA_TRY(cudaStreamSynchronize(s));
        timer->add_launches(5);
        return LFMM_OK;
    };
    for (;;) {
        F.L.assign(np, 0);
        int Lmax = 0;
        int64_t cells = 0;
        std::vector<int64_t> cell_off(np + 1, 0);
        for (int p = 0; p < np; ++p) {
            F.L[p] = std::max(0, F.K[p] - ls);
            Lmax = std::max(Lmax, F.L[p]);
            cell_off[p] = cells;
            cells += (int64_t)1 << (2 * F.L[p]);
        }
        cell_off[np] = cells;
        kb = std::max(1, Lmax);
        if (Lmax > 20 || pbits + 2 * kb + 7 > 63)
            return fail(LFMM_EUNSUPPORTED, "forest problem needs more than 2^20 leaves per side");
        std::copy(F.L.begin(), F.L.end(), xyl.begin() + 2 * np);
        LFMM_CUDA_TRY(cudaMemcpyAsync(dx0, xyl.data(), xyl.size() * sizeof(int32_t), cudaMemcpyHostToDevice, s));
        const int bits = pbits + 2 * kb;
        dense = cells <= std::max<int64_t>(2 * (ns + nt), (int64_t)1 << 22);
        DevBuf cb;
        if (dense) {
            if ((st = cb.get((size_t)(np + 1) * sizeof(int64_t) + (size_t)2 * cells * sizeof(int32_t) + 16, s))) return st;
            int64_t* doff = (int64_t*)cb.ptr;
            int32_t* cnt = (int32_t*)(doff + np + 1);
            LFMM_CUDA_TRY(cudaMemcpyAsync(doff, cell_off.data(), (np + 1) * sizeof(int64_t), cudaMemcpyHostToDevice, s));
            LFMM_CUDA_TRY(cudaMemsetAsync(cnt, 0, (size_t)2 * cells * sizeof(int32_t), s));
            LFMM_CUDA_TRY(cudaMemsetAsync(mx, 0, 2 * sizeof(int), s));
            dense_count_kernel<<<grid_of(ns), kT, 0, s>>>((const int2*)src, ns, spid, dx0, dy0, dL, doff, ls, cnt);
            max_count_kernel<<<grid_of(cells), kT, 0, s>>>(cnt, cells, mx);
            if (!same) {
                dense_count_kernel<<<grid_of(nt), kT, 0, s>>>((const int2*)tgt, nt, tpid, dx0, dy0, dL, doff, ls,
                                                             cnt + cells);
                max_count_kernel<<<grid_of(cells), kT, 0, s>>>(cnt + cells, cells, mx + 1);
            }
            LFMM_CUDA_TRY(cudaGetLastError());
            LFMM_CUDA_TRY(cudaMemcpyAsync(hw, mx, 2 * sizeof(int), cudaMemcpyDeviceToHost, s));
            LFMM_CUDA_TRY(cudaStreamSynchronize(s));
            timer->add_launches(same ? 2 : 4);
            maxs = hw[0];
            maxt = same ? hw[0] : hw[1];
        } else {
            if ((st = sort_side(true, bits, &maxs))) return st;
            if (same) maxt = maxs;
            else if ((st = sort_side(false, bits, &maxt))) return st;
        }
        if (std::max(maxs, maxt) <= leaf_size || ls == 0) {
            if (dense) {  // keep the grids' offsets and counts for the counting sort
                std::swap(cbk.ptr, cb.ptr);
                cbk.s = s;
                cells_k = cells;
            }
            break;
        }
        --ls;
    }
    F.ls = ls;
    F.side = 1 << ls;
    F.kb = kb;
    F.max_src = maxs;
    F.max_tgt = maxt;
    const int kbits = pbits + 2 * kb;          // bits of a packed key
    int Lmax = 0;
    for (int p = 0; p < np; ++p) Lmax = std::max(Lmax, F.L[p]);
    // ---- 2. points in leaf order, occupied leaves with their first source and target
    void* vp;
    if ((st = alloc(F, &vp, (size_t)2 * (ns + (same ? 0 : nt)) * sizeof(int32_t), s))) return st;
    F.sloc = (int32_t*)vp;
    F.sperm = F.sloc + ns;
    F.tloc = same ? F.sloc : F.sperm + ns;
    F.tperm = same ? F.sperm : F.tloc + nt;
    int M = 0;
    // the number of leaves on the device; on the host it is known with the boxes below
    // (dense grids), or already (sorted keys)
    DevBuf gb, mbuf;
    const int32_t* M_d = nullptr;
    if (dense) {
        // counting sort on the grids: first slot of every leaf by one exclusive scan of the
        // counts, points placed by atomic cursors; occupied leaves by one compaction
        const int64_t cells = cells_k;
        if (cells > INT32_MAX / 2) return fail(LFMM_EUNSUPPORTED, "forest leaf grids too large");
        int64_t* doff = (int64_t*)cbk.ptr;
        int32_t* cs = (int32_t*)(doff + np + 1);
        int32_t* ct = same ? nullptr : cs + cells;
        const int64_t sc = scan_tmp_ints(cells);
        if ((st = gb.get((size_t)(4 * (cells + 1) + 2 * sc) * sizeof(int32_t), s))) return st;
        int32_t* ss = (int32_t*)gb.ptr;      // [cells + 1] first source of each leaf
        int32_t* ts = ss + (cells + 1);      // [cells + 1] first target (targets != sources)
        int32_t* gflag = ts + (cells + 1);
        int32_t* gpos = gflag + (cells + 1);
        int32_t* gsum = gpos + (cells + 1);
        // occupied leaves before the counts turn into cursors
        occupied_flag_kernel<<<grid_of(cells), kT, 0, s>>>(cs, ct, cells, gflag);
        LFMM_CUDA_TRY(exscan(gflag, gpos, cells, gsum, s));
        LFMM_CUDA_TRY(exscan(cs, ss, cells, gsum + sc, s));
        if (!same) LFMM_CUDA_TRY(exscan(ct, ts, cells, gsum + sc, s));
        M_d = gpos + cells;
        const int64_t cap = std::min<int64_t>(cells, same ? ns : ns + nt);  // leaves at most
        if ((st = alloc(F, &vp, (size_t)(cap + 1) * sizeof(uint64_t), s))) return st;
        F.rl_key = (uint64_t*)vp;
        if ((st = alloc(F, &vp, (size_t)(same ? 2 : 3) * (cap + 1) * sizeof(int32_t), s))) return st;
        F.rl_s = (int32_t*)vp;
        F.rl_id = F.rl_s + (cap + 1);
        F.rl_t = same ? F.rl_s : F.rl_id + (cap + 1);
        occupied_compact_kernel<<<grid_of(cells), kT, 0, s>>>(gflag, gpos, cells, doff, np, dL, kb, ss, same ? ss : ts,
                                                              F.rl_key, F.rl_s, F.rl_t);
        // the counts become cursors (each leaf's first slot), then the points are placed
        LFMM_CUDA_TRY(cudaMemcpyAsync(cs, ss, (size_t)cells * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
        dense_scatter_kernel<<<grid_of(ns), kT, 0, s>>>((const int2*)src, ns, spid, dx0, dy0, dL, doff, ls, cs, F.sloc,
                                                        F.sperm);
        if (!same) {
            LFMM_CUDA_TRY(cudaMemcpyAsync(ct, ts, (size_t)cells * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
            dense_scatter_kernel<<<grid_of(nt), kT, 0, s>>>((const int2*)tgt, nt, tpid, dx0, dy0, dL, doff, ls, ct,
                                                            F.tloc, F.tperm);
        }
        LFMM_CUDA_TRY(cudaGetLastError());
        timer->add_launches(16);
    } else {
        point_order_kernel<<<grid_of(ns), kT, 0, s>>>((const int2*)src, ns, sv, spid, dx0, dy0, ls, F.sloc, F.sperm);
        if (!same)
            point_order_kernel<<<grid_of(nt), kT, 0, s>>>((const int2*)tgt, nt, tv, tpid, dx0, dy0, ls, F.tloc, F.tperm);
        LFMM_CUDA_TRY(cudaGetLastError());
        if (same) {
            if ((st = alloc(F, &vp, (size_t)(ns + 1) * sizeof(uint64_t), s))) return st;
            F.rl_key = (uint64_t*)vp;
            if ((st = unique_runs(sk, ns, ~0ull, F.rl_key, nullptr, flag, pos, ssum, &M, s))) return st;
        } else {
            // unique source leaves and unique target leaves, merged by one more sort
            int mm = 0, mt = 0;
            if ((st = unique_runs(sk, ns, ~0ull, kspare, nullptr, flag, pos, ssum, &mm, s))) return st;
            if ((st = unique_runs(tk, nt, ~0ull, kspare + mm, nullptr, flag, pos, ssum, &mt, s))) return st;
            LFMM_CUDA_TRY(radix_sort(kspare, nullptr, (int64_t)mm + mt, kbits, sbuf, s));
            if ((st = alloc(F, &vp, (size_t)(mm + mt + 1) * sizeof(uint64_t), s))) return st;
            F.rl_key = (uint64_t*)vp;
            if ((st = unique_runs(kspare, (int64_t)mm + mt, ~0ull, F.rl_key, nullptr, flag, pos, ssum, &M, s))) return st;
        }
        if ((st = alloc(F, &vp, (size_t)(same ? 2 : 3) * (M + 1) * sizeof(int32_t), s))) return st;
        F.rl_s = (int32_t*)vp;
        F.rl_id = F.rl_s + (M + 1);
        F.rl_t = same ? F.rl_s : F.rl_id + (M + 1);
        leaf_ranges_kernel<<<grid_of(M + 1), kT, 0, s>>>(F.rl_key, M, sk, ns, same ? sk : tk, same ? ns : nt, F.rl_s,
                                                         F.rl_t);
        LFMM_CUDA_TRY(cudaGetLastError());
        timer->add_launches(12);
    }

    // ---- 3. boxes of every level
    F.kmax = Lmax - 2;  // may be negative: no far field anywhere
    const int nk = std::max(F.kmax, 0) + 1;
    const int kmx = std::max(F.kmax, 0);
    int64_t NB = 0;
    std::vector<int64_t> hc((size_t)4 * nk + 1);
    int64_t* dcls = nullptr;
    int32_t *bp_all = nullptr, *bxy_all = nullptr, *par_all = nullptr, *il_all = nullptr, *ch_all = nullptr,
            *leaf_rl = nullptr;
    // per-box records of all levels in one allocation (level k at box_off[k])
    int64_t* cstart = nullptr;
    auto alloc_records = [&]() -> int {
        int r;
        if ((r = alloc(F, &vp, (size_t)NB * (4 + 3 + 27) * sizeof(int32_t) + (size_t)M * sizeof(int32_t) +
                                   (size_t)(5 * nk) * sizeof(int64_t) + 16, s)))
            return r;
        ch_all = (int32_t*)vp;  // (16-byte records first)
        dcls = (int64_t*)(ch_all + 4 * NB);  // 5 nk, level-local class starts
        bp_all = (int32_t*)(dcls + 5 * nk);
        bxy_all = bp_all + NB;
        par_all = bxy_all + NB;
        il_all = par_all + NB;
        leaf_rl = il_all + 27 * NB;
        return LFMM_OK;
    };
    BitGrid G = {};
    int64_t words = 0;
    std::vector<uint32_t> goff;
    if (nk <= kGridLevels) {
        if (np > 1) goff.resize((size_t)nk * np);
        for (int k = 0; k < nk && words >= 0; ++k) {
            int64_t stride = 0;
            for (int p = 0; p < np; ++p) {
                if (np > 1) goff[(size_t)k * np + p] = (uint32_t)stride;
                if (k > 0 && F.L[p] - k < 2) continue;
                const int64_t h = std::max<int64_t>(1, ((int64_t)1 << (F.L[p] - k)) >> 1);
                stride += (h * h + 31) / 32;
            }
            G.base[k] = (uint32_t)words;
            G.stride[k] = (uint32_t)stride;
            words += 4 * stride;
            if (words > grid_words_max(ns + nt)) words = -1;
        }
    } else {
        words = -1;
    }
    DevBuf gbits, starts;
    if ((st = starts.get((size_t)(4 * nk + 1) * sizeof(int64_t) + (size_t)(4 * nk + 2) * sizeof(int), s))) return st;
    cstart = (int64_t*)starts.ptr;  // 4 nk + 1
    int* starts_out = (int*)(cstart + 4 * nk + 1);
    if (!dense) {
        if ((st = mbuf.get(sizeof(int32_t), s))) return st;
        LFMM_CUDA_TRY(cudaMemcpyAsync(mbuf.ptr, &M, sizeof(int32_t), cudaMemcpyHostToDevice, s));
        M_d = (const int32_t*)mbuf.ptr;
    }
    if (words > 0 && 4 * nk + 2 <= kReadbackWords) {
        // bits, running counts, scan sums, offsets
        const int64_t sc = scan_tmp_ints(words);
        if ((st = gbits.get((size_t)(2 * words + 1 + sc) * sizeof(int32_t) + goff.size() * sizeof(uint32_t), s))) return st;
        G.nk = nk;
        G.np = np;
        G.kmax = F.kmax;
        G.L = dL;
        G.bits = (uint32_t*)gbits.ptr;
        int32_t* before = (int32_t*)(G.bits + words);
        int32_t* wsum = before + words + 1;
        G.before = before;
        if (np > 1) {
            G.off = (const uint32_t*)(wsum + sc);
            LFMM_CUDA_TRY(cudaMemcpyAsync((void*)G.off, goff.data(), goff.size() * sizeof(uint32_t), cudaMemcpyHostToDevice, s));
        }
        LFMM_CUDA_TRY(cudaMemsetAsync(G.bits, 0, (size_t)words * sizeof(uint32_t), s));
        const int64_t cap = dense ? std::min<int64_t>(cells_k, ns + nt) : M;
        grid_set_kernel<<<grid_of(cap), kT, 0, s>>>(G, F.rl_key, M_d, kb);
        LFMM_CUDA_TRY(exscan<true>((const int32_t*)G.bits, before, words, wsum, s));
        DevBuf dc;  // (the level-local class starts, copied into the records once these exist)
        if ((st = dc.get((size_t)5 * nk * sizeof(int64_t), s))) return st;
        grid_starts_kernel<<<1, 128, 0, s>>>(G, words, M_d, cstart, (int64_t*)dc.ptr, starts_out);
        LFMM_CUDA_TRY(cudaGetLastError());
        LFMM_CUDA_TRY(cudaMemcpyAsync(hw, starts_out, (size_t)(4 * nk + 2) * sizeof(int), cudaMemcpyDeviceToHost, s));
        LFMM_CUDA_TRY(cudaStreamSynchronize(s));
        M = hw[0];
        for (int t = 0; t <= 4 * nk; ++t) hc[t] = hw[1 + t];
        NB = hc[4 * nk];
        if ((st = alloc_records())) return st;
        LFMM_CUDA_TRY(cudaMemcpyAsync(dcls, dc.ptr, (size_t)5 * nk * sizeof(int64_t), cudaMemcpyDeviceToDevice, s));
        grid_records_kernel<<<grid_of(words), kT, 0, s>>>(G, words, bp_all, bxy_all);
        grid_leaves_kernel<<<grid_of(M), kT, 0, s>>>(G, F.rl_key, M, kb, F.rl_id, leaf_rl);
        grid_links_kernel<<<grid_of(NB), kT, 0, s>>>(G, NB, cstart, bp_all, bxy_all, par_all, ch_all, il_all);
        LFMM_CUDA_TRY(cudaGetLastError());
        timer->add_launches(5 + exscan_launches(words));
    } else {
    if (dense) {  // the number of leaves
        LFMM_CUDA_TRY(cudaMemcpyAsync(hw, M_d, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
        LFMM_CUDA_TRY(cudaStreamSynchronize(s));
        M = hw[0];
    }
    // without the grids: A = the leaves (k = 0), then the boxes of levels
    // k = 1 .. kmax, sorted by (k, problem, row, column); compact ids number each level's
    // boxes in class-major order; links by search in A
    const int lbits = ceil_log2(nk);
    int E = 0, U = 0;
    DevBuf ebuf, abuf;
    // level >= 1 keys of the row-segment heads
    const int64_t nh = (int64_t)M * kmx;
    if (nh > INT32_MAX / 2) return fail(LFMM_EUNSUPPORTED, "tree too deep for the box lists");
    {
        DevBuf hb;
        if ((st = hb.get((size_t)(2 * (nh + 1) + scan_tmp_ints(nh)) * sizeof(int32_t), s))) return st;
        int32_t* hflag = (int32_t*)hb.ptr;
        int32_t* hpos = hflag + (nh + 1);
        int32_t* hsum = hpos + (nh + 1);
        if (nh > 0) {
            head_flag_kernel<<<grid_of(nh), kT, 0, s>>>(F.rl_key, M, kmx, dL, kb, hflag);
            LFMM_CUDA_TRY(exscan(hflag, hpos, nh, hsum, s));
            LFMM_CUDA_TRY(cudaMemcpyAsync(&E, hpos + nh, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
            LFMM_CUDA_TRY(cudaStreamSynchronize(s));
        }
        // A (M + E keys at most) and, past it, the emitted keys
        if ((st = abuf.get((size_t)(M + 2 * (int64_t)E + 1) * sizeof(uint64_t), s))) return st;
        if (E > 0) {
            head_key_kernel<<<grid_of(nh), kT, 0, s>>>(F.rl_key, M, kmx, kb, kbits, hflag, hpos,
                                                       (uint64_t*)abuf.ptr + M + E);
            LFMM_CUDA_TRY(cudaGetLastError());
        }
        timer->add_launches(5);
    }
    uint64_t* A = (uint64_t*)abuf.ptr;
    LFMM_CUDA_TRY(cudaMemcpyAsync(A, F.rl_key, (size_t)M * sizeof(uint64_t), cudaMemcpyDeviceToDevice, s));
    // scratch of the level sorts: E keys, then the class sort of all boxes
    const int64_t nlev = std::max<int64_t>((int64_t)M + E, 1);
    SortBufs lsb;
    const int64_t lh = sort_hist_ints(nlev);
    if ((st = ebuf.get((size_t)nlev * (2 * sizeof(uint64_t) + 2 * sizeof(uint32_t) + sizeof(int32_t)) +
                           (size_t)(lh + scan_tmp_ints(lh) + 3 * (nlev + 1) + scan_tmp_ints(nlev) + 8) * sizeof(int32_t),
                       s)))
        return st;
    uint64_t* ck = (uint64_t*)ebuf.ptr;
    lsb.k2 = ck + nlev;
    uint32_t* cidx = (uint32_t*)(lsb.k2 + nlev);
    lsb.v2 = cidx + nlev;
    int32_t* local_of = (int32_t*)(lsb.v2 + nlev);
    lsb.hist = local_of + nlev;
    lsb.sums = lsb.hist + lh;
    int32_t* lflag = lsb.sums + scan_tmp_ints(lh);
    int32_t* lpos = lflag + (nlev + 1);
    int32_t* lsum = lpos + (nlev + 1);
    if (E > 0) {
        uint64_t* ek = A + M + E;
        LFMM_CUDA_TRY(radix_sort(ek, nullptr, E, kbits + lbits, lsb, s));
        if ((st = unique_runs(ek, E, ~0ull, A + M, nullptr, lflag, lpos, lsum, &U, s))) return st;
        timer->add_launches(4 + 5 * ((kbits + lbits + 7) / 8));
    }
    NB = (int64_t)M + U;
    // class-major order of every level (4 nk <= 84 partition keys: one digit)
    class_key_kernel<<<grid_of(NB), kT, 0, s>>>(A, NB, kb, kbits, ck, cidx);
    LFMM_CUDA_TRY(cudaGetLastError());
    LFMM_CUDA_TRY(radix_pass(ck, cidx, lsb.k2, lsb.v2, NB, 0, lsb, s));
    std::swap(ck, lsb.k2);
    std::swap(cidx, lsb.v2);
    if ((st = alloc_records())) return st;
    class_starts_kernel<<<(4 * nk + 1 + kT - 1) / kT, kT, 0, s>>>(ck, NB, nk, cstart);
    box_records_kernel<<<grid_of(NB), kT, 0, s>>>(A, ck, cidx, NB, cstart, kb, kbits, bp_all, bxy_all, local_of, leaf_rl);
    // the [first, end) of every box row of A, so that the links' searches (parent, two child
    // rows, six neighbour rows per box) cover one row instead of all of A; without it (a
    // table far larger than the boxes) they search all of A
    DevBuf rowbuf;
    const int2* rows = nullptr;
    const int64_t* row_off = nullptr;
    {
        std::vector<int64_t> ro((size_t)nk * np + 1, 0);
        int64_t R = 0;
        for (int k = 0; k < nk; ++k)
            for (int p = 0; p < np; ++p) {
                ro[(size_t)k * np + p] = R;
                if (F.L[p] >= k) R += (int64_t)1 << (F.L[p] - k);
            }
        ro[(size_t)nk * np] = R;
        if (R <= 8 * NB + ((int64_t)1 << 20)) {
            if ((st = rowbuf.get((size_t)R * sizeof(int2) + ro.size() * sizeof(int64_t) + 16, s))) return st;
            int2* rt = (int2*)rowbuf.ptr;
            int64_t* ro_d = (int64_t*)(rt + R);
            LFMM_CUDA_TRY(cudaMemsetAsync(rt, 0, (size_t)R * sizeof(int2), s));
            LFMM_CUDA_TRY(cudaMemcpyAsync(ro_d, ro.data(), ro.size() * sizeof(int64_t), cudaMemcpyHostToDevice, s));
            row_range_kernel<<<grid_of(NB), kT, 0, s>>>(A, NB, kb, kbits, np, ro_d, rt);
            rows = rt;
            row_off = ro_d;
            timer->add_launches(1);
        }
    }
    links_kernel<<<grid_of(NB), kT, 0, s>>>(NB, ck, A, NB, local_of, bp_all, bxy_all, dL, kb, kbits, F.kmax, rows,
                                            row_off, np, par_all, ch_all, il_all);
    LFMM_CUDA_TRY(cudaGetLastError());
    LFMM_CUDA_TRY(cudaMemcpyAsync(F.rl_id, local_of, (size_t)M * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
    timer->add_launches(4 + 5);
    LFMM_CUDA_TRY(cudaMemcpyAsync(hc.data(), cstart, hc.size() * sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    LFMM_CUDA_TRY(cudaStreamSynchronize(s));
    std::vector<int64_t> hl((size_t)5 * nk);
    for (int k = 0; k < nk; ++k)
        for (int c = 0; c <= 4; ++c) hl[5 * k + c] = hc[4 * k + c] - hc[4 * k];
    LFMM_CUDA_TRY(cudaMemcpyAsync(dcls, hl.data(), hl.size() * sizeof(int64_t), cudaMemcpyHostToDevice, s));
    LFMM_CUDA_TRY(cudaStreamSynchronize(s));  // hl is a local
    }
    F.n_leaves = M;
    // class ranges of every level
    {
        F.levels.assign(nk, ForestLevel());
        for (int k = 0; k < nk; ++k) {
            ForestLevel& lv = F.levels[k];
            lv.box_off = hc[4 * k];
            lv.nb = hc[4 * k + 4] - hc[4 * k];
            for (int c = 0; c <= 4; ++c) lv.cls[c] = hc[4 * k + c] - lv.box_off;
            lv.d_cls = dcls + 5 * k;
            lv.bp = bp_all + lv.box_off;
            lv.bxy = bxy_all + lv.box_off;
            lv.par = par_all + lv.box_off;
            lv.il = il_all + 27 * lv.box_off;
            lv.ch = k >= 1 ? ch_all + 4 * lv.box_off : nullptr;
            lv.rl = k == 0 ? leaf_rl : nullptr;
        }
        F.total_boxes = NB;
    }

    // ---- 4. strips of the near-field sweep
    const int msr = std::max(1, maxs), mtg = std::max(1, maxt);
    const int SW = std::min({kStripMaxSW, kStripCapSrc / (3 * msr) - 2, kStripCapTgt / mtg});
    if (SW < 1) return fail(LFMM_EUNSUPPORTED, "leaves too full for the near-field staging (" + std::to_string(msr) +
                                                   " sources / " + std::to_string(mtg) + " targets)");
    // (the same leaves are refused whatever the element type)
    F.SW = wide ? std::min({kStripMaxSW, near8_caps(F.side) / (3 * msr) - 2, kStripCapTgt / mtg}) : SW;
    {
        strip_flag_kernel<<<grid_of(M), kT, 0, s>>>(F.rl_key, F.rl_t, M, kb, F.SW, flag);
        LFMM_CUDA_TRY(exscan(flag, pos, M, ssum, s));
        const size_t n4 = (size_t)std::max(M, 1);  // strips at most; their number stays on the device
        if ((st = alloc(F, &vp, 3 * n4 * sizeof(int4) + 16, s))) return st;
        F.strips = (int4*)vp;
        F.strip_rows = F.strips + n4;
        F.n_strips_d = (int32_t*)(F.strip_rows + 2 * n4);
        F.n_strips = M;
        LFMM_CUDA_TRY(cudaMemcpyAsync(F.n_strips_d, pos + M, sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
        strip_record_kernel<<<grid_of(M), kT, 0, s>>>(F.rl_key, flag, pos, M, kb, F.SW, F.strips);
        strip_rows_kernel<<<grid_of(M), kT, 0, s>>>(F.strips, F.n_strips_d, F.rl_key, M, dL, kb, F.SW, F.strip_rows);
        LFMM_CUDA_TRY(cudaGetLastError());
        timer->add_launches(3 + exscan_launches(M));
    }
    return LFMM_OK;  // temporaries are freed in stream order
}

}  // namespace lfmm
