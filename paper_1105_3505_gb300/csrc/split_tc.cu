// M2M, M2L and L2L of the binary64-accurate paths on the 5th-generation tensor cores
// (Sec. 7, Sec. 8.2 steps 2-4), P_pad 64.
//
// The tensor cores have no 48- or 53-bit product, but they form sums of small integers
// exactly.  A row of expansions (and an operator matrix) is scaled by a power of two to
// |x| <= 1 and cut into six slices of nine bits,
//
//     x = sum_i a_i 2^(-8 - 9 i),   a_i integer, |a_i| <= 256,   i = 0 .. 5,
//
// 53 bits of the row's (operator's) largest entry, each slice exact in fp16; an entry 2^-k of
// the largest keeps 53 - k.  A product of two slices is at most 2^16, a sum
// over the 64 coefficients at most 2^22, and the products of equal weight (i + j = g) are
// added in one fp32 accumulator: up to four of them stay below 2^24, exact whatever the
// accumulator's rounding; five and more occur only from g = 4 on, 36 bits below the leading
// weight.  (The splitting follows the error-free matrix products of Ozaki, Ogita, Oishi and
// Rump, Numer. Algorithms 59 (2012), with power-of-two scaling per row.)  Of the 36 products
// float-float forms those of g <= 5 (21, error about 2^-51 of the largest term), binary64 those
// of g <= 6 (26, 2^-60).  Rows for the level below that come out under 2^-100 of their reference
// (sums that cancel to their rounding) are taken for zero.
//
// One kernel does the three translations; a work item is 128 target boxes (TMEM lanes) and
// a chunk of the steps of their sums: 27 interaction offsets (M2L, boxes of one parity
// class), four children (M2M) or the parent (L2L).  Per step
//   warps 8-9   gather the 128 sliced source rows by box list, slice by slice, into a ring
//               of six 16 KB stages (16-byte cp.async into the 128-byte swizzle, one
//               64-coefficient row of a slice being exactly 128 bytes); lane 0 of warp 8
//               also fetches the step's 48 KB sliced operator by a bulk copy (two stages);
//   warp 10     issues, per slice i of the sources, the MMAs with slices 0 .. 5 - i of the
//               operator: consecutive slices land in consecutive accumulators, so they are
//               one MMA with N up to 256;
//   warps 0-7   read the accumulators back (a row's 64 outputs over two warps), join the
//               weights by exact additions and add the step into float pairs (triples for
//               binary64) relative to the row's largest source exponent;
//   warp 11     sums the compensated charge / constant channel of the boxes.
// Every level's M2L is independent of the others', so all levels share one launch; the
// downward pass that follows adds the chunks' sums and the parent's contribution level by
// level, and writes the rows sliced again for the level below.
// Every wait is bounded; on expiry LFMM_ETIMEOUT is recorded, the roles run out without
// waiting, and the teardown waits (bounded) for the copies and MMAs in flight.
//
// What bounds it: a step needs 2,700 tensor cycles (128 x 64 x 64 x 21 products) and 1,900
// for the read-back, one after the other because the accumulators of a step fill 384 (448)
// of the 512 TMEM columns; the float-float products on the FP32 pipes that it replaces took
// 61,000 cycles a step, the binary64 ones 262,000.  Measured (ncu, cold caches): the M2L of
// 400,009 points at leaf size 128, float-float p = 16 (8.4 k boxes) 942 -> 108 us, of 178 k
// clustered points 1,713 -> 151 us, of 100 k points in binary64 1,137 -> 54 us.  Those
// figures are with the producers reading each row's index between two copies (10,500 cycles
// a step, clock64 trace); reading a step's indices first, adding the chunks once instead of
// in the downward pass, and small_level_kernel for levels of few boxes (28 and 18 us a
// level as tensor-core launches) then took eval_df_400k from 968 to 806 us, eval_fp64_100k
// 636 -> 488, request_178k_1e10 1,456 -> 1,159 and a disk's Krylov iteration 387 -> 188 us.
// Errors against the exact sum, these translations against those on the CUDA cores in the
// path's own arithmetic, everything else alike (geometric means over twelve inputs each, sizes,
// orders and leaves over the range in use): kept plans in float-float 8.2e-14 against 8.4e-14,
// in binary64 1.031e-13 against 1.037e-13 (truncation of the expansions), clustered and
// uniform requests 4.3e-14 against 4.8e-14, a disk's double layer 1.9e-13 against 3.9e-13.
#include "split_tc.h"

#include <cuda_fp16.h>

#include <type_traits>

#include "device_common.h"
#include "tc_common.h"

namespace lfmm {

namespace {

enum { kM2L = 0, kM2M = 1, kL2L = 2 };

constexpr int kARing = 6, kBRing = 2;
constexpr uint32_t kABytes = 128 * 128;
constexpr int kSgThreads = 384;  // three warps per scheduler: 168 registers a thread for the read-back
constexpr int kSrcInts = 128 * 28;  // source rows of an item: 128 boxes x 28 steps
constexpr int kExpShorts = 128 * 28;
constexpr size_t kSgSmem = 1024 + (size_t)kARing * kABytes + (size_t)kBRing * kSgTileBytes +
                           (size_t)kSrcInts * 4 + (size_t)kExpShorts * 2;
static_assert(kSgSmem <= 227 * 1024, "split ring exceeds shared memory");

// exponents of sliced rows and operators: |x| <= 2^e
constexpr int kExpZero = -30000;  // all coefficients zero
constexpr int kExpNan = 30000;    // an infinity or NaN among them: everything they reach is NaN

// NC floats per accumulated value; G - 1 accumulators (weights g = 0 .. G - 2)
template <typename T>
struct SgT;
template <>
struct SgT<DF> {
    static constexpr int NC = 2, G = 7, COLS = 8;
};
template <>
struct SgT<double> {
    static constexpr int NC = 3, G = 8, COLS = 4;
};

struct SgLevel {
    const int32_t* list;   // compact: il [27], ch [4] or par [1] of each box
    const uint8_t* src;    // sliced rows of the sources' level
    const int32_t* src_e;  // and their exponents
    const uint8_t* tiles;  // the level's sliced operators
    const int32_t* tile_e;
    const void* mono;      // M2L: deflation constants
    const void* Qin;       // M2L: charges of the level; M2M: of the children
    int64_t out0;          // first row of the level in the outputs
    int lg;                // uniform form: log2 of the boxes per side; -1: compact
};

struct SgParams {
    SgLevel lv[kSgMaxLevels];
    int64_t first[4 * kSgMaxLevels];  // per (level, class): first box (compact form)
    int count[4 * kSgMaxLevels];
    int tile_end[4 * kSgMaxLevels];
    int n_seg, n_items, n_chunks, has_par;
    float* part;        // [chunk][row][NC][64] sums of the M2L steps (L2L: chunk 0, the whole sum)
    int32_t* part_e;    // [chunk][row]
    void* cpart;        // [chunk][row]
    int64_t part_rows;
    uint8_t* dst;       // sliced rows out (null: none)
    int32_t* dst_e;
    int64_t dst0;       // first row of the level there
    void* u;            // the level's rows of T out (null: none)
    void* Cout;         // M2M: charges out; L2L: constants out
    const void* Cpar;
};

__device__ __forceinline__ float pow2f(int e) {  // 2^e, 0 below the normal range
    return e < -126 ? 0.f : __int_as_float((min(e, 127) + 127) << 23);
}

template <int N>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, float (&v)[N]);
template <>
__device__ __forceinline__ void tmem_ld<8>(uint32_t taddr, float (&v)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "r"(taddr)
                 : "memory");
}
template <>
__device__ __forceinline__ void tmem_ld<4>(uint32_t taddr, float (&v)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
                 : "r"(taddr)
                 : "memory");
}

__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

// v (NC floats, decreasing) * 2^8 cut into slices: digit() takes the next one
template <int NC>
__device__ __forceinline__ float next_digit(float (&v)[NC]) {
    const float a = rintf(v[0]);
    v[0] -= a;
#pragma unroll
    for (int c = 0; c + 1 < NC; ++c) {
        const DF t = two_sum(v[c], v[c + 1]);
        v[c] = t.hi;
        v[c + 1] = t.lo;
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) v[c] *= 512.f;
    return a;
}

// 2^-e x and the exponent e of a row from the largest magnitude's bits
__device__ __forceinline__ int row_exp(uint32_t mx) {
    if (mx == 0) return kExpZero;
    if (mx >= 0x7f800000u) return kExpNan;
    return max((int)(mx >> 23) - 126, -126);
}

// Slices of one row of T (64 coefficients, two per lane of a warp) and its exponent.
template <typename T>
__device__ __forceinline__ void slice_row(const T (&x)[2], int lane, uint8_t* __restrict__ dst,
                                          int32_t* __restrict__ dst_e) {
    uint32_t w[kSgSlices];
    int e;
    if constexpr (std::is_same<T, DF>::value) {
        uint32_t mx = max(__float_as_uint(x[0].hi) & 0x7fffffffu, __float_as_uint(x[1].hi) & 0x7fffffffu);
        mx = __reduce_max_sync(kFull, mx);
        e = row_exp(mx);
        const bool dead = abs(e) >= kExpNan;
        float v[2][2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            v[i][0] = dead ? 0.f : ldexpf(x[i].hi, 8 - e);
            v[i][1] = dead ? 0.f : ldexpf(x[i].lo, 8 - e);
        }
#pragma unroll
        for (int s = 0; s < kSgSlices; ++s) {
            const __half2 h = __floats2half2_rn(next_digit(v[0]), next_digit(v[1]));
            w[s] = *reinterpret_cast<const uint32_t*>(&h);
        }
    } else {
        uint32_t mx = max((uint32_t)__double2hiint(x[0]) & 0x7fffffffu, (uint32_t)__double2hiint(x[1]) & 0x7fffffffu);
        if (mx == 0 && (x[0] != 0.0 || x[1] != 0.0)) mx = 1;
        mx = __reduce_max_sync(kFull, mx);
        e = mx == 0 ? kExpZero : mx >= 0x7ff00000u ? kExpNan : max((int)(mx >> 20) - 1022, -1022);
        const bool dead = abs(e) >= kExpNan;
        double v0 = dead ? 0.0 : ldexp(x[0], 8 - e), v1 = dead ? 0.0 : ldexp(x[1], 8 - e);
#pragma unroll
        for (int s = 0; s < kSgSlices; ++s) {
            const double a0 = rint(v0), a1 = rint(v1);
            v0 = (v0 - a0) * 512.0;
            v1 = (v1 - a1) * 512.0;
            const __half2 h = __floats2half2_rn((float)a0, (float)a1);
            w[s] = *reinterpret_cast<const uint32_t*>(&h);
        }
    }
    uint32_t* row = reinterpret_cast<uint32_t*>(dst);
#pragma unroll
    for (int s = 0; s < kSgSlices; ++s) row[32 * s + lane] = w[s];
    if (lane == 0) *dst_e = e;
}

// Slices of nb rows of T, a warp per row.
template <typename T>
__global__ void __launch_bounds__(256) slice_rows_kernel(const T* __restrict__ x, int64_t nb, uint8_t* __restrict__ dst,
                                                         int32_t* __restrict__ dst_e) {
    griddep_wait();
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; b < nb; b += nw) {
        const VecT<T, 2> p = *reinterpret_cast<const VecT<T, 2>*>(x + b * 64 + 2 * lane);
        slice_row(p.v, lane, dst + b * kSgRowBytes, dst_e + b);
    }
}

// Sliced image of one operator, op[q][p] (input q, output p, 64 x 64): per slice 64 output
// rows of 128 bytes (64 inputs), 128-byte swizzle.  blockIdx.x: the operator.
struct SgOpList {
    const void* op[kSgOps];
};
template <typename T>
__global__ void __launch_bounds__(256) slice_ops_kernel(const SgOpList ops, uint8_t* __restrict__ tiles,
                                                        int32_t* __restrict__ tile_e) {
    const T* op = (const T*)ops.op[blockIdx.x];
    uint8_t* tile = tiles + (size_t)blockIdx.x * kSgTileBytes;
    __shared__ double s_mx[8];
    double mx = 0.0;
    if (op)
        for (int i = threadIdx.x; i < 64 * 64; i += 256) mx = fmax(mx, fabs((double)op[i]));
    for (int o = 16; o; o >>= 1) mx = fmax(mx, __shfl_xor_sync(kFull, mx, o));
    if ((threadIdx.x & 31) == 0) s_mx[threadIdx.x >> 5] = mx;
    __syncthreads();
    for (int w = 0; w < 8; ++w) mx = fmax(mx, s_mx[w]);
    int e = 0;
    if (mx > 0.0) frexp(mx, &e);  // mx < 2^e
    for (int i = threadIdx.x; i < 64 * 64; i += 256) {
        const int n = i >> 6, k = i & 63;
        double v = op ? ldexp((double)op[k * 64 + n], 8 - e) : 0.0;
        for (int s = 0; s < kSgSlices; ++s) {
            const double a = rint(v);
            v = (v - a) * 512.0;
            *reinterpret_cast<__half*>(tile + s * 8192 + n * 128 + (((k >> 3) ^ (n & 7)) << 4) + (k & 7) * 2) =
                __float2half_rn((float)a);
        }
    }
    if (threadIdx.x == 0) tile_e[blockIdx.x] = e;
}

// One value's weights a[0] .. a[G - 2] (integers) joined and added, scaled, into acc:
// sum_g a[g] 2^(-9 g) c 2^18 is what is added (c in units of weight 2).
__device__ __forceinline__ void join_add(const float (&a)[6], float c, float (&acc)[2]) {
    const float s1 = fmaf(a[0], 512.f, a[1]);
    const float e1 = fmaf(a[0], 512.f, -s1) + a[1];
    const float s2 = fmaf(s1, 512.f, a[2]);
    const float e2 = fmaf(s1, 512.f, -s2) + a[2];
    const float lo = fmaf(fmaf(a[3], 512.f, a[4]), 512.f, a[5]);
    const float l = fmaf(lo, 0x1p-27f, fmaf(e1, 512.f, e2));
    const DF t = two_sum(acc[0], s2 * c);
    acc[0] = t.hi;
    acc[1] = fmaf(l, c, acc[1] + t.lo);
}
__device__ __forceinline__ void join_add(const float (&a)[7], float c, float (&acc)[3]) {
    const float s1 = fmaf(a[0], 512.f, a[1]);
    const float e1 = fmaf(a[0], 512.f, -s1) + a[1];
    const float s2 = fmaf(s1, 512.f, a[2]);
    const float e2 = fmaf(s1, 512.f, -s2) + a[2];
    const float m = fmaf(e1, 512.f, e2);
    const float t1 = fmaf(a[3], 512.f, a[4]);
    const float f1 = fmaf(a[3], 512.f, -t1) + a[4];
    const float t2 = fmaf(t1, 512.f, a[5]);
    const float f2 = fmaf(t1, 512.f, -t2) + a[5];
    const float r = fmaf(a[6], 0x1p-9f, fmaf(f1, 512.f, f2));
    const float c27 = c * 0x1p-27f;
    DF x = two_sum(acc[0], s2 * c);
    acc[0] = x.hi;
    DF y = two_sum(acc[1], x.lo);
    DF z = two_sum(y.hi, m * c);
    DF w = two_sum(z.hi, t2 * c27);
    acc[1] = w.hi;
    acc[2] += (y.lo + z.lo) + fmaf(r, c27, w.lo);
}
__device__ __forceinline__ void renorm(float (&v)[2]) {
    const DF t = fast_two_sum(v[0], v[1]);
    v[0] = t.hi;
    v[1] = t.lo;
}
__device__ __forceinline__ void renorm(float (&v)[3]) {
    DF t = two_sum(v[1], v[2]);
    DF h = two_sum(v[0], t.hi);
    DF m = two_sum(h.lo, t.lo);
    v[0] = h.hi;
    v[1] = m.hi;
    v[2] = m.lo;
}
__device__ __forceinline__ void add_scaled(float (&v)[2], const float (&x)[2], float f) {
    const DF t = two_sum(v[0], x[0] * f);
    v[0] = t.hi;
    v[1] = fmaf(x[1], f, v[1] + t.lo);
}
__device__ __forceinline__ void add_scaled(float (&v)[3], const float (&x)[3], float f) {
    const DF t = two_sum(v[0], x[0] * f);
    v[0] = t.hi;
    DF y = two_sum(v[1], t.lo);
    DF z = two_sum(y.hi, x[1] * f);
    v[1] = z.hi;
    v[2] += (y.lo + z.lo) + x[2] * f;
}

// One work item: boxes [0, rows) of tile `pos0 ..` of a (level, class), steps [st0, st1).
struct Item {
    int lev, cls, rows, st0, st1, z;
    int64_t box0;  // compact: first box; uniform: first position in class order
};

template <int MODE>
__device__ __forceinline__ Item decode_item(const SgParams& P, const int* s_end, int item) {
    Item I;
    const int tile = item / P.n_chunks;
    I.z = item - tile * P.n_chunks;
    int s = 0;
    while (tile >= s_end[s]) ++s;
    const int t = tile - (s ? s_end[s - 1] : 0);
    I.lev = s >> 2;
    I.cls = s & 3;
    I.rows = min(128, P.count[s] - 128 * t);
    I.box0 = P.first[s] + 128 * (int64_t)t;
    const int n = MODE == kM2L ? 27 : MODE == kM2M ? 4 : P.has_par;
    const int per = (n + P.n_chunks - 1) / P.n_chunks;
    I.st0 = MODE == kM2L ? min(n, I.z * per) : 0;
    I.st1 = MODE == kM2L ? min(n, I.st0 + per) : n;
    return I;
}

// row r of the item: its box (row in the level)
template <int MODE>
__device__ __forceinline__ int64_t box_of_row(const SgLevel& L, const Item& I, int r) {
    return L.lg >= 0 && MODE != kM2M ? 4 * (I.box0 + r) + I.cls : I.box0 + r;
}

// source row of box b at step st (-1: none)
template <int MODE>
__device__ __forceinline__ int source_of(const SgLevel& L, const signed char (*dxy)[2], int64_t b, int st) {
    if (L.lg < 0) return L.list[b * (MODE == kM2L ? 27 : MODE == kM2M ? 4 : 1) + st];
    if (MODE == kM2M) return (int)(4 * b + st);
    if (MODE == kL2L) return (int)(b >> 2);
    uint32_t x, y;
    unmorton2((uint32_t)b, x, y);
    const int xx = (int)x + dxy[st][0], yy = (int)y + dxy[st][1], n = 1 << L.lg;
    return (xx < 0 || yy < 0 || xx >= n || yy >= n) ? -1 : (int)morton2((uint32_t)xx, (uint32_t)yy);
}

template <typename T, int MODE>
__global__ void __launch_bounds__(kSgThreads, 1) split_gemm_kernel(const __grid_constant__ SgParams P,
                                                                   int* __restrict__ status) {
    using Cfg = SgT<T>;
    constexpr int NC = Cfg::NC, G = Cfg::G, COLS = Cfg::COLS;
    using M = Mono<T>;
    using V = typename M::V;
    extern __shared__ __align__(1024) unsigned char sg_smem[];
    const uint32_t base = smem_u32(sg_smem) + ((1024u - (smem_u32(sg_smem) & 1023u)) & 1023u);
    unsigned char* base_p = sg_smem + (base - smem_u32(sg_smem));
    const uint32_t b_base = base + kARing * kABytes;
    int* s_src = reinterpret_cast<int*>(base_p + kARing * kABytes + kBRing * kSgTileBytes);
    short* s_exp = reinterpret_cast<short*>(s_src + kSrcInts);
    __shared__ __align__(8) uint64_t afull[kARing], aempty[kARing], bfull[kBRing], bempty[kBRing], acc_full, acc_empty;
    __shared__ uint32_t s_tmem;
    __shared__ int s_end[4 * kSgMaxLevels];
    __shared__ signed char s_dxy[4][27][2];
    __shared__ unsigned char s_op[4][27];
    __shared__ uint32_t s_mx[2][128];
    __shared__ int s_abort, s_aissued, s_bissued;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int* vabort = &s_abort;
    if (threadIdx.x < 4 * 27) {
        const int c = threadIdx.x / 27, st = threadIdx.x % 27;
        int dx, dy;
        interaction_slot(c & 1, c >> 1, st, dx, dy);
        s_dxy[c][st][0] = (signed char)dx;
        s_dxy[c][st][1] = (signed char)dy;
        s_op[c][st] = (unsigned char)offset_index(dx, dy);
    }
    if (threadIdx.x >= 128 && threadIdx.x - 128 < P.n_seg) s_end[threadIdx.x - 128] = P.tile_end[threadIdx.x - 128];
    if (threadIdx.x == 0) {
        for (int i = 0; i < kARing; ++i) {
            mbar_init(&afull[i], 2 * 32);  // every producer lane's copies
            mbar_init(&aempty[i], 1);
        }
        for (int i = 0; i < kBRing; ++i) {
            mbar_init(&bfull[i], 1);
            mbar_init(&bempty[i], 1);
        }
        mbar_init(&acc_full, 1);
        mbar_init(&acc_empty, 8);
        fence_barrier_init();
        s_abort = s_aissued = s_bissued = 0;
    }
    if (warp == 0) {
        tmem_alloc(&s_tmem, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    griddep_wait();
    const uint32_t wb = ((volatile int*)status)[3] > 0 ? (uint32_t)((volatile int*)status)[3] : 0xffffffffu;
    auto abort_now = [&]() {
        atomicExch(&s_abort, 1);
        atomicExch(status, LFMM_ETIMEOUT);
    };

    if (warp >= 8 && warp < 10) {
        // ---- gather of the source rows, operator copies
        const int pw = warp - 8;
        int* my_src = s_src + pw * 64 * 28;
        const int sub = lane >> 3, ch = lane & 7;
        int aslot = 0, ause = 0, step = 0;
        bool stop = false;
        for (int item = blockIdx.x; item < P.n_items && !stop; item += gridDim.x) {
            const Item I = decode_item<MODE>(P, s_end, item);
            const SgLevel& L = P.lv[I.lev];
            for (int rl = lane; rl < 64; rl += 32) {
                const int r = 64 * pw + rl;
                const bool bv = r < I.rows;
                const int64_t b = box_of_row<MODE>(L, I, r);
#pragma unroll 1
                for (int k0 = I.st0; k0 < I.st1; k0 += 7) {
                    int v[7];
#pragma unroll
                    for (int t = 0; t < 7; ++t)
                        v[t] = bv && k0 + t < I.st1 ? source_of<MODE>(L, s_dxy[I.cls], b, k0 + t) : -1;
#pragma unroll
                    for (int t = 0; t < 7; ++t)
                        if (k0 + t < I.st1) my_src[rl * 28 + k0 + t - I.st0] = v[t];
                }
            }
            __syncwarp();
            const uint8_t* src = L.src;
            for (int st = I.st0; st < I.st1 && !stop; ++st, ++step) {
                const int bslot = step & 1;
                if (pw == 0 && lane == 0) {
                    if (step >= kBRing && !mbar_poll_bounded(&bempty[bslot], (uint32_t)((step / kBRing - 1) & 1), wb)) {
                        abort_now();
                    } else {
                        const int op = MODE == kM2L ? s_op[I.cls][st] : MODE == kL2L ? 40 + I.cls : 44 + st;
                        mbar_arrive_expect_tx(&bfull[bslot], (uint32_t)kSgTileBytes);
                        bulk_g2s_u32(b_base + (uint32_t)(bslot * kSgTileBytes), L.tiles + (size_t)op * kSgTileBytes,
                                     (uint32_t)kSgTileBytes, &bfull[bslot]);
                        s_bissued = step + 1;
                    }
                }
                // the lane's sixteen rows of the step, in 16-byte units (read before the copies:
                // the copies' memory clobber would put a shared-memory load's latency between
                // any two of them, 1,400 instead of 250 cycles a slice)
                uint32_t from16[16];
#pragma unroll
                for (int g = 0; g < 16; ++g) {
                    const int si = my_src[(4 * g + sub) * 28 + st - I.st0];
                    from16[g] = si < 0 ? ~0u : (uint32_t)si * (uint32_t)(kSgRowBytes / 16) + ch;
                }
                for (int sl = 0; sl < kSgSlices; ++sl) {
                    bool ok = *vabort == 0;
                    if (ok && ause > 0 && lane == 0) ok = mbar_poll_bounded(&aempty[aslot], (uint32_t)((ause - 1) & 1), wb);
                    if (!__all_sync(kFull, ok)) {
                        if (lane == 0) abort_now();
                        stop = true;
                        break;
                    }
                    const uint32_t sa = base + (uint32_t)aslot * kABytes;
#pragma unroll
                    for (int g = 0; g < 16; ++g) {
                        const int r = 64 * pw + 4 * g + sub;
                        const bool none = from16[g] == ~0u;
                        const uint8_t* from = src + (none ? 0 : (size_t)from16[g] * 16 + sl * 128);
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(
                                         sa + (uint32_t)(r * 128 + ((ch ^ (r & 7)) << 4))),
                                     "l"(from), "r"(none ? 0 : 16)
                                     : "memory");
                    }
                    cp_async_mbar_arrive_noinc(&afull[aslot]);
                    if (++aslot == kARing) {
                        aslot = 0;
                        ++ause;
                    }
                }
            }
            __syncwarp();
        }
        asm volatile("cp.async.wait_all;\n" ::: "memory");
    } else if (warp == 10) {
        // ---- products
        if (lane == 0) {
            int aslot = 0, ause = 0, step = 0, gs = 0;
            bool stop = false;
            for (int item = blockIdx.x; item < P.n_items && !stop; item += gridDim.x) {
                const Item I = decode_item<MODE>(P, s_end, item);
                for (int st = I.st0; st < I.st1 && !stop; ++st, ++step) {
                    const int bslot = step & 1;
                    if (*vabort || !mbar_poll_bounded(&bfull[bslot], (uint32_t)((step / kBRing) & 1), wb) ||
                        (step > 0 && !mbar_poll_bounded(&acc_empty, (uint32_t)((step - 1) & 1), wb))) {
                        abort_now();
                        stop = true;
                        break;
                    }
                    const uint64_t db = smem_desc_sw128(b_base + (uint32_t)(bslot * kSgTileBytes));
#pragma unroll
                    for (int i = 0; i < kSgSlices; ++i) {
                        if (!mbar_poll_bounded(&afull[aslot], (uint32_t)(ause & 1), wb)) {
                            abort_now();
                            stop = true;
                            break;
                        }
                        fence_proxy_async_smem();  // the gathered rows, seen by the tensor core
                        tc_fence_after();
                        const uint64_t da = smem_desc_sw128(base + (uint32_t)aslot * kABytes);
                        const uint32_t d = tmem + 64 * i;
                        constexpr int kMax = kSgSlices;
                        const int nb = G - 1 - i < kMax ? G - 1 - i : kMax;  // operator slices 0 .. nb - 1
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) {
                            const uint32_t acc = (i > 0 || kk > 0) ? 1u : 0u;
                            const int n0 = nb < 4 ? nb : 4;
                            mma_f16_ss(d, da + 2 * kk, db + 2 * kk, idesc_f16(128, 64 * n0), acc);
                            if (G == 8 && i == 1) {  // the last weight's first product
                                mma_f16_ss(d + 256, da + 2 * kk, db + 2 * kk + (4 * 8192 >> 4), idesc_f16(128, 64), 1u);
                                mma_f16_ss(d + 320, da + 2 * kk, db + 2 * kk + (5 * 8192 >> 4), idesc_f16(128, 64),
                                           kk > 0 ? 1u : 0u);
                            } else if (nb > 4) {
                                mma_f16_ss(d + 256, da + 2 * kk, db + 2 * kk + (4 * 8192 >> 4),
                                           idesc_f16(128, 64 * (nb - 4)), acc);
                            }
                        }
                        mma_commit(&aempty[aslot]);
                        s_aissued = ++gs;
                        if (++aslot == kARing) {
                            aslot = 0;
                            ++ause;
                        }
                    }
                    if (stop) break;
                    mma_commit(&bempty[bslot]);
                    mma_commit(&acc_full);
                }
            }
        }
    } else if (warp == 11) {
        // ---- charges (M2M) and constants (M2L, L2L)
        for (int item = blockIdx.x; item < P.n_items; item += gridDim.x) {
            const Item I = decode_item<MODE>(P, s_end, item);
            const SgLevel& L = P.lv[I.lev];
            for (int r = lane; r < I.rows; r += 32) {
                const int64_t b = box_of_row<MODE>(L, I, r);
                const V* Qin = (const V*)L.Qin;
                if (MODE == kM2L) {
                    const T* mono = (const T*)L.mono;
                    V sum = M::zero();
                    for (int k0 = I.st0; k0 < I.st1; k0 += 9) {
                        int sb[9];
                        V qv[9];
#pragma unroll
                        for (int t = 0; t < 9; ++t)
                            sb[t] = k0 + t < I.st1 ? source_of<MODE>(L, s_dxy[I.cls], b, k0 + t) : -1;
#pragma unroll
                        for (int t = 0; t < 9; ++t) qv[t] = sb[t] >= 0 ? Qin[sb[t]] : M::zero();
#pragma unroll
                        for (int t = 0; t < 9; ++t)
                            if (sb[t] >= 0) {
                                const int o = s_op[I.cls][k0 + t];
                                sum = M::add(sum, M::mul(M::make(mono[o], mono[kNumOffsets + o]), qv[t]));
                            }
                    }
                    ((V*)P.cpart)[I.z * P.part_rows + L.out0 + b] = sum;
                } else if (MODE == kM2M) {
                    V qv[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int cb = source_of<MODE>(L, s_dxy[0], b, c);
                        qv[c] = cb >= 0 ? Qin[cb] : M::zero();
                    }
                    ((V*)P.Cout)[b] = M::add(M::add(qv[0], qv[1]), M::add(qv[2], qv[3]));
                } else {
                    const int pb = P.has_par ? source_of<MODE>(L, s_dxy[0], b, 0) : -1;
                    V sum = pb >= 0 ? ((const V*)P.Cpar)[pb] : M::zero();
                    sum = M::add(sum, ((const V*)P.cpart)[L.out0 + b]);
                    ((V*)P.Cout)[b] = sum;
                }
            }
        }
    } else {
        // ---- read-back: row r (TMEM lane), outputs [32 half, 32 half + 32)
        const int r = (warp & 3) * 32 + lane, half = warp >> 2;
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        short* my_exp = s_exp + r * 28;
        int step = 0;
        bool dead = false;
        for (int item = blockIdx.x; item < P.n_items; item += gridDim.x) {
            const Item I = decode_item<MODE>(P, s_end, item);
            const SgLevel& L = P.lv[I.lev];
            const bool valid = r < I.rows;
            const int64_t b = box_of_row<MODE>(L, I, r);
            const int ns = I.st1 - I.st0;
            epi_sync();  // the previous item's exponents are read
            for (int st = half; st < ns; st += 2) {
                const int si = valid ? source_of<MODE>(L, s_dxy[I.cls], b, I.st0 + st) : -1;
                my_exp[st] = (short)(si < 0 ? kExpZero : L.src_e[si]);
            }
            epi_sync();
            int eref = kExpZero;
            for (int st = 0; st < ns; ++st)
                if (my_exp[st] != kExpNan) eref = max(eref, (int)my_exp[st]);
            if (MODE == kL2L && valid) eref = max(eref, P.part_e[L.out0 + b]);
            float acc[32][NC];
#pragma unroll
            for (int j = 0; j < 32; ++j)
#pragma unroll
                for (int c = 0; c < NC; ++c) acc[j][c] = 0.f;
            if (MODE == kL2L && valid) {  // the M2L's sum, loaded while the parent's product runs
                const int64_t row = L.out0 + b;
                const float f = pow2f(P.part_e[row] - eref);
                const float4* from = reinterpret_cast<const float4*>(P.part + row * (64 * NC) + 32 * half);
#pragma unroll
                for (int c = 0; c < NC; ++c)
#pragma unroll
                    for (int j = 0; j < 32; j += 4) {
                        const float4 q = from[16 * c + j / 4];
                        acc[j][c] = q.x * f, acc[j + 1][c] = q.y * f, acc[j + 2][c] = q.z * f, acc[j + 3][c] = q.w * f;
                    }
            }
            for (int st = 0; st < ns; ++st, ++step) {
                if (!dead) {
                    const bool ok = *vabort == 0 && mbar_poll_bounded(&acc_full, (uint32_t)(step & 1), wb);
                    if (!__all_sync(kFull, ok)) {
                        if (lane == 0) abort_now();
                        dead = true;
                    }
                }
                if (dead) continue;
                tc_fence_after();
                const int es = my_exp[st];
                const int op = MODE == kM2L ? s_op[I.cls][I.st0 + st] : MODE == kL2L ? 40 + I.cls : 44 + st;
                const float c = es == kExpNan    ? __int_as_float(0x7fffffff)
                                : es == kExpZero ? 0.f
                                                 : pow2f(es - eref + L.tile_e[op] - 34);
#pragma unroll
                for (int j0 = 0; j0 < 32; j0 += COLS) {
                    float w[G - 1][COLS];
#pragma unroll
                    for (int g = 0; g < G - 1; ++g) tmem_ld<COLS>(tmem + lane_base + 64 * g + 32 * half + j0, w[g]);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < COLS; ++j) {
                        float a[G - 1];
#pragma unroll
                        for (int g = 0; g < G - 1; ++g) a[g] = w[g][j];
                        join_add(a, c, acc[j0 + j]);
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&acc_empty);
            }
#pragma unroll
            for (int j = 0; j < 32; ++j) renorm(acc[j]);
            if (MODE == kM2L) {
                if (valid) {
                    const int64_t row = I.z * P.part_rows + L.out0 + b;
                    float4* to = reinterpret_cast<float4*>(P.part + row * (64 * NC) + 32 * half);
#pragma unroll
                    for (int c = 0; c < NC; ++c)
#pragma unroll
                        for (int j = 0; j < 32; j += 4)
                            to[16 * c + j / 4] = make_float4(acc[j][c], acc[j + 1][c], acc[j + 2][c], acc[j + 3][c]);
                    if (half == 0) P.part_e[row] = eref;
                }
                continue;
            }
            if (P.u && valid) {
                T* to = (T*)P.u + b * 64 + 32 * half;
#pragma unroll
                for (int j = 0; j < 32; j += 2) {
                    if constexpr (std::is_same<T, DF>::value) {
                        *reinterpret_cast<float4*>(to + j) =
                            make_float4(ldexpf(acc[j][0], eref), ldexpf(acc[j][1], eref), ldexpf(acc[j + 1][0], eref),
                                        ldexpf(acc[j + 1][1], eref));
                    } else {
                        *reinterpret_cast<double2*>(to + j) =
                            make_double2(ldexp((double)acc[j][0] + ((double)acc[j][1] + (double)acc[j][2 % NC]), eref),
                                         ldexp((double)acc[j + 1][0] + ((double)acc[j + 1][1] + (double)acc[j + 1][2 % NC]),
                                               eref));
                    }
                }
            }
            if (P.dst) {
                uint32_t mx = 0;
#pragma unroll
                for (int j = 0; j < 32; ++j) mx = max(mx, __float_as_uint(acc[j][0]) & 0x7fffffffu);
                s_mx[half][r] = mx;
                epi_sync();
                mx = max(s_mx[0][r], s_mx[1][r]);
                int e = row_exp(mx);
                if (e != kExpNan && e < -100) e = kExpZero;  // rounding of sums that cancel
                const float f = abs(e) >= kExpNan ? 0.f : pow2f(8 - e);
                if (valid) {
                    uint8_t* to = P.dst + (P.dst0 + b) * kSgRowBytes + 64 * half;
#pragma unroll
                    for (int j = 0; j < 32; ++j)
#pragma unroll
                        for (int c = 0; c < NC; ++c) acc[j][c] = f == 0.f ? 0.f : acc[j][c] * f;
#pragma unroll 1
                    for (int s = 0; s < kSgSlices; ++s) {
                        uint32_t w[16];
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            const __half2 h = __floats2half2_rn(next_digit(acc[2 * j]), next_digit(acc[2 * j + 1]));
                            w[j] = *reinterpret_cast<const uint32_t*>(&h);
                        }
#pragma unroll
                        for (int j = 0; j < 16; j += 4)
                            *reinterpret_cast<uint4*>(to + 128 * s + 4 * j) = make_uint4(w[j], w[j + 1], w[j + 2], w[j + 3]);
                    }
                    if (half == 0) P.dst_e[P.dst0 + b] = abs(e) >= kExpNan ? e : eref + e;
                }
            }
        }
    }
    __syncwarp();
    __syncthreads();
    if (s_abort && threadIdx.x == 0) {
        // the operator copies and MMAs in flight (the producer lanes waited for their rows)
        const int nb = s_bissued, m = s_aissued;
        for (int g = nb > kBRing ? nb - kBRing : 0; g < nb; ++g)
            mbar_poll_bounded(&bfull[g % kBRing], (uint32_t)((g / kBRing) & 1));
        if (m > 0) mbar_poll_bounded(&aempty[(m - 1) % kARing], (uint32_t)(((m - 1) / kARing) & 1));
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// The chunks of every row's M2L added in chunk order into chunk 0, a warp per row and two
// outputs per lane.
template <typename T>
__global__ void __launch_bounds__(256) sum_chunks_kernel(float* __restrict__ part, int32_t* __restrict__ part_e,
                                                         void* __restrict__ cpart, int64_t rows, int chunks) {
    griddep_wait();
    constexpr int NC = SgT<T>::NC;
    using M = Mono<T>;
    using V = typename M::V;
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; b < rows; b += nw) {
        const int e = __reduce_max_sync(kFull, lane < chunks ? part_e[lane * rows + b] : kExpZero);
        float v[2][NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) v[0][c] = v[1][c] = 0.f;
        V sum = M::zero();
        for (int z = 0; z < chunks; ++z) {
            const float f = pow2f(part_e[z * rows + b] - e);
            const float2* from = reinterpret_cast<const float2*>(part + (z * rows + b) * (64 * NC));
            float x[2][NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const float2 q = from[32 * c + lane];
                x[0][c] = q.x;
                x[1][c] = q.y;
            }
            add_scaled(v[0], x[0], f);
            add_scaled(v[1], x[1], f);
            if (lane == 0) sum = M::add(sum, ((const V*)cpart)[z * rows + b]);
        }
        renorm(v[0]);
        renorm(v[1]);
        float2* to = reinterpret_cast<float2*>(part + b * (64 * NC));
#pragma unroll
        for (int c = 0; c < NC; ++c) to[32 * c + lane] = make_float2(v[0][c], v[1][c]);
        if (lane == 0) {
            part_e[b] = e;
            ((V*)cpart)[b] = sum;
        }
    }
}

// M2M (UP) or L2L of a level of few boxes on the CUDA cores, in T: a block per box, 64 outputs
// x 16 (UP) or 4 groups of 16 inputs, each thread holding its 16 operator entries in
// registers (L2L: reloaded when the block's boxes change class); the groups' sums are added
// in group order and the first warp writes the row of T and, with dst set, its slices.  A
// tensor-core launch spends 10-15 us on its steps' and its slicing's latency however few its
// boxes are; this takes about 4 us while the blocks fit the chip.
struct SmallP {
    int64_t nb, row0;          // boxes; first row of the level in the expansion arrays
    int64_t cls[5];            // L2L, compact form
    const int32_t* list;       // UP: children [4]; L2L: parent [1] (compact form)
    int lg;                    // uniform form
    int has_par;
    const void* op;            // UP: m2m [256][64]; L2L: l2l [4][64][64]
    const void* x;             // rows of the children's / the parent's level
    const void* Xin;           // their charges / constants
    const float* part;         // L2L: the M2L's sums (rows of the level)
    const int32_t* part_e;
    const void* cpart;
    void* y;                   // rows out
    void* Yout;                // charges / constants out
    uint8_t* dst;              // sliced rows out (null: none)
    int32_t* dst_e;
};

template <typename T, bool UP>
__global__ void __launch_bounds__(UP ? 1024 : 256) small_level_kernel(const __grid_constant__ SmallP P) {
    griddep_wait();
    constexpr int NG = UP ? 16 : 4, NC = SgT<T>::NC;
    using M = Mono<T>;
    using V = typename M::V;
    __shared__ T s_x[NG * 16], s_red[NG][64];
    const int o = threadIdx.x & 63, g = threadIdx.x >> 6, lane = threadIdx.x & 31;
    const int64_t per = (P.nb + gridDim.x - 1) / gridDim.x;
    const int64_t b0 = blockIdx.x * per, b1 = min(P.nb, b0 + per);
    T op[16];
    int cls = -1;
    for (int64_t b = b0; b < b1; ++b) {
        int c = 0;
        if (!UP) c = P.lg >= 0 ? (int)(b & 3) : (b >= P.cls[1]) + (b >= P.cls[2]) + (b >= P.cls[3]);
        if (c != cls) {
            cls = c;
#pragma unroll
            for (int i = 0; i < 16; ++i) op[i] = ldg((const T*)P.op + (size_t)c * 4096 + (16 * g + i) * 64 + o);
        }
        if (threadIdx.x < NG * 16) {
            const int ch = threadIdx.x >> 6;
            int src = -1;
            if (UP) src = P.list[4 * b + ch];
            else if (P.has_par) src = P.lg >= 0 ? (int)(b >> 2) : P.list[b];
            s_x[threadIdx.x] = src >= 0 ? ((const T*)P.x)[(size_t)src * 64 + o] : T(0);
        }
        __syncthreads();
        T acc = T(0);
#pragma unroll
        for (int i = 0; i < 16; ++i) acc = fma(op[i], s_x[16 * g + i], acc);
        s_red[g][o] = acc;
        __syncthreads();
        if (UP) {  // sixteen groups to four
            T v = s_red[0][0];
            if (threadIdx.x < 256) v = (s_red[4 * g][o] + s_red[4 * g + 1][o]) + (s_red[4 * g + 2][o] + s_red[4 * g + 3][o]);
            __syncthreads();
            if (threadIdx.x < 256) s_red[g][o] = v;
            __syncthreads();
        }
        if (threadIdx.x < 32) {
            T v[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int q = 2 * lane + j;
                v[j] = (s_red[0][q] + s_red[1][q]) + (s_red[2][q] + s_red[3][q]);
            }
            if (!UP) {
                const float2* from = reinterpret_cast<const float2*>(P.part + (P.row0 + b) * (64 * NC));
                const int e = P.part_e[P.row0 + b];
                float2 x[NC];
#pragma unroll
                for (int k = 0; k < NC; ++k) x[k] = from[32 * k + lane];
                if constexpr (std::is_same<T, DF>::value) {
                    v[0] += DF{ldexpf(x[0].x, e), ldexpf(x[1].x, e)};
                    v[1] += DF{ldexpf(x[0].y, e), ldexpf(x[1].y, e)};
                } else {
                    v[0] += ldexp((double)x[0].x + ((double)x[1].x + (double)x[2 % NC].x), e);
                    v[1] += ldexp((double)x[0].y + ((double)x[1].y + (double)x[2 % NC].y), e);
                }
            }
            T* y = (T*)P.y + (size_t)b * 64;
            y[2 * lane] = v[0];
            y[2 * lane + 1] = v[1];
            if (P.dst) slice_row(v, lane, P.dst + b * kSgRowBytes, P.dst_e + b);
            if (lane == 0) {
                const V* X = (const V*)P.Xin;
                V* Y = (V*)P.Yout;
                if (UP) {
                    V q[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int src = P.list[4 * b + k];
                        q[k] = src >= 0 ? X[src] : M::zero();
                    }
                    Y[b] = M::add(M::add(q[0], q[1]), M::add(q[2], q[3]));
                } else {
                    const int src = !P.has_par ? -1 : P.lg >= 0 ? (int)(b >> 2) : P.list[b];
                    const V up = src >= 0 ? X[src] : M::zero();
                    Y[b] = M::add(up, ((const V*)P.cpart)[P.row0 + b]);
                }
            }
        }
        __syncthreads();
    }
}

// Levels of up to this many boxes take small_level_kernel (M2M, L2L): the work of one box
// (16,384 and 4,096 multiply-adds, 15 FP32 operations each or one at 1/64 rate) against a
// tensor-core launch's latency.
template <typename T>
constexpr int64_t kSmallUp = std::is_same<T, DF>::value ? 2048 : 304;
template <typename T>
constexpr int64_t kSmallDown = std::is_same<T, DF>::value ? 4096 : 912;

// Work space: sliced rows and exponents of q (all levels) and of u (levels k >= 1), the
// chunks' sums, exponents and constants.
struct SgWork {
    uint8_t *q, *u;
    int32_t *qe, *ue;
    float* part;
    int32_t* part_e;
    void* cpart;
    int64_t bytes;
};
SgWork carve(const SgTree& t, int nc, int chunks, void* work) {
    SgWork w;
    int64_t n = 0;
    auto take = [&](int64_t bytes) {
        const int64_t at = n;
        n += (bytes + 255) & ~(int64_t)255;
        return (uint8_t*)work + at;
    };
    const int64_t inner = t.rows - t.lv[0].nb;
    w.q = take(t.rows * kSgRowBytes);
    w.u = take(inner * kSgRowBytes);
    w.qe = (int32_t*)take(t.rows * 4);
    w.ue = (int32_t*)take(inner * 4);
    w.part = (float*)take((int64_t)chunks * t.rows * 64 * nc * 4);
    w.part_e = (int32_t*)take((int64_t)chunks * t.rows * 4);
    w.cpart = take((int64_t)chunks * t.rows * 8);
    w.bytes = n;
    return w;
}

}  // namespace

SgTree sg_uniform_tree(int L, int split) {
    SgTree t;
    t.nk = L - 1;
    t.split = split;
    for (int l = 2; l <= L; ++l) {
        SgTree::Level& lv = t.lv[L - l];
        lv.nb = (int64_t)1 << (2 * l);
        lv.off = t.rows;
        lv.lg = l;
        t.rows += lv.nb;
    }
    return t;
}

int sg_chunks(const SgTree& t, int num_sms) {
    if (t.split > 0) return std::min(t.split, 9);
    int64_t tiles = 0;
    for (int k = 0; k < t.nk; ++k)
        for (int c = 0; c < 4; ++c) {
            const int64_t n = t.lv[k].lg >= 0 ? t.lv[k].nb / 4 : t.lv[k].cls[c + 1] - t.lv[k].cls[c];
            tiles += (n + 127) / 128;
        }
    int best = 1;
    double cost = 0;
    for (int c = 1; c <= 9; ++c) {
        const double v = (double)((tiles * c + num_sms - 1) / num_sms) * ((27 + c - 1) / c + 2.0) + 0.1 * c;
        if (c == 1 || v < cost) {
            best = c;
            cost = v;
        }
    }
    return best;
}

int64_t sg_work_bytes(const SgTree& t, int precision, int num_sms) {
    return carve(t, precision == LFMM_DF ? 2 : 3, sg_chunks(t, num_sms), nullptr).bytes;
}

cudaError_t sg_build_operators(DeviceOps& ops, void* mem, cudaStream_t s) {
    const int nl = ops.n_levels;
    const size_t per = (size_t)kSgOps * kSgTileBytes;
    uint8_t* tiles = (uint8_t*)mem;
    int32_t* exps = (int32_t*)(tiles + nl * per);
    const size_t op = (size_t)64 * 64 * (ops.precision == LFMM_DF ? sizeof(DF) : sizeof(double));
    ops.sg_tiles.clear();
    ops.sg_e.clear();
    for (int k = 0; k < nl; ++k) {
        ops.sg_tiles.push_back(tiles + k * per);
        ops.sg_e.push_back(exps + k * kSgOps);
        SgOpList l;
        for (int o = 0; o < kNumOffsets; ++o) l.op[o] = (const char*)ops.tifo[k] + o * op;
        for (int c = 0; c < 4; ++c) {
            l.op[40 + c] = k + 1 < nl ? (const char*)ops.l2l[k + 1] + c * op : nullptr;
            l.op[44 + c] = k >= 1 ? (const char*)ops.m2m[k] + c * op : nullptr;
        }
        if (ops.precision == LFMM_DF)
            slice_ops_kernel<DF><<<kSgOps, 256, 0, s>>>(l, ops.sg_tiles[k], ops.sg_e[k]);
        else
            slice_ops_kernel<double><<<kSgOps, 256, 0, s>>>(l, ops.sg_tiles[k], ops.sg_e[k]);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <typename T>
cudaError_t sg_far_field(const SgTree& t, const DeviceOps& ops, T* q, T* u, void* Q, void* C, void* work,
                         bool q_all, int* status, int num_sms, cudaStream_t s, int* launches) {
    constexpr int NC = SgT<T>::NC;
    const int chunks = sg_chunks(t, num_sms);
    const SgWork w = carve(t, NC, chunks, work);
    using V8 = char[8];
    auto Qm = [&](int k) { return (void*)((V8*)Q + t.lv[k].off); };
    auto Cm = [&](int k) { return (void*)((V8*)C + t.lv[k].off); };
    auto qrow = [&](int k) { return w.q + t.lv[k].off * kSgRowBytes; };
    int64_t uoff[kSgMaxLevels] = {0};
    for (int k = 2; k < t.nk; ++k) uoff[k] = uoff[k - 1] + t.lv[k - 1].nb;
    cudaError_t e = ensure_dynamic_smem((const void*)split_gemm_kernel<T, kM2L>, kSgSmem);
    if (e == cudaSuccess) e = ensure_dynamic_smem((const void*)split_gemm_kernel<T, kM2M>, kSgSmem);
    if (e == cudaSuccess) e = ensure_dynamic_smem((const void*)split_gemm_kernel<T, kL2L>, kSgSmem);
    if (e != cudaSuccess) return e;
    // boxes of level k as up to four segments (class ranges); returns the tiles so far
    auto segments = [&](SgParams& P, int i, int k, int tiles) {
        const SgTree::Level& lv = t.lv[k];
        for (int c = 0; c < 4; ++c) {
            P.first[4 * i + c] = lv.lg >= 0 ? 0 : lv.cls[c];
            P.count[4 * i + c] = (int)(lv.lg >= 0 ? lv.nb / 4 : lv.cls[c + 1] - lv.cls[c]);
            tiles += (P.count[4 * i + c] + 127) / 128;
            P.tile_end[4 * i + c] = tiles;
        }
        return tiles;
    };
    auto go = [&](auto mode, const SgParams& P) -> cudaError_t {
        constexpr int MODE = decltype(mode)::value;
        if (P.n_items <= 0) return cudaSuccess;
        ++*launches;
        return launch_dependent(split_gemm_kernel<T, MODE>, dim3((unsigned)std::min(P.n_items, num_sms)),
                                dim3(kSgThreads), kSgSmem, s, P, status);
    };
    auto clear = [](SgParams& P) {
        P = SgParams();
        P.n_chunks = 1;
    };
    auto small_up = [&](int k) { return t.lv[k].nb > 0 && t.lv[k].nb <= kSmallUp<T>; };
    auto small_down = [&](int k) { return t.lv[k].nb > 0 && t.lv[k].nb <= kSmallDown<T>; };
    SgParams P;
    // ---- slices of the leaf expansions (or of every level's), then M2M level by level
    {
        const int64_t n = q_all ? t.rows : t.lv[0].nb, off = q_all ? 0 : t.lv[0].off;
        const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((n + 7) / 8, (int64_t)num_sms * 16));
        e = launch_dependent(slice_rows_kernel<T>, dim3((unsigned)blocks), dim3(256), 0, s, q + off * 64, n,
                             w.q + off * kSgRowBytes, w.qe + off);
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    for (int k = 1; k < t.nk && !q_all; ++k) {
        if (small_up(k)) {
            SmallP S = {};
            S.nb = t.lv[k].nb;
            S.list = t.lv[k].ch;
            S.lg = -1;
            S.op = ops.m2m[k];
            S.x = q + t.lv[k - 1].off * 64;
            S.Xin = Qm(k - 1);
            S.y = q + t.lv[k].off * 64;
            S.Yout = Qm(k);
            S.dst = qrow(k);
            S.dst_e = w.qe + t.lv[k].off;
            e = launch_dependent(small_level_kernel<T, true>, dim3((unsigned)std::min<int64_t>(S.nb, 2 * num_sms)),
                                 dim3(1024), 0, s, S);
            if (e != cudaSuccess) return e;
            ++*launches;
            continue;
        }
        clear(P);
        P.n_seg = 1;
        P.count[0] = (int)t.lv[k].nb;
        P.tile_end[0] = P.n_items = (P.count[0] + 127) / 128;
        SgLevel& L = P.lv[0];
        L.list = t.lv[k].ch;
        L.src = qrow(k - 1);
        L.src_e = w.qe + t.lv[k - 1].off;
        L.tiles = ops.sg_tiles[k];
        L.tile_e = ops.sg_e[k];
        L.Qin = Qm(k - 1);
        L.lg = t.lv[k].lg;
        P.dst = w.q;
        P.dst_e = w.qe;
        P.dst0 = t.lv[k].off;
        P.Cout = Qm(k);
        if (k + 1 < t.nk && small_up(k + 1)) P.u = q + t.lv[k].off * 64;  // read as rows of T there
        e = go(std::integral_constant<int, kM2M>(), P);
        if (e != cudaSuccess) return e;
    }
    // ---- M2L of every level
    clear(P);
    int tiles = 0;
    for (int k = 0; k < t.nk; ++k) {
        tiles = segments(P, k, k, tiles);
        SgLevel& L = P.lv[k];
        L.list = t.lv[k].il;
        L.src = qrow(k);
        L.src_e = w.qe + t.lv[k].off;
        L.tiles = ops.sg_tiles[k];
        L.tile_e = ops.sg_e[k];
        L.mono = ops.mono[k];
        L.Qin = Qm(k);
        L.out0 = t.lv[k].off;
        L.lg = t.lv[k].lg;
    }
    P.n_seg = 4 * t.nk;
    P.n_chunks = chunks;
    P.n_items = tiles * chunks;
    P.part = w.part;
    P.part_e = w.part_e;
    P.cpart = w.cpart;
    P.part_rows = t.rows;
    e = go(std::integral_constant<int, kM2L>(), P);
    if (e != cudaSuccess) return e;
    // ---- the chunks' sums, then L2L coarse to fine
    if (chunks > 1) {
        const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((t.rows + 7) / 8, (int64_t)num_sms * 8));
        e = launch_dependent(sum_chunks_kernel<T>, dim3((unsigned)blocks), dim3(256), 0, s, w.part, w.part_e, w.cpart,
                             t.rows, chunks);
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    for (int k = t.nk - 1; k >= 0; --k) {
        if (small_down(k)) {
            SmallP S = {};
            S.nb = t.lv[k].nb;
            S.row0 = t.lv[k].off;
            std::copy(t.lv[k].cls, t.lv[k].cls + 5, S.cls);
            S.list = t.lv[k].par;
            S.lg = t.lv[k].lg;
            S.has_par = k + 1 < t.nk ? 1 : 0;
            if (S.has_par) {
                S.op = ops.l2l[k + 1];
                S.x = u + t.lv[k + 1].off * 64;
                S.Xin = Cm(k + 1);
            } else {
                S.op = ops.tifo[0];  // times zero
            }
            S.part = w.part;
            S.part_e = w.part_e;
            S.cpart = w.cpart;
            S.y = u + t.lv[k].off * 64;
            S.Yout = Cm(k);
            if (k > 0 && !small_down(k - 1)) {
                S.dst = w.u + uoff[k] * kSgRowBytes;
                S.dst_e = w.ue + uoff[k];
            }
            e = launch_dependent(small_level_kernel<T, false>, dim3((unsigned)std::min<int64_t>(S.nb, 8 * num_sms)),
                                 dim3(256), 0, s, S);
            if (e != cudaSuccess) return e;
            ++*launches;
            continue;
        }
        clear(P);
        P.n_items = segments(P, 0, k, 0);
        P.n_seg = 4;
        P.has_par = k + 1 < t.nk ? 1 : 0;
        P.part = w.part;
        P.part_e = w.part_e;
        P.cpart = w.cpart;
        P.part_rows = t.rows;
        SgLevel& L = P.lv[0];
        L.tiles = ops.sg_tiles[k];
        L.tile_e = ops.sg_e[k];
        L.out0 = t.lv[k].off;
        L.lg = t.lv[k].lg;
        if (P.has_par) {
            L.list = t.lv[k].par;
            L.src = w.u + uoff[k + 1] * kSgRowBytes;
            L.src_e = w.ue + uoff[k + 1];
            P.Cpar = Cm(k + 1);
        }
        P.Cout = Cm(k);
        if (k > 0 && !small_down(k - 1)) {
            P.dst = w.u;
            P.dst_e = w.ue;
            P.dst0 = uoff[k];
        } else {
            P.u = u + t.lv[k].off * 64;
        }
        e = go(std::integral_constant<int, kL2L>(), P);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template cudaError_t sg_far_field<DF>(const SgTree&, const DeviceOps&, DF*, DF*, void*, void*, void*, bool, int*,
                                      int, cudaStream_t, int*);
template cudaError_t sg_far_field<double>(const SgTree&, const DeviceOps&, double*, double*, void*, void*, void*,
                                          bool, int*, int, cudaStream_t, int*);

}  // namespace lfmm
