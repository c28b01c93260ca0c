// Skeletons and translation operators of the per-level model boxes (Sec. 5, 7, 8.1).
//
// Leaf level (side s): the candidate skeleton is the set Y of lattice points on the
// boundary of the box [0,s)^2 (Sec. 5).  A pivoted (Businger-Golub) Householder QR of
// A^{F,Y}, F the proxy ring, picks P columns; the dense-leaf operator of Remark 8.2,
// T_ofs (P x s^2), solves the least-squares problem eq. 5.1 for every lattice point of
// the box.  If the box has at most P points, the skeleton is all of them and T_ofs = I.
//
// Level k above the leaf (side 2^k s): candidates are the four children's skeletons,
// shifted into the quadrants of the model box (Sec. 8.1, step 3); the same QR picks P
// of them and the least-squares solution S (P x 4P_child) gives T_ofo = column blocks
// of S and T_ifi = their transposes (Sec. 7).
//
// Proxy ring: lattice points on the boundary of [-s, 2s-1]^2, i.e. the outer edge of
// the 3x3 block of same-level boxes around the model box.  Every box on the
// interaction list lies strictly outside it and the box itself strictly inside, so
// matching potentials there reproduces the far field outward (outgoing expansion)
// and the incoming field inward (Sec. 4.2 well-separatedness, 6a = 3 box sides).
// Per edge, `ppe` evenly spaced points are kept (all of them if the edge is shorter);
// the remark of Sec. 5 reports 40 per edge enough for 1e-10.
//
// M2L (T_ifo) for box offset o (in box sides) is phi sampled between skeletons
// (Sec. 7, Sec. 8.1 step 4): T[p][q] = phi(skel_p - skel_q - o*side).  The 40 offsets
// are all (ox, oy) in [-3,3]^2 outside [-1,1]^2: the distinct relative positions of
// interaction-list boxes under Def. 6.1 (the "42" printed in Sec. 8.1 step 4 counts
// more than Def. 6.1 allows).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <numeric>
#include <tuple>
#include <type_traits>

#include "lfmm_internal.h"
#include "split_tc.h"

namespace lfmm {

OffsetTable::OffsetTable() {
    int n = 0;
    for (int i = 0; i < 49; ++i) index[i] = -1;
    for (int oy = -3; oy <= 3; ++oy)
        for (int ox = -3; ox <= 3; ++ox) {
            if (std::abs(ox) <= 1 && std::abs(oy) <= 1) continue;
            this->ox[n] = ox;
            this->oy[n] = oy;
            index[(oy + 3) * 7 + (ox + 3)] = n;
            ++n;
        }
}

const OffsetTable& offsets() {
    static const OffsetTable t;
    return t;
}

namespace {

using Pt = std::array<int, 2>;

struct Mat {  // column-major
    int m = 0, n = 0;
    std::vector<double> a;
    Mat() = default;
    Mat(int m_, int n_) : m(m_), n(n_), a((size_t)m_ * n_, 0.0) {}
    double& operator()(int i, int j) { return a[(size_t)j * m + i]; }
    double operator()(int i, int j) const { return a[(size_t)j * m + i]; }
};

std::vector<Pt> proxy_ring(int side, int ppe) {
    const int a = -side, b = 2 * side - 1, len = b - a;
    const int n = std::min(ppe, len);
    std::vector<Pt> out;
    out.reserve(4 * n);
    for (int e = 0; e < 4; ++e)
        for (int i = 0; i < n; ++i) {
            const int pos = a + (int)std::llround((double)i * len / n);
            const int rev = a + b - pos;
            switch (e) {
                case 0: out.push_back({pos, a}); break;
                case 1: out.push_back({b, pos}); break;
                case 2: out.push_back({rev, b}); break;
                default: out.push_back({a, rev}); break;
            }
        }
    return out;
}

std::vector<Pt> box_boundary(int s) {
    std::vector<Pt> out;
    if (s == 1) return {{0, 0}};
    for (int x = 0; x < s; ++x) out.push_back({x, 0});
    for (int y = 1; y < s; ++y) out.push_back({s - 1, y});
    for (int x = s - 2; x >= 0; --x) out.push_back({x, s - 1});
    for (int y = s - 2; y >= 1; --y) out.push_back({0, y});
    return out;
}

Mat kernel_matrix(const std::vector<Pt>& F, const std::vector<Pt>& Y) {
    Mat A((int)F.size(), (int)Y.size());
    for (int j = 0; j < A.n; ++j)
        for (int i = 0; i < A.m; ++i)
            A(i, j) = phi_host((int64_t)F[i][0] - Y[j][0], (int64_t)F[i][1] - Y[j][1]);
    return A;
}

// Householder QR with column pivoting on A (in place), stopping after kmax steps or
// when the largest remaining column norm drops below rtol times the first one.
struct PivotedQR {
    Mat A;                    // R above the diagonal, Householder vectors below
    std::vector<double> tau;
    std::vector<int> piv;     // column order
    int rank = 0;
};

PivotedQR pivoted_qr(Mat A, int kmax, double rtol) {
    PivotedQR q;
    const int m = A.m, n = A.n;
    q.piv.resize(n);
    std::iota(q.piv.begin(), q.piv.end(), 0);
    const int kend = std::min(kmax, std::min(m, n));
    double norm0 = 0.0;
    int k = 0;
    for (; k < kend; ++k) {
        int best = k;
        double bestv = -1.0;
        for (int j = k; j < n; ++j) {
            double s = 0.0;
            for (int i = k; i < m; ++i) s += A(i, j) * A(i, j);
            if (s > bestv) {
                bestv = s;
                best = j;
            }
        }
        const double bn = std::sqrt(bestv);
        if (k == 0) norm0 = bn;
        if (bn == 0.0 || bn <= rtol * norm0) break;
        if (best != k) {
            for (int i = 0; i < m; ++i) std::swap(A(i, k), A(i, best));
            std::swap(q.piv[k], q.piv[best]);
        }
        const double x0 = A(k, k);
        const double beta = -std::copysign(bn, x0);
        const double v0 = x0 - beta;
        for (int i = k + 1; i < m; ++i) A(i, k) /= v0;
        const double t = (beta - x0) / beta;
        A(k, k) = beta;
        q.tau.push_back(t);
        for (int j = k + 1; j < n; ++j) {
            double d = A(k, j);
            for (int i = k + 1; i < m; ++i) d += A(i, k) * A(i, j);
            d *= t;
            A(k, j) -= d;
            for (int i = k + 1; i < m; ++i) A(i, j) -= d * A(i, k);
        }
    }
    q.rank = k;
    q.A = std::move(A);
    return q;
}

// X (rank x nb) minimising || A[:, piv[:rank]] X - B ||_2  (row-major result)
std::vector<double> least_squares(const PivotedQR& q, Mat B) {
    const int m = q.A.m, r = q.rank;
    for (int k = 0; k < r; ++k)
        for (int j = 0; j < B.n; ++j) {
            double d = B(k, j);
            for (int i = k + 1; i < m; ++i) d += q.A(i, k) * B(i, j);
            d *= q.tau[k];
            B(k, j) -= d;
            for (int i = k + 1; i < m; ++i) B(i, j) -= d * q.A(i, k);
        }
    std::vector<double> X((size_t)r * B.n, 0.0);
    for (int j = 0; j < B.n; ++j)
        for (int i = r - 1; i >= 0; --i) {
            double v = B(i, j);
            for (int l = i + 1; l < r; ++l) v -= q.A(i, l) * X[(size_t)l * B.n + j];
            X[(size_t)i * B.n + j] = v / q.A(i, i);
        }
    return X;
}

constexpr double kRankTol = 1e-14;

void build_leaf(ModelOps& mo) {
    const int s = mo.leaf_side, P = mo.P_target;
    LevelOps lv;
    lv.side = s;
    std::vector<Pt> all;
    for (int y = 0; y < s; ++y)
        for (int x = 0; x < s; ++x) all.push_back({x, y});
    if (s * s <= P) {
        lv.P = s * s;
        for (auto& p : all) {
            lv.skel.push_back(p[0]);
            lv.skel.push_back(p[1]);
        }
        mo.tofs.assign((size_t)lv.P * s * s, 0.0);
        for (int i = 0; i < lv.P; ++i) mo.tofs[(size_t)i * s * s + i] = 1.0;
    } else {
        const std::vector<Pt> Y = box_boundary(s);
        const std::vector<Pt> F = proxy_ring(s, mo.ppe);
        PivotedQR q = pivoted_qr(kernel_matrix(F, Y), P, kRankTol);
        lv.P = q.rank;
        for (int i = 0; i < q.rank; ++i) {
            lv.skel.push_back(Y[q.piv[i]][0]);
            lv.skel.push_back(Y[q.piv[i]][1]);
        }
        mo.tofs = least_squares(q, kernel_matrix(F, all));
    }
    mo.levels.push_back(std::move(lv));
}

void build_level(ModelOps& mo) {
    const LevelOps& ch = mo.levels.back();
    LevelOps lv;
    lv.side = 2 * ch.side;
    std::vector<Pt> Y;
    for (int c = 0; c < 4; ++c) {
        const int dx = (c & 1) * ch.side, dy = (c >> 1) * ch.side;
        for (int q = 0; q < ch.P; ++q) Y.push_back({ch.skel[2 * q] + dx, ch.skel[2 * q + 1] + dy});
    }
    const std::vector<Pt> F = proxy_ring(lv.side, mo.ppe);
    Mat A = kernel_matrix(F, Y);
    PivotedQR q = pivoted_qr(A, mo.P_target, kRankTol);
    lv.P = q.rank;
    for (int i = 0; i < q.rank; ++i) {
        lv.skel.push_back(Y[q.piv[i]][0]);
        lv.skel.push_back(Y[q.piv[i]][1]);
    }
    lv.S = least_squares(q, std::move(A));
    mo.levels.push_back(std::move(lv));
}

std::mutex g_cache_mu;
std::map<std::tuple<int, int, int>, std::unique_ptr<ModelOps>> g_cache;

}  // namespace

void tifo_matrix(const LevelOps& lv, int o, std::vector<double>& out) {
    const OffsetTable& ot = offsets();
    const int64_t ox = (int64_t)ot.ox[o] * lv.side, oy = (int64_t)ot.oy[o] * lv.side;
    out.assign((size_t)lv.P * lv.P, 0.0);
    for (int p = 0; p < lv.P; ++p)
        for (int q = 0; q < lv.P; ++q)
            out[(size_t)p * lv.P + q] =
                phi_host(lv.skel[2 * p] - lv.skel[2 * q] - ox, lv.skel[2 * p + 1] - lv.skel[2 * q + 1] - oy);
}

ModelOps* get_model_ops(int leaf_side, int P, int ppe, int n_levels, std::string* err) {
    if (leaf_side < 1 || leaf_side > kMaxLeafSide || (leaf_side & (leaf_side - 1)) ||
        P < 1 || P > kMaxP || ppe < 8 || n_levels < 1 || n_levels > 31) {
        if (err) *err = "invalid model-box parameters";
        return nullptr;
    }
    ModelOps* mo;
    {
        std::lock_guard<std::mutex> g(g_cache_mu);
        auto& slot = g_cache[{leaf_side, P, ppe}];
        if (!slot) {
            slot.reset(new ModelOps());
            slot->leaf_side = leaf_side;
            slot->P_target = P;
            slot->ppe = ppe;
        }
        mo = slot.get();
    }
    std::lock_guard<std::mutex> g(mo->mu);
    if (mo->levels.empty()) build_leaf(*mo);
    while ((int)mo->levels.size() < n_levels) build_level(*mo);
    return mo;
}

// ------------------------------------------------------------------ device upload

namespace {

// TF32 with round-to-nearest (ties away): keep 10 explicit mantissa bits.
float tf32_rna(float x) {
    uint32_t u;
    std::memcpy(&u, &x, 4);
    u = (u + 0x1000u) & 0xFFFFE000u;
    float r;
    std::memcpy(&r, &u, 4);
    return r;
}

// Tensor-core B operand of one operator for K-block h (k in [32h, 32h + 32)): the
// operator's v(n, k) (n = output p < NP) split into TF32 hi and lo and stacked as one
// K-major matrix of 2 NP rows (hi rows, then lo rows) x 32 K in fp32, laid out as the
// 128-byte-swizzled shared-memory image (row r at 128 r bytes, 16-byte chunk c of the
// row at chunk c ^ (r mod 8)).  NP / 32 such blocks per operator, block h at
// dst + h * 64 NP floats.
void write_tc_tile(float* dst, int NP, const float (*v)[64]) {
    for (int h = 0; h < NP / 32; ++h) {
        float* blk = dst + (size_t)h * 64 * NP;
        for (int n = 0; n < NP; ++n)
            for (int c = 0; c < 8; ++c) {  // ((NP + n) & 7 == n & 7)
                float* at = blk + (size_t)n * 32 + ((c ^ (n & 7)) << 2);
                for (int k = 0; k < 4; ++k) {
                    const float x = v[n][32 * h + 4 * c + k];
                    const float hv = tf32_rna(x);
                    at[k] = hv;
                    at[k + (size_t)NP * 32] = tf32_rna(x - hv);
                }
            }
    }
}

uint32_t float_bits(float x) {
    uint32_t u;
    std::memcpy(&u, &x, 4);
    return u;
}
float bits_float(uint32_t u) {
    float x;
    std::memcpy(&x, &u, 4);
    return x;
}
// binary16 round to nearest even of |x| < 2^15; below 2^-14 the grid has a spacing of 2^-24,
// as binary32 has from 0.5 on, so adding 0.5 rounds to it.
uint32_t half_rne(float x) {
    const uint32_t sign = (float_bits(x) >> 16) & 0x8000u;
    const float a = std::fabs(x);
    const uint32_t tiny = float_bits(a + 0.5f) - 0x3f000000u;
    uint32_t u = float_bits(a) - ((127u - 15u) << 23);
    u = (u + 0xfffu + ((u >> 13) & 1u)) >> 13;
    return sign | (a < 6.103515625e-05f ? tiny : u);
}
// the finite binary16 h (its exponent field moved to binary32's, subnormals included)
float half_value(uint32_t h) { return bits_float((h & 0x7fffu) << 13 | (h & 0x8000u) << 16) * 0x1p112f; }

// The same operators for the fp16 tensor-core M2L: x(n, k) scaled by a power of two so
// that the largest magnitude lies in [2^14, 2^15), split into fp16 hi and lo and stacked as
// one K-major matrix of 2 NP rows (hi rows, then lo rows) of 128 bytes (64 halves; NP = 32
// uses the first 32), 128-byte swizzled.  Returns the factor that undoes the scaling.
float write_half_tile(uint16_t* dst, int NP, const float (*x)[64]) {
    uint32_t top = 0;  // the largest magnitude's bits
    for (int n = 0; n < NP; ++n)
        for (int k = 0; k < NP; ++k) top = std::max(top, float_bits(x[n][k]) & 0x7fffffffu);
    const int sh = top ? std::min(14 - std::ilogb(bits_float(top)), 100) : 0;
    const float up = std::ldexp(1.0f, sh);  // (products with it round as ldexp rounds)
    for (int n = 0; n < NP; ++n) {
        uint32_t h[64], l[64];  // (words, and a loop of its own, so that it vectorises)
        for (int k = 0; k < NP; ++k) {
            const float v = x[n][k] * up;
            h[k] = half_rne(v);
            l[k] = half_rne(v - half_value(h[k]));
        }
        for (int k = 0; k < NP; ++k) {
            uint16_t* at = dst + (size_t)n * 64 + (((k >> 3) ^ (n & 7)) << 3) + (k & 7);
            at[0] = (uint16_t)h[k];
            at[(size_t)NP * 64] = (uint16_t)l[k];  // row NP + n: the same swizzle
        }
    }
    return std::ldexp(1.0f, -sh);
}

// Element offsets of the operators in their image.
struct ImageOffsets {
    size_t tofs = 0, tab = 0;
    std::vector<size_t> m2m, l2l, tifo, mono;  // per level
};

template <typename T>
std::vector<T> operator_image(const ModelOps& mo, int NP, int n_levels, int H, int W, ImageOffsets& off) {
    const int s = mo.leaf_side;
    auto align = [](size_t v) { return (v + 31) & ~(size_t)31; };  // 128/256-byte aligned blocks
    size_t n = 0;
    off.tofs = n;
    n = align(n + (size_t)s * s * NP);
    off.tab = n;
    n = align(n + (size_t)(2 * H + 1) * W + 2);
    off.m2m.assign(n_levels, 0);
    off.l2l.assign(n_levels, 0);
    off.tifo.assign(n_levels, 0);
    off.mono.assign(n_levels, 0);
    for (int k = 0; k < n_levels; ++k) {
        off.mono[k] = n;
        n = align(n + (size_t)2 * kNumOffsets);
        if (k >= 1) {
            off.m2m[k] = n;
            n = align(n + (size_t)4 * NP * NP);
            off.l2l[k] = n;
            n = align(n + (size_t)4 * NP * NP);
        }
        off.tifo[k] = n;
        n = align(n + (size_t)kNumOffsets * NP * NP);
    }
    std::vector<T> img(n, T(0));
    // leaf T_ofs, transposed: tofsT[J][p]
    const LevelOps& leaf = mo.levels[0];
    for (int p = 0; p < leaf.P; ++p)
        for (int J = 0; J < s * s; ++J)
            img[off.tofs + (size_t)J * NP + p] = (T)mo.tofs[(size_t)p * s * s + J];
    // P2P table: entry (dx, dy), |dx|,|dy| <= H, at (dy + H) * W + (dx + H), deflated by
    // phi0 = phi(s, 0) (about the middle of the near-field range); phi0 times the charge of
    // the 3x3 leaf block is added back in the compensated channel.  phi0 as (hi, lo) after
    // the table.
    const double phi0 = phi_host(s, 0);
    for (int dy = -H; dy <= H; ++dy)
        for (int dx = -H; dx <= H; ++dx)
            img[off.tab + (size_t)(dy + H) * W + (dx + H)] = (T)(phi_host(dx, dy) - phi0);
    {
        const size_t e = off.tab + (size_t)(2 * H + 1) * W;
        const T hi = (T)phi0;
        img[e] = hi;
        img[e + 1] = (T)(phi0 - (double)hi);
    }
    std::vector<double> t;
    for (int k = 0; k < n_levels; ++k) {
        const LevelOps& lv = mo.levels[k];
        if (k >= 1) {
            const LevelOps& ch = mo.levels[k - 1];
            const int cols = 4 * ch.P;
            for (int c = 0; c < 4; ++c)
                for (int q = 0; q < ch.P; ++q)
                    for (int p = 0; p < lv.P; ++p) {
                        const double v = lv.S[(size_t)p * cols + c * ch.P + q];
                        img[off.m2m[k] + (size_t)(c * NP + q) * NP + p] = (T)v;   // [c*NP+q][p]
                        img[off.l2l[k] + ((size_t)c * NP + p) * NP + q] = (T)v;   // [c][p_par][q_child]
                    }
        }
        // Deflated M2L: T_ifo minus its centre-to-centre value c_o = phi(o * side).  The
        // removed rank-one part c_o 1 1^T acts on a box's total charge Q; the kernels
        // carry c_o * Q in a compensated scalar channel (values ~|Q| that cancel across
        // boxes and levels), so rounding of the expansions only meets the small remainder.
        const OffsetTable& ot = offsets();
        for (int o = 0; o < kNumOffsets; ++o) {
            tifo_matrix(lv, o, t);
            const double c = phi_host((int64_t)ot.ox[o] * lv.side, (int64_t)ot.oy[o] * lv.side);
            const T hi = (T)c;
            img[off.mono[k] + o] = hi;
            img[off.mono[k] + kNumOffsets + o] = (T)(c - (double)hi);
            for (int q = 0; q < lv.P; ++q)
                for (int p = 0; p < lv.P; ++p)
                    img[off.tifo[k] + ((size_t)o * NP + q) * NP + p] = (T)(t[(size_t)p * lv.P + q] - c);
        }
    }
    return img;
}

// Floats of one level's tensor-core tiles: 40 offsets and 4 L2L classes (rows: TF32 hi and lo,
// NP / 32 blocks of 64 NP floats each; halves: fp16 hi and lo, 2 NP rows of 128 bytes, then the
// floats that undo the scaling); 1 KB aligned.
size_t tile_floats(int NP, bool halves) {
    const size_t n = (size_t)(kNumOffsets + 4) * (halves ? 2 * NP * 32 + 1 : 2 * NP * NP);
    return (n + 255) & ~(size_t)255;
}
size_t tile_bytes(int NP, bool halves, int levels) { return tile_floats(NP, halves) * levels * sizeof(float); }
size_t sliced_bytes(int n_levels) { return (sg_operator_bytes(n_levels) + 1023) / 1024 * 1024; }

// Tiles of levels have .. want - 1 from the binary32 image, in `mem` (1 KB aligned) or, if null,
// in an allocation of their own; on the device when the call returns.  L2L tile of class c at
// the child's level k: B[n = child p][k = parent q] = S_{k+1}[q][c P_k + p].
cudaError_t add_tiles(DeviceOps& d, bool halves, int want, void* mem, const std::vector<float>& img,
                      const ImageOffsets& off, cudaStream_t stream) {
    int& have = halves ? d.have.halves : d.have.rows;
    const int NP = d.NP, k0 = have;
    std::vector<float> out(tile_floats(NP, halves) * (want - k0), 0.0f);
    float v[64][64];
    for (int k = k0; k < want; ++k) {
        float* lvl = out.data() + tile_floats(NP, halves) * (k - k0);
        for (int op = 0; op < kNumOffsets + 4; ++op) {
            if (op >= kNumOffsets && k + 1 >= d.n_levels) break;
            const float* from = op < kNumOffsets ? img.data() + off.tifo[k] + (size_t)op * NP * NP
                                                 : img.data() + off.l2l[k + 1] + (size_t)(op - kNumOffsets) * NP * NP;
            for (int q = 0; q < NP; ++q)
                for (int p = 0; p < NP; ++p) v[p][q] = from[(size_t)q * NP + p];
            if (halves)
                lvl[(size_t)(kNumOffsets + 4) * 2 * NP * 32 + op] =
                    write_half_tile(reinterpret_cast<uint16_t*>(lvl + (size_t)op * 2 * NP * 32), NP, v);
            else
                write_tc_tile(lvl + (size_t)op * 2 * NP * NP, NP, v);
        }
    }
    void* own = nullptr;
    cudaError_t e = cudaSuccess;
    if (!mem) {
        e = cudaMalloc(&own, out.size() * sizeof(float));
        if (e != cudaSuccess) return e;
        mem = own;
    }
    e = cudaMemcpyAsync(mem, out.data(), out.size() * sizeof(float), cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) {
        if (own) cudaFree(own);
        return e;
    }
    if (own) d.retired.push_back(own);
    for (int k = k0; k < want; ++k) {
        float* lvl = (float*)mem + tile_floats(NP, halves) * (k - k0);
        if (halves) {
            d.tch[k] = lvl;
            d.tch_scale[k] = lvl + (size_t)(kNumOffsets + 4) * 2 * NP * 32;
        } else {
            d.tc[k] = lvl;
        }
    }
    have = want;
    return cudaSuccess;
}

// The sliced operators of every level likewise.
cudaError_t add_sliced(DeviceOps& d, void* mem, cudaStream_t stream) {
    void* own = nullptr;
    cudaError_t e = cudaSuccess;
    if (!mem) {
        e = cudaMalloc(&own, sliced_bytes(d.n_levels));
        if (e != cudaSuccess) return e;
        mem = own;
    }
    e = sg_build_operators(d, mem, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);  // plans on other streams use them too
    if (e != cudaSuccess) {
        if (own) cudaFree(own);
        return e;
    }
    if (own) d.retired.push_back(own);
    d.have.sliced = true;
    return cudaSuccess;
}

}  // namespace

const DeviceOps* get_device_ops(ModelOps* mo, int precision, int NP, int n_levels, OpsImages* want,
                                cudaStream_t stream, std::string* err) {
    std::lock_guard<std::mutex> g(mo->mu);
    while ((int)mo->levels.size() < n_levels) build_level(*mo);
    auto& slot = mo->dev[precision == LFMM_MIXED ? 1 : (precision == LFMM_DF ? 2 : 0)][NP == 64 ? 1 : 0];
    auto failed = [&](const char* what, cudaError_t e) {
        cudaGetLastError();
        if (err) *err = std::string(what) + cudaGetErrorString(e);
        return nullptr;
    };
    if (slot && slot->n_levels >= n_levels) {
        // brought here by plans that used fewer of the images
        const bool rows = slot->have.rows < want->rows, halves = slot->have.halves < want->halves;
        if (rows || halves) {
            // from the operators on the device (quicker than computing them again)
            std::vector<float> img(slot->bytes / sizeof(float));
            ImageOffsets off;
            for (int k = 0; k < slot->n_levels; ++k) {
                off.tifo.push_back((float*)slot->tifo[k] - (float*)slot->base);
                off.l2l.push_back(k >= 1 ? (float*)slot->l2l[k] - (float*)slot->base : 0);
            }
            cudaError_t e = cudaMemcpyAsync(img.data(), slot->base, slot->bytes, cudaMemcpyDeviceToHost, stream);
            if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
            if (e == cudaSuccess && rows) e = add_tiles(*slot, false, want->rows, nullptr, img, off, stream);
            if (e == cudaSuccess && halves) e = add_tiles(*slot, true, want->halves, nullptr, img, off, stream);
            if (e != cudaSuccess) return failed("operator tiles: ", e);
        }
        if (want->sliced && !slot->have.sliced && add_sliced(*slot, nullptr, stream) != cudaSuccess) {
            cudaGetLastError();
            want->sliced = false;
        }
        return slot.get();
    }
    const int nl = std::max(n_levels, slot ? slot->n_levels : 0);
    std::unique_ptr<DeviceOps> d(new DeviceOps());
    d->NP = NP;
    d->precision = precision;
    d->n_levels = nl;
    d->leaf_side = mo->leaf_side;
    d->tab_H = 2 * mo->leaf_side - 1;
    d->tab_W = p2p_table_width(mo->leaf_side);
    d->m2m.resize(nl);
    d->l2l.resize(nl);
    d->tifo.resize(nl);
    d->mono.resize(nl);
    d->tc.assign(nl, nullptr);
    d->tch.assign(nl, nullptr);
    d->tch_scale.assign(nl, nullptr);
    ImageOffsets off;
    const char* what = "";
    auto upload = [&](auto zero) -> cudaError_t {
        using T = decltype(zero);
        const std::vector<T> img = operator_image<T>(*mo, NP, nl, d->tab_H, d->tab_W, off);
        const size_t own = d->bytes = img.size() * sizeof(T);
        const size_t tiles = (own + 1023) / 1024 * 1024;
        const size_t slices = tiles + tile_bytes(NP, false, want->rows) + tile_bytes(NP, true, want->halves);
        what = "cudaMalloc(operators): ";
        cudaError_t e = cudaErrorMemoryAllocation;
        if (want->sliced && (e = cudaMalloc(&d->base, slices + sliced_bytes(nl))) != cudaSuccess) {
            cudaGetLastError();
            want->sliced = false;  // the plan can do without
        }
        if (e != cudaSuccess) e = cudaMalloc(&d->base, slices);
        if (e != cudaSuccess) return e;
        what = "upload(operators): ";
        char* b = (char*)d->base;
        e = cudaMemcpyAsync(b, img.data(), own, cudaMemcpyHostToDevice, stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
        d->tofsT = b + off.tofs * sizeof(T);
        d->p2p_table = b + off.tab * sizeof(T);
        for (int k = 0; k < nl; ++k) {
            d->m2m[k] = k >= 1 ? b + off.m2m[k] * sizeof(T) : nullptr;
            d->l2l[k] = k >= 1 ? b + off.l2l[k] * sizeof(T) : nullptr;
            d->tifo[k] = b + off.tifo[k] * sizeof(T);
            d->mono[k] = b + off.mono[k] * sizeof(T);
        }
        if constexpr (std::is_same<T, float>::value) {
            if (e == cudaSuccess && want->rows > 0) e = add_tiles(*d, false, want->rows, b + tiles, img, off, stream);
            if (e == cudaSuccess && want->halves > 0)
                e = add_tiles(*d, true, want->halves, b + tiles + tile_bytes(NP, false, want->rows), img, off, stream);
        }
        if (e == cudaSuccess && want->sliced) e = add_sliced(*d, b + slices, stream);
        if (e != cudaSuccess) cudaFree(d->base);
        return e;
    };
    const cudaError_t e = precision == LFMM_MIXED ? upload(0.0f) : precision == LFMM_DF ? upload(DF(0.0)) : upload(0.0);
    if (e != cudaSuccess) return failed(what, e);
    if (slot) d->retired.push_back(slot.release());  // plans built earlier may still use it
    slot = std::move(d);
    return slot.get();
}

}  // namespace lfmm
