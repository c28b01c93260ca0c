// Far-field translations of the binary64-accurate paths (LFMM_DF, LFMM_FP64) on the
// tensor cores, at P_pad 64: the operands split into small integers held exactly in fp16
// (split_tc.cu).
#pragma once

#include "lfmm_internal.h"

namespace lfmm {

constexpr int kSgMaxLevels = 16;
constexpr int kSgSlices = 6;                                  // slices per operand
constexpr int64_t kSgRowBytes = kSgSlices * 64 * 2;           // one box's sliced expansion
constexpr int64_t kSgTileBytes = (int64_t)kSgSlices * 64 * 128;  // one sliced operator
constexpr int kSgOps = 48;  // per level: 40 T_ifo, 4 L2L (from the parents), 4 M2M (from the children)

// A tree whose levels k = 0 (leaves) .. nk - 1 hold expansions.  Compact form: box lists as
// in ForestLevel.  Uniform form (lg >= 0): every box of a 2^lg x 2^lg level in Morton order.
struct SgTree {
    int nk = 0;
    struct Level {
        int64_t nb = 0, off = 0;  // boxes; first row in the expansion arrays
        int64_t cls[5] = {0};     // class starts (compact form)
        const int32_t *il = nullptr, *par = nullptr, *ch = nullptr;
        int lg = -1;
    } lv[kSgMaxLevels];
    int64_t rows = 0;      // expansion rows over all levels
    int split = 0;         // opts.m2l_split
};

// The level structure of a uniform tree (levels 2 .. L, leaf level L >= 2).
SgTree sg_uniform_tree(int L, int split);
// Whether a plan's far field runs here: binary64-accurate path at P_pad 64 unless
// opts.tc_min_level > 30 keeps the tensor cores out.  Pruned trees and forests always do;
// uniform trees from the leaf level on from which the mixed path's M2L takes the tensor cores
// (6 unless opts.tc_min_level says otherwise).  The line is the mixed path's, not a measured
// one: here the slices are ahead at every level (evaluations of 500 points, leaf level 2, to
// 30,000, leaf level 5, tc_min_level 2 against 31: float-float 79-184 against 154-408 us,
// binary64 79-288 against 270-706; 60,000 points, level 6: 240 against 746, 413 against 1,546).
inline bool sg_applies(int precision, int NP, int tc_min_level) {
    return precision != LFMM_MIXED && NP == 64 && tc_min_level <= 30;
}
inline bool sg_applies_uniform(int precision, int NP, int L, int tc_min_level) {
    return sg_applies(precision, NP, tc_min_level) && L >= std::max(2, tc_min_level == 0 ? kDefaultTcMinLevel : tc_min_level) && L - 1 <= kSgMaxLevels;
}
SgTree forest_sg_tree(const Forest& F);
// K chunks of the M2L (more than one when its 128-box tiles would leave SMs idle).
int sg_chunks(const SgTree& t, int num_sms);
// Bytes of the work space of one evaluation.
int64_t sg_work_bytes(const SgTree& t, int precision, int num_sms);
// Sliced operators of every level of `ops` (binary64-accurate paths, P_pad 64), in `mem` (1 KB
// aligned, sg_operator_bytes of it).
constexpr size_t sg_operator_bytes(int n_levels) {
    return (size_t)n_levels * kSgOps * (kSgTileBytes + sizeof(int32_t));
}
cudaError_t sg_build_operators(DeviceOps& ops, void* mem, cudaStream_t s);
// M2M (unless q_all: the expansions of every level are in q already), M2L and L2L: from the
// leaf expansions and charges in q / Q to the leaf incoming expansions and constants in
// u / C (rows as in t.lv[k].off; other levels' rows of q and u are scratch).
template <typename T>
cudaError_t sg_far_field(const SgTree& t, const DeviceOps& ops, T* q, T* u, void* Q, void* C, void* work,
                         bool q_all, int* status, int num_sms, cudaStream_t s, int* launches);

}  // namespace lfmm
