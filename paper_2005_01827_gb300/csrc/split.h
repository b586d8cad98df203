// split.h -- split-precision segment records and launchers (internal).
#pragma once
#include <cuda_runtime.h>

#include "kernels.h"

namespace lisa {

// FP32 staged data per bin: s_A, s_E, s_T (s_X = sqrt(w_X) 2^-64), then -2 sqrt(w_X) d_X
// for X = A, E, T (re, im); 36 bytes, so that a tile of 1024 bins takes 36 KB of shared
// memory and four blocks per SM leave L1 room for the segment records.
constexpr int kBinFloats = 9;

// One spline segment of one (walker, m) in the split-precision form, 224 bytes: the
// fixed-point phase record (kernels.h; the high half of word 7 as in the FP64 path), the first
// bin, and the sum S^X = sum A 2^64 T^X over the active modes of this m as a quartic in
// n = j - kb0 for the channels X = A, E, T: s[X] = {s0, the rest of s0, s1, s2, s3, s4},
// (re, im) pairs.  ok = 0: the quartics do not hold (see segprep_kernel) and the modes' own
// records below are used.
// Stored over the segment's spline coefficients of the first mode of that m, which are not
// needed any more (this precision has coefficients of the phase alone).
struct __align__(16) GroupRec {
    unsigned long long ph[kPhaseWords];
    int kb0, ok;
    float2 s[3][6];
    int pad[2];
};
static_assert(sizeof(GroupRec) == 224, "at most 256 bytes, a segment's coefficients");
__host__ __device__ inline GroupRec *group_rec(double *coef, size_t wm, int K, int s) {
    return reinterpret_cast<GroupRec *>(coef + (wm * (size_t)(K - 1) + s) * 32);
}

// A segment's modes on their own, written where the cubics of their sum do not hold.
// With t = (j - kb0) / W over the segment's W bins: c[k] is the t^k coefficient of
// A 2^64, and for channel x = 0, 1, 2 (A, E, T) c[4 + 8 x + 2 k] and c[4 + 8 x + 2 k + 1]
// are the t^k coefficients of Re T^X and Im T^X, interleaved so that the pair is one
// packed f32x2 operand.
struct __align__(16) SegRec {
    float c[28];
    float invw;
    int pad[3];
};
static_assert(sizeof(SegRec) == 128, "segment record is 128 bytes");

cudaError_t launch_prep_split(const double *bins, int N, float *out, cudaStream_t s);
// chunk: bins that a thread of the dense kernel takes together
cudaError_t launch_segprep(const StageDims &d, const StageBufs &b, SegRec *segs, int chunk,
                           cudaStream_t s);
cudaError_t launch_dense_split(const StageDims &d, const StageBufs &b, const SegRec *segs,
                               const float *bins, const DenseTune &t, cudaStream_t s);

}  // namespace lisa
