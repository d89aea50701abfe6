// Shared by the reverse mode's translation units: dense cubes, the transposed
// differences and the walk over the voxels.
#pragma once

#include <type_traits>

#include "gsstv_internal.cuh"

namespace gsstv {
namespace {

constexpr int BX = 32, BY = 8, NTA = BX * BY;

struct Dims {
    int n1, n2, n3;
    int vp;                                       // row pitch of v (floats)
    int rows;                                     // n3 * n1
    long long plane;                              // n1 * n2
    long long N;                                  // voxels
};

struct SV {
    const float *u, *s, *t, *w1, *w2, *y1, *y2, *y3, *y4;
};
struct SW {
    float *u, *s, *t, *w1, *w2, *y1, *y2, *y3, *y4;
};

// read-only data (states k, k+1 and v; never written during a pass)
__device__ __forceinline__ float rd(const float* p, long long k) { return __ldg(p + k); }

// ---- stencils on dense cubes (value at voxel l = (b, i, j) of an operator's
// output).  They read through the read-only path: every kernel applies them
// only to arrays that no thread writes while it runs.  IN = the voxel is
// interior in its band (1 <= i <= N1-2, 1 <= j <= N2-2): then every spatial
// neighbour they touch exists and no boundary mask applies, so the checks
// are compiled out; the band neighbours are checked either way.

// transposes: (D_v^T y)(i) = y(i-1) [i >= 1] - y(i) [i <= N1-2]
template <bool IN>
__device__ __forceinline__ float dvT(const float* y, const Dims& d, long long l, int i) {
    float r = 0.f;
    if (IN || i >= 1) r += rd(y, l - d.n2);
    if (IN || i <= d.n1 - 2) r -= rd(y, l);
    return r;
}
template <bool IN>
__device__ __forceinline__ float dhT(const float* y, const Dims& d, long long l, int j) {
    float r = 0.f;
    if (IN || j >= 1) r += rd(y, l - 1);
    if (IN || j <= d.n2 - 2) r -= rd(y, l);
    return r;
}
// D^T y for a dual pair y (2 planes of N)
template <bool IN>
__device__ __forceinline__ float dT(const float* y, const Dims& d, long long l, int i, int j) {
    return dvT<IN>(y, d, l, i) + dhT<IN>(y + d.N, d, l, j);
}
// (D_s^T D^T y)(b) = (D^T y)(b-1) [b >= 1] - (D^T y)(b) [b <= N3-2]
template <bool IN>
__device__ __forceinline__ float dsT_dT(const float* y, const Dims& d, long long l, int b, int i, int j) {
    float r = 0.f;
    if (b >= 1) r += dT<IN>(y, d, l - d.plane, i, j);
    if (b <= d.n3 - 2) r -= dT<IN>(y, d, l, i, j);
    return r;
}
// The voxels of this thread: column j of the block, rows (b*N1 + i) strided
// by the grid; body(b, i, j, l, interior) per voxel, interior a
// std::integral_constant<bool, ...> selecting the unchecked stencils.  The
// choice is made per warp (one row, 32 columns): a warp with a border voxel
// takes the checked path for all its lanes, so no warp runs both.
template <int UNROLL = 1, class F>
__device__ __forceinline__ void for_voxels(const Dims& d, F&& body) {
    const int j = blockIdx.x * BX + threadIdx.x;
    if (j >= d.n2) return;
    const unsigned lanes = __activemask();          // the same lanes in every iteration
    const bool jin = j >= 1 && j <= d.n2 - 2;
#pragma unroll UNROLL
    for (int row = blockIdx.y * BY + threadIdx.y; row < d.rows; row += gridDim.y * BY) {
        const int b = row / d.n1, i = row - b * d.n1;
        const long long l = (long long)row * d.n2 + j;
        if (__all_sync(lanes, jin && i >= 1 && i <= d.n1 - 2))
            body(b, i, j, l, std::true_type{});
        else
            body(b, i, j, l, std::false_type{});
    }
}

}  // namespace
}  // namespace gsstv
