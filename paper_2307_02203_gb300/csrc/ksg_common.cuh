// Device helpers shared by the KSG kernels (brute-force and pruned).
#pragma once

#include <cuda_runtime.h>

namespace ndf {

// sorted ascending a[0..K1): insert d, dropping the largest; identity if d >= a[K1-1]
template <int K1>
__device__ __forceinline__ void topk_insert(float (&a)[K1], float d) {
#pragma unroll
    for (int p = K1 - 1; p > 0; --p) a[p] = fmaxf(a[p - 1], fminf(a[p], d));
    a[0] = fminf(a[0], d);
}

// #{p : |fl(a[p] - c)| < e} in the ascending array a[0..n) by two binary
// searches on predicates that are monotone in p.
__device__ __forceinline__ int count_within(const float* a, int n, float c, float e) {
    int lo = 0, len = n;
    while (len > 0) {  // first p with fl(c - a[p]) < e
        int h = len >> 1;
        if (!((c - a[lo + h]) < e)) {
            lo += h + 1;
            len -= h + 1;
        } else {
            len = h;
        }
    }
    int hi = 0;
    len = n;
    while (len > 0) {  // first p with fl(a[p] - c) >= e
        int h = len >> 1;
        if (!((a[hi + h] - c) >= e)) {
            hi += h + 1;
            len -= h + 1;
        } else {
            len = h;
        }
    }
    return hi > lo ? hi - lo : 0;
}

// Binary searches of several bounds at once over ascending arrays of n values, branchless and
// without range checks: pred(p) is true up to the bound and false from it on.  A first probe at
// top - 1 (top = the largest power of two <= n) chooses the window of top - 1 values that holds
// the bound (the first ones, or the last ones: everything before n - (top - 1) <= top is true
// then); steps top / 2, .., 1 stay inside it.  One load, one subtract, one compare and one add
// per bound and step; the bounds' dependent load chains overlap.
template <int C, class Pred>
__device__ __forceinline__ void partition_points(int n, int top, int (&pos)[C], Pred&& pred) {
#pragma unroll
    for (int c = 0; c < C; ++c) pos[c] = pred(c, top - 1) ? n - (top - 1) : 0;
#pragma unroll
    for (int s = 11; s >= 0; --s) {  // n <= 8191
        const int step = 1 << s;
        if (step < top) {
#pragma unroll
            for (int c = 0; c < C; ++c)
                if (pred(c, pos[c] + step - 1)) pos[c] += step;
        }
    }
}

// pos[c] = #{p : a[p] < y[c]} in the ascending a[0..n)
template <int C>
__device__ __forceinline__ void lower_bounds(const float* a, int n, int top, const float (&y)[C], int (&pos)[C]) {
    partition_points<C>(n, top, pos, [&](int c, int p) { return a[p] < y[c]; });
}

// count_within for two arrays at once: na = #{p : |fl(a[p] - c)| < e} in the
// ascending a[0..n), nb = the same for (b, d).  The predicates are those of
// count_within and monotone in p, so the counts are identical.
__device__ __forceinline__ void count_within_pair(const float* a, const float* b,
                                                  int n, int top, float c, float d, float e, int& na,
                                                  int& nb) {
    int q[4];
    partition_points<4>(n, top, q, [&](int i, int p) {
        return i == 0 ? !((c - a[p]) < e) : i == 1 ? !((a[p] - c) >= e) : i == 2 ? !((d - b[p]) < e) : !((b[p] - d) >= e);
    });
    na = q[1] > q[0] ? q[1] - q[0] : 0;
    nb = q[3] > q[2] ? q[3] - q[2] : 0;
}

// The non-strict counts of KSG algorithm 2 for two arrays at once, by the same
// searches: na = #{p : |fl(a[p] - c)| <= ea}, nb = #{p : |fl(b[p] - d)| <= eb}
// (the predicates of count_le).
__device__ __forceinline__ void count_le_pair(const float* a, const float* b, int n,
                                              int top, float c, float ea, float d, float eb, int& na,
                                              int& nb) {
    int q[4];
    partition_points<4>(n, top, q, [&](int i, int p) {
        return i == 0 ? !((c - a[p]) <= ea) : i == 1 ? !((a[p] - c) > ea) : i == 2 ? !((d - b[p]) <= eb) : !((b[p] - d) > eb);
    });
    na = q[1] > q[0] ? q[1] - q[0] : 0;
    nb = q[3] > q[2] ? q[3] - q[2] : 0;
}

// the largest power of two <= n (n >= 1)
__device__ __forceinline__ int pow2_floor(int n) { return 1 << (31 - __clz(n)); }

// #{p : |fl(a[p] - c)| <= e} in the ascending sequence at(0..n) (non-strict, as
// KSG algorithm 2 counts), by two binary searches on monotone predicates.
template <class Get>
__device__ __forceinline__ int count_le(Get at, int n, float c, float e) {
    int lo = 0, len = n;
    while (len > 0) {  // first p with fl(c - a[p]) <= e
        const int h = len >> 1;
        if (!((c - at(lo + h)) <= e)) { lo += h + 1; len -= h + 1; }
        else len = h;
    }
    int hi = 0;
    len = n;
    while (len > 0) {  // first p with fl(a[p] - c) > e
        const int h = len >> 1;
        if (!((at(hi + h) - c) > e)) { hi += h + 1; len -= h + 1; }
        else len = h;
    }
    return hi > lo ? hi - lo : 0;
}

// KSG algorithm 2: the largest |dx| and |dy| over the members j != s whose joint
// max-norm distance to the x-sorted point s is <= e (they lie in the x-window
// |dx| <= e around position s, scanned outward).  pt(j) returns the x-sorted point.
template <class Get>
__device__ __forceinline__ void alg2_extents(Get pt, int M, int s, float2 ps, float e, float& ex,
                                             float& ey) {
    ex = 0.0f;
    ey = 0.0f;
    for (int j = s + 1; j < M; ++j) {
        const float2 c = pt(j);
        const float dx = c.x - ps.x;
        if (dx > e) break;
        const float dy = fabsf(ps.y - c.y);
        if (fmaxf(dx, dy) <= e) {
            ex = fmaxf(ex, dx);
            ey = fmaxf(ey, dy);
        }
    }
    for (int j = s - 1; j >= 0; --j) {
        const float2 c = pt(j);
        const float dx = ps.x - c.x;
        if (dx > e) break;
        const float dy = fabsf(ps.y - c.y);
        if (fmaxf(dx, dy) <= e) {
            ex = fmaxf(ex, dx);
            ey = fmaxf(ey, dy);
        }
    }
}

__device__ __forceinline__ double block_sum(double v, double* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) red[w] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x < 32) {
        int nw = (blockDim.x + 31) >> 5;
        t = threadIdx.x < nw ? red[threadIdx.x] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    }
    return t;  // valid in thread 0
}

}  // namespace ndf
