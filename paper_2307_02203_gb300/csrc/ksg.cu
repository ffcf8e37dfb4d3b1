// KSG mutual-information volumes: algorithm 1 of the k-NN estimator cited in
// Sec. 3.2 (timed on the CPU in Sec. 6.2, Table 1), for R reference vertices
// against every query vertex.
//
// Per pair (x = reference column, y = query column, M joint samples):
//   d_ij  = max(|x_i - x_j|, |y_i - y_j|)           FP32, exactly rounded
//   eps_i = k-th smallest d_ij over j != i
//         = (k+1)-th smallest over all j (the self distance 0 is always the smallest)
//   nx_i  = #{j != i : |x_i - x_j| < eps_i},  ny_i likewise
//   I     = psi(k) + psi(M) - (1/M) sum_i [psi(nx_i + 1) + psi(ny_i + 1)]   (FP64)
//
// GPU design:
//   stage   one CTA per reference sorts its column (values + member ids).
//   volume  persistent CTAs walk work items (reference group, tile of VT query
//           vertices).  The tile's query columns and their sorted copies (sorted
//           once per field) are loaded once, coalesced across the VT vertices, and
//           serve the G references of the group.  For each (reference, vertex)
//           the CTA lays the joint points out in x-sorted order in a padded shared
//           array; thread t owns the 4 consecutive sorted points 4t..4t+3 (and
//           4(t+T).. when M > 4T) and visits candidates outward in x-order, all
//           lanes of a warp in lockstep on consecutive positions (no bank
//           conflicts), the running top-(k+1) distances in registers.  Per
//           candidate one packed subtract per point gives (dx, dy), the distance
//           is one min/max, the threshold test u = d - t runs on the FMA pipe
//           (negative exactly when d < t; no flush to zero), the four tests merge
//           in a min tree, and a branch-free min/max network inserts.
//   modes   brute force: every other point exactly once, wrapping through a
//           doubled copy of the array.  Pruned (exact): no wrap; one side of a
//           thread's scan ends at the first candidate whose x-gap to the thread's
//           outermost point on that side reaches the largest current threshold of
//           its points.  Every later candidate on that side has at least that gap,
//           hence at least that max-norm distance, and an insert needs a strictly
//           smaller one; thresholds only shrink, so eps_i is the brute-force value
//           bit for bit.  A warp leaves the scan when all its lanes are done.
//   counts  binary search in the sorted x and in the column's sorted copy with the
//           same FP32 |difference| < eps predicate (monotone in sorted order); the
//           digamma sum is FP64, block-reduced.
#include <float.h>
#include <limits.h>
#include <math.h>

#include <algorithm>

#include "device_common.cuh"
#include "ksg_common.cuh"
#include "ndf_internal.h"

namespace ndf {

constexpr int kKsgPts = 4;  // sorted points owned by one thread
constexpr int kKsgMaxThreads = 512;

__host__ __device__ __forceinline__ int padi(int i) { return i + (i >> 2); }  // bank padding

// ---------------------------------------------------------------- stage
// one CTA per reference: sorted reference values and their member ids
// (refs == nullptr: references ref0, ref0 + 1, ...)
// A device-resident index outside [0, N) (host-given ones are checked before the
// launch) stages NaN values with the identity order: the reference's volume is
// meaningless but every later access stays in bounds, and the status word tells
// the next host check.
__global__ void __launch_bounds__(1024)
    ksg_stage_kernel(const float* __restrict__ field, int M, int64_t N,
                     const int64_t* __restrict__ refs, int64_t ref0, float* __restrict__ xs_all,
                     int* __restrict__ perm_all, unsigned* __restrict__ status,
                     unsigned long long* __restrict__ work) {
    pdl_launch();
    if (blockIdx.x == 0 && threadIdx.x == 0) *work = 0ull;  // the searches' work counter
    __shared__ float key[kKsgMaxM];
    __shared__ int val[kKsgMaxM];
    const int64_t ref = refs ? refs[blockIdx.x] : ref0 + blockIdx.x;
    if (ref < 0 || ref >= N) {
        if (threadIdx.x == 0 && status) atomicOr(status, kDevBadInput);
        for (int i = threadIdx.x; i < M; i += blockDim.x) {
            xs_all[(int64_t)blockIdx.x * M + i] = __int_as_float(0x7fc00000);
            perm_all[(int64_t)blockIdx.x * M + i] = i;
        }
        return;
    }
    int n2 = 1;
    while (n2 < M) n2 <<= 1;
    for (int i = threadIdx.x; i < n2; i += blockDim.x) {
        key[i] = i < M ? field[(int64_t)i * N + ref] : FLT_MAX;
        val[i] = i < M ? i : INT_MAX;
    }
    __syncthreads();
    for (int kk = 2; kk <= n2; kk <<= 1) {
        for (int j = kk >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < n2; i += blockDim.x) {
                const int l = i ^ j;
                if (l > i) {
                    const bool up = (i & kk) == 0;
                    const float a = key[i], b = key[l];
                    const int va = val[i], vb = val[l];
                    const bool gt = (a > b) || (a == b && va > vb);
                    if (gt == up) {
                        key[i] = b; key[l] = a;
                        val[i] = vb; val[l] = va;
                    }
                }
            }
            __syncthreads();
        }
    }
    float* xs = xs_all + (int64_t)blockIdx.x * M;
    int* pm = perm_all + (int64_t)blockIdx.x * M;
    for (int i = threadIdx.x; i < M; i += blockDim.x) {
        xs[i] = key[i];
        pm[i] = val[i];
    }
}

// The same for up to 1024 members, one warp per reference: RG (key, member) pairs per lane,
// element 32 r + lane in register r, sorted by a bitonic network (strides of 32 and more are
// register pairs, the others shuffles).  No barriers and 32 warps' worth of references per SM
// at once: 100,000 references of 500 members take 0.99 ms instead of 3.97 ms with one CTA of
// 1024 threads and 45 barriers each.
// A lone reference with many members stays with the CTA above (launch_ksg).
__device__ __forceinline__ bool stage_less(float a, int va, float b, int vb) {
    return a < b || (a == b && va < vb);
}
template <int RG, int RS, int SIZE>
__device__ __forceinline__ void stage_register_strides(float (&key)[RG], int (&val)[RG]) {
    if constexpr (RS >= 1) {
#pragma unroll
        for (int r = 0; r < RG; ++r) {
            if (r & RS) continue;
            const int q = r | RS;
            const bool up = ((r * 32) & SIZE) == 0;
            if (up ? stage_less(key[q], val[q], key[r], val[r]) : stage_less(key[r], val[r], key[q], val[q])) {
                const float tk = key[r];
                const int tv = val[r];
                key[r] = key[q];
                val[r] = val[q];
                key[q] = tk;
                val[q] = tv;
            }
        }
        stage_register_strides<RG, RS / 2, SIZE>(key, val);
    }
}
template <int RG, int SIZE>
__device__ __forceinline__ void stage_sort(float (&key)[RG], int (&val)[RG]) {
    if constexpr (SIZE <= 32 * RG) {
        const int lane = threadIdx.x & 31;
        stage_register_strides<RG, SIZE / 64, SIZE>(key, val);
#pragma unroll 1
        for (int stride = SIZE >= 32 ? 16 : SIZE / 2; stride > 0; stride >>= 1) {
            const bool lower = (lane & stride) == 0;
#pragma unroll
            for (int r = 0; r < RG; ++r) {
                const float ok = __shfl_xor_sync(0xffffffffu, key[r], stride);
                const int ov = __shfl_xor_sync(0xffffffffu, val[r], stride);
                const bool up = ((r * 32 + lane) & SIZE) == 0;
                if (stage_less(ok, ov, key[r], val[r]) == (lower == up)) {
                    key[r] = ok;
                    val[r] = ov;
                }
            }
        }
        stage_sort<RG, SIZE * 2>(key, val);
    }
}
template <int RG>
__global__ void __launch_bounds__(128)
    ksg_stage_warp_kernel(const float* __restrict__ field, int M, int64_t N, const int64_t* __restrict__ refs,
                          int64_t ref0, int R, float* __restrict__ xs_all, int* __restrict__ perm_all,
                          unsigned* __restrict__ status, unsigned long long* __restrict__ work) {
    const int lane = threadIdx.x & 31;
    const int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    pdl_launch();
    if (row == 0 && lane == 0) *work = 0ull;
    if (row >= R) return;
    const int64_t ref = refs ? refs[row] : ref0 + row;
    float* xs = xs_all + row * M;
    int* pm = perm_all + row * M;
    if (ref < 0 || ref >= N) {
        if (lane == 0 && status) atomicOr(status, kDevBadInput);
        for (int i = lane; i < M; i += 32) {
            xs[i] = __int_as_float(0x7fc00000);
            pm[i] = i;
        }
        return;
    }
    float key[RG];
    int val[RG];
#pragma unroll
    for (int r = 0; r < RG; ++r) {
        const int i = 32 * r + lane;
        key[r] = i < M ? field[(int64_t)i * N + ref] : FLT_MAX;
        val[r] = i < M ? i : INT_MAX;
    }
    stage_sort<RG, 2>(key, val);
#pragma unroll
    for (int r = 0; r < RG; ++r) {
        const int i = 32 * r + lane;
        if (i < M) {
            xs[i] = key[r];
            pm[i] = val[r];
        }
    }
}

// ---------------------------------------------------------------- helpers
__device__ __forceinline__ unsigned long long pack_f2(float2 v) {
    return ((unsigned long long)__float_as_uint(v.y) << 32) | __float_as_uint(v.x);
}

// (a.x - b.x, a.y - b.y), each rounded to nearest like a scalar FP32 subtract
__device__ __forceinline__ float2 sub_f32x2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return make_float2(__uint_as_float((unsigned)d), __uint_as_float((unsigned)(d >> 32)));
}

struct KsgArgs {
    const float* field;   // query field [M][N]
    const float* sorted;  // its columns sorted ascending [M][N]
    int M, k, VT, G, R;
    int64_t N, v_begin, v_end;
    const float* xs_all;  // [R][M] sorted reference values
    const int* perm_all;  // [R][M] member id of each sorted position
    const double* psi;    // psi(n), n <= M + 1
    const long long* psi_fix;  // the same in fixed point, with M's bits (psi_fix_bits)
    double psi_scale;     // 2^-bits
    float* out;           // out[r * out_stride + (v - v_begin)]
    int64_t out_stride;
    int variant;          // KSG algorithm 1 or 2
    int paired;           // pairs (reference i, vertex v_begin + i) only, R = v_end - v_begin
    double* dbg_mi;       // debug outputs for (reference 0, vertex v_begin), may be null
    float* dbg_eps;       // eps (algorithm 1) or the x extent (algorithm 2)
    float* dbg_ey;        // the y extent (algorithm 2)
    int32_t* dbg_nx;
    int32_t* dbg_ny;
    unsigned long long* evals;  // distance evaluations performed (self excluded), may be null
};

// shared-memory carve-up (bytes) of the brute-force kernel
struct KsgSmem {
    size_t red, xsg, permg, ytile, ystile, pts, total;
    __host__ __device__ KsgSmem(int M, int VT, int G) {
        size_t o = 0;
        red = o; o += 33 * sizeof(double);
        xsg = o; o += sizeof(float) * (size_t)M * G;
        permg = o; o += sizeof(int) * (size_t)M * G;
        o = (o + 15) & ~size_t(15);
        ytile = o; o += sizeof(float) * (size_t)M * VT;
        ystile = o; o += sizeof(float) * (size_t)M * VT;
        o = (o + 15) & ~size_t(15);
        pts = o; o += sizeof(float2) * (size_t)(padi(2 * M) + 4);
        total = o;
    }
};

// ---------------------------------------------------------------- volume
template <int K1>
__global__ void __launch_bounds__(kKsgMaxThreads) ksg_volume_kernel(KsgArgs A) {
    extern __shared__ __align__(16) unsigned char smem[];
    const KsgSmem L(A.M, A.VT, A.G);
    double* red = reinterpret_cast<double*>(smem + L.red);
    float* xsg = reinterpret_cast<float*>(smem + L.xsg);
    int* permg = reinterpret_cast<int*>(smem + L.permg);
    float* ytile = reinterpret_cast<float*>(smem + L.ytile);
    float* ystile = reinterpret_cast<float*>(smem + L.ystile);
    float2* pts = reinterpret_cast<float2*>(smem + L.pts);

    const int M = A.M, T = blockDim.x, tid = threadIdx.x;
    const int64_t N = A.N;
    const int64_t nv = A.v_end - A.v_begin;
    const int64_t tiles = (nv + A.VT - 1) / A.VT;
    const int groups = (A.R + A.G - 1) / A.G;
    const double psi_k = A.psi[A.k], psi_M = A.psi[M];
    unsigned long long my_evals = 0;
    int loaded_group = -1;

    for (int64_t item = blockIdx.x; item < (int64_t)groups * tiles; item += gridDim.x) {
        const int group = (int)(item / tiles);
        const int64_t tile = item - (int64_t)group * tiles;
        const int r0 = group * A.G;
        const int gcount = A.R - r0 < A.G ? A.R - r0 : A.G;
        const int64_t vt0 = A.v_begin + tile * A.VT;
        const int vcount = (int)(A.v_end - vt0 < A.VT ? A.v_end - vt0 : A.VT);
        __syncthreads();  // the previous item is done with every shared buffer
        if (group != loaded_group) {
            for (int i = tid; i < gcount * M; i += T) {
                xsg[i] = A.xs_all[(int64_t)r0 * M + i];
                permg[i] = A.perm_all[(int64_t)r0 * M + i];
            }
            loaded_group = group;
        }
        for (int idx = tid; idx < M * A.VT; idx += T) {
            const int m = idx / A.VT, p = idx - m * A.VT;
            const bool in = p < vcount;
            ytile[p * M + m] = in ? __ldcs(A.field + (int64_t)m * N + vt0 + p) : 0.0f;
            ystile[p * M + m] = in ? __ldcs(A.sorted + (int64_t)m * N + vt0 + p) : 0.0f;
        }
        for (int p = 0; p < vcount; ++p) {
            const float* ycol = ytile + p * M;
            const float* ys = ystile + p * M;  // the column, sorted (for n_y)
            for (int g = 0; g < gcount; ++g) {
                const float* xs = xsg + (size_t)g * M;
                const int* perm = permg + (size_t)g * M;
                __syncthreads();  // tiles ready / the previous pair is done with pts
                for (int s = tid; s < M; s += T) {
                    const float2 q = make_float2(xs[s], ycol[perm[s]]);
                    pts[padi(s)] = q;
                    pts[padi(s + M)] = q;
                }
                __syncthreads();

                double acc = 0.0;
                for (int base = 0; base < M; base += kKsgPts * T) {
                    const int b0 = base + kKsgPts * tid;
                    const int n_own = M - b0 >= kKsgPts ? kKsgPts : (M - b0 > 0 ? M - b0 : 0);
                    // ---- joint k-NN: top-(k+1) distances (self included) per owned point
                    unsigned long long P[kKsgPts];
                    float px[kKsgPts], py[kKsgPts];
                    float a[kKsgPts][K1];
#pragma unroll
                    for (int q = 0; q < kKsgPts; ++q) {
                        // a missing point sits at +inf: never inserted
                        const bool valid = q < n_own;
                        const float2 pq = valid ? pts[padi(b0 + q)] : make_float2(INFINITY, INFINITY);
                        px[q] = pq.x;
                        py[q] = pq.y;
                        P[q] = pack_f2(pq);
#pragma unroll
                        for (int j = 0; j < K1; ++j) a[q][j] = FLT_MAX;
                    }
                    auto visit = [&](float2 c) {
                        const unsigned long long C = pack_f2(c);
                        float d[kKsgPts], u[kKsgPts];
#pragma unroll
                        for (int q = 0; q < kKsgPts; ++q) {
                            const float2 dd = sub_f32x2(P[q], C);
                            d[q] = fmaxf(fabsf(dd.x), fabsf(dd.y));
                            u[q] = d[q] - a[q][K1 - 1];
                        }
                        if (fminf(fminf(u[0], u[1]), fminf(u[2], u[3])) < 0.0f) {
#pragma unroll
                            for (int q = 0; q < kKsgPts; ++q) topk_insert<K1>(a[q], d[q]);
                        }
                    };
                    if (n_own > 0) {
#pragma unroll
                        for (int c = 0; c < kKsgPts; ++c)
                            if (c < n_own) visit(pts[padi(b0 + c)]);
                    }
                    if (n_own > 0) {
                        const int rb = b0 + n_own - 1, lb = b0 + M;
                        const int Rn = (M - n_own + 1) >> 1, Ln = (M - n_own) >> 1;
                        for (int o = 1; o <= Rn; ++o) {
                            visit(pts[padi(rb + o)]);
                            if (o <= Ln) visit(pts[padi(lb - o)]);
                        }
                        my_evals += (unsigned long long)n_own * (unsigned long long)(M - 1);
                    }
                    // ---- marginal counts and the digamma sum
                    const bool dbg = A.dbg_eps && r0 + g == 0 && p == 0 && tile == 0;
#pragma unroll
                    for (int q = 0; q < kKsgPts; ++q) {
                        if (q < n_own) {
                            const float e = a[q][K1 - 1];
                            int cx, cy;
                            float ex = e, ey = e;
                            if (A.variant == 2) {
                                alg2_extents([&](int j) { return pts[padi(j)]; }, M, b0 + q,
                                             make_float2(px[q], py[q]), e, ex, ey);
                                cx = count_le([&](int j) { return xs[j]; }, M, px[q], ex) - 1;
                                cy = count_le([&](int j) { return ys[j]; }, M, py[q], ey) - 1;
                                acc += A.psi[cx] + A.psi[cy];
                            } else {
                                const int self = e > 0.0f ? 1 : 0;
                                cx = count_within(xs, M, px[q], e) - self;
                                cy = count_within(ys, M, py[q], e) - self;
                                acc += A.psi[cx + 1] + A.psi[cy + 1];
                            }
                            if (dbg) {
                                const int mi = perm[b0 + q];
                                A.dbg_eps[mi] = ex;
                                if (A.dbg_ey) A.dbg_ey[mi] = ey;
                                A.dbg_nx[mi] = cx;
                                A.dbg_ny[mi] = cy;
                            }
                        }
                    }
                }
                const double tot = block_sum(acc, red);
                if (tid == 0) {
                    const double mi = psi_k - (A.variant == 2 ? 1.0 / A.k : 0.0) + psi_M - tot / (double)M;
                    const int64_t v = vt0 + p;
                    A.out[(int64_t)(r0 + g) * A.out_stride + (v - A.v_begin)] = (float)mi;
                    if (A.dbg_mi && r0 + g == 0 && p == 0 && tile == 0) *A.dbg_mi = mi;
                }
            }
        }
    }
    if (A.evals) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) my_evals += __shfl_xor_sync(0xffffffffu, my_evals, o);
        if ((tid & 31) == 0) atomicAdd(A.evals, my_evals);
    }
}

// ---------------------------------------------------------------- pruned volume
// Exact pruned search.  A group of kGroupWarps warps takes one (reference, vertex)
// pair at a time from a global counter, so groups never wait for one another.
// Within a pair each lane scans one point at a time, outward in x-order; a side of
// the scan stops at the first candidate whose x-gap reaches the point's current
// k-th distance (self excluded: the list b holds the k nearest others, eps_i =
// b[k-1]).  Every later candidate on that side is at least that far in x, hence
// in the max-norm, and an insert needs a strictly smaller distance; the threshold
// only shrinks, so eps_i equals the brute-force value bit for bit.
//
// Each step takes two candidates, one per scan slot, and is branch-free: the
// point array carries two sentinels at each end (x = -inf / +inf, an x-gap no
// threshold passes), a closed slot re-reads a candidate beyond its threshold, and
// both distances enter the list through one merge network (measured 10% faster
// than two single inserts).  Every kServiceSteps steps a lane whose point is done
// stores eps and takes the next point from the group's counter (extremes of the x
// distribution first: their scans are the longest).  The counts and the digamma
// sum follow in an evenly split loop over the points.  The group's warps share
// the pair's arrays (16 B x M), which sets how many warps fit on an SM.
constexpr int kServiceSteps = 4;
constexpr int kPad = 2;            // sentinels per end
constexpr int kGroupWarps = 2;     // warps per pair
constexpr int kMaxGroupsPerCta = 14;
constexpr int kGroupSmemPerM = sizeof(float2) + 2 * sizeof(float);  // pts, ys, eps
struct GroupCtl {
    unsigned long long item;
    int next;
    int pad;
    double part[kGroupWarps];
};
constexpr int kGroupSmemFixed = 2 * kPad * sizeof(float2) + sizeof(GroupCtl);

// b ascending; inserts lo <= hi, keeping the KK smallest:
// new b[p] = min(b[p], max(b[p-1], lo), max(b[p-2], hi))
template <int KK>
__device__ __forceinline__ void insert2(float (&b)[KK], float lo, float hi) {
#pragma unroll
    for (int p = KK - 1; p >= 2; --p) b[p] = fminf(fminf(b[p], fmaxf(b[p - 1], lo)), fmaxf(b[p - 2], hi));
    if (KK >= 2) b[1] = fminf(fminf(b[1], fmaxf(b[0], lo)), hi);
    b[0] = fminf(b[0], lo);
}

__device__ __forceinline__ int count_within_x(const float2* a, int n, float c, float e) {
    int lo = 0, len = n;
    while (len > 0) {  // first p with fl(c - a[p].x) < e
        const int h = len >> 1;
        if (!((c - a[lo + h].x) < e)) { lo += h + 1; len -= h + 1; }
        else len = h;
    }
    int hi = 0;
    len = n;
    while (len > 0) {  // first p with fl(a[p].x - c) >= e
        const int h = len >> 1;
        if (!((a[hi + h].x - c) >= e)) { hi += h + 1; len -= h + 1; }
        else len = h;
    }
    return hi > lo ? hi - lo : 0;
}

__device__ __forceinline__ void group_sync(int group) {
    asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "r"(32 * kGroupWarps) : "memory");
}

template <int K1>
__global__ void __launch_bounds__(32 * kGroupWarps * kMaxGroupsPerCta, 1)
    ksg_pruned_kernel(KsgArgs A, unsigned long long* work) {
    constexpr int KK = K1 - 1;
    constexpr int GT = 32 * kGroupWarps;  // threads per group
    extern __shared__ __align__(16) unsigned char smem[];
    const int M = A.M, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int group = warp / kGroupWarps, gw = warp % kGroupWarps, gt = threadIdx.x % GT;
    const int ngroups = blockDim.x / GT;
    GroupCtl* ctl = reinterpret_cast<GroupCtl*>(smem) + group;
    float2* S = reinterpret_cast<float2*>(reinterpret_cast<GroupCtl*>(smem) + ngroups) +
                (size_t)group * (M + 2 * kPad) + kPad;
    float* ys = reinterpret_cast<float*>(reinterpret_cast<float2*>(reinterpret_cast<GroupCtl*>(smem) +
                                                                   ngroups) +
                                         (size_t)ngroups * (M + 2 * kPad)) +
                (size_t)group * 2 * M;
    float* epsw = ys + M;
    const int64_t N = A.N, nv = A.v_end - A.v_begin;
    const unsigned long long items =
        A.paired ? (unsigned long long)nv : (unsigned long long)A.R * (unsigned long long)nv;
    const double psi_k = A.psi[A.k], psi_M = A.psi[M];
    const unsigned lt_mask = (1u << lane) - 1u;
    if (gt < kPad) {
        S[-1 - gt] = make_float2(-INFINITY, 0.0f);
        S[M + gt] = make_float2(INFINITY, 0.0f);
    }
    unsigned my_evals = 0;
    unsigned long long evals_total = 0;

    for (;;) {
        group_sync(group);  // the previous pair is finished by both warps
        if (gt == 0) {
            ctl->item = atomicAdd(work, 1ull);
            ctl->next = 0;
        }
        group_sync(group);
        const unsigned long long item = ctl->item;
        if (item >= items) break;
        const int r = A.paired ? (int)item : (int)(item / (unsigned long long)nv);
        const int64_t v = A.v_begin + (int64_t)(A.paired ? item : item - (unsigned long long)r * nv);
        const float* xs = A.xs_all + (int64_t)r * M;
        const int* perm = A.perm_all + (int64_t)r * M;
        for (int s = gt; s < M; s += GT) {
            S[s] = make_float2(xs[s], A.field[(int64_t)perm[s] * N + v]);
            ys[s] = A.sorted[(int64_t)s * N + v];
        }
        group_sync(group);

        // ---- joint k-NN distances.  Two scan slots per lane, each a position and a
        // stride: slot 1 starts right of the point (+1), slot 2 left (-1).  A slot
        // advances while its candidate's x-gap is below the threshold and otherwise
        // stays on that candidate, so a closed side costs no bookkeeping.  At the
        // service points a lane whose one side has closed sends that slot to the
        // other side (the two slots then interleave with stride 2), a lane whose
        // both sides have closed stores eps and takes a new point.  Idle lanes point
        // both slots at sentinels.
        int i = -1, pr = M, pl = -1, sr = 1, sl = -1;
        bool drained = false;  // the group's counter has passed M
        unsigned steps = 0;
        float px = 0.0f;
        unsigned long long P = 0;
        float b[KK];
#pragma unroll
        for (int c = 0; c < KK; ++c) b[c] = FLT_MAX;
        for (;;) {
            if (i >= 0) {
                const float t = b[KK - 1];
                const bool dead1 = fabsf(px - S[pr].x) >= t;
                const bool dead2 = fabsf(px - S[pl].x) >= t;
                if (dead1 && dead2) {
                    epsw[i] = t;
                    my_evals += 2u * steps;
                    i = -1;
                    pr = M;
                    pl = -1;
                } else if (dead1 && sr == 1) {
                    pr = pl + sl;  // slot 1 joins the left side
                    sr = 2 * sl;
                    sl = sr;
                } else if (dead2 && sl == -1) {
                    pl = pr + sr;  // slot 2 joins the right side
                    sl = 2 * sr;
                    sr = sl;
                }
            }
            const unsigned idle = __ballot_sync(0xffffffffu, i < 0);
            if (drained && idle == 0xffffffffu) break;
            if (!drained && idle != 0u) {
                int base = 0;
                if (lane == 0) base = atomicAdd(&ctl->next, __popc(idle));
                base = __shfl_sync(0xffffffffu, base, 0);
                const int g = base + __popc(idle & lt_mask);
                if (i < 0 && g < M) {
                    i = (g & 1) ? M - 1 - (g >> 1) : (g >> 1);
                    const float2 pi = S[i];
                    px = pi.x;
                    P = pack_f2(pi);
#pragma unroll
                    for (int c = 0; c < KK; ++c) b[c] = FLT_MAX;
                    pr = i + 1;
                    pl = i - 1;
                    sr = 1;
                    sl = -1;
                    steps = 0;
                }
                drained = base + __popc(idle) >= M;
            }
            if (i >= 0) steps += kServiceSteps;
#pragma unroll
            for (int st = 0; st < kServiceSteps; ++st) {
                const float2 e1 = sub_f32x2(P, pack_f2(S[pr]));
                const float2 e2 = sub_f32x2(P, pack_f2(S[pl]));
                const float g1 = fabsf(e1.x), g2 = fabsf(e2.x);
                const float t = b[KK - 1];
                const float d1 = fmaxf(g1, fabsf(e1.y)), d2 = fmaxf(g2, fabsf(e2.y));
                insert2<KK>(b, fminf(d1, d2), fmaxf(d1, d2));
                // the pre-insert threshold makes the side test conservative (exact)
                if (g1 < t) pr += sr;
                if (g2 < t) pl += sl;
            }
        }
        group_sync(group);  // every eps of the pair is stored

        // ---- marginal counts and the digamma sum
        const bool dbg = A.dbg_eps && r == 0 && v == A.v_begin;
        double acc = 0.0;
        for (int s = gt; s < M; s += GT) {
            const float e = epsw[s];
            const float2 ps = S[s];
            int cx, cy;
            float ex = e, ey = e;
            if (A.variant == 2) {
                alg2_extents([&](int j) { return S[j]; }, M, s, ps, e, ex, ey);
                cx = count_le([&](int j) { return S[j].x; }, M, ps.x, ex) - 1;
                cy = count_le([&](int j) { return ys[j]; }, M, ps.y, ey) - 1;
                acc += A.psi[cx] + A.psi[cy];
            } else {
                const int self = e > 0.0f ? 1 : 0;
                cx = count_within_x(S, M, ps.x, e) - self;
                cy = count_within(ys, M, ps.y, e) - self;
                acc += A.psi[cx + 1] + A.psi[cy + 1];
            }
            if (dbg) {
                const int mi = perm[s];
                A.dbg_eps[mi] = ex;
                if (A.dbg_ey) A.dbg_ey[mi] = ey;
                A.dbg_nx[mi] = cx;
                A.dbg_ny[mi] = cy;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) ctl->part[gw] = acc;
        group_sync(group);
        if (gt == 0) {
            double tot = 0.0;
#pragma unroll
            for (int w = 0; w < kGroupWarps; ++w) tot += ctl->part[w];
            const double mi = psi_k - (A.variant == 2 ? 1.0 / A.k : 0.0) + psi_M - tot / (double)M;
            A.out[A.paired ? (v - A.v_begin) : (int64_t)r * A.out_stride + (v - A.v_begin)] = (float)mi;
            if (dbg && A.dbg_mi) *A.dbg_mi = mi;
        }
        evals_total += my_evals;
        my_evals = 0;
    }
    if (A.evals) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) evals_total += __shfl_xor_sync(0xffffffffu, evals_total, o);
        if (lane == 0) atomicAdd(A.evals, evals_total);
    }
}

// ---------------------------------------------------------------- block search
// The same estimator (algorithm 1) with a two-level search.  The members of a
// pair are cut into x-blocks of 64 consecutive x-ranks; inside each block they are
// sorted by y (one warp-wide bitonic sort of 64 (y, rank) keys, two per lane).  A
// lane takes the member at one position of block b and
//   scans its own block outward in y from its own position,
//   then the blocks b + 1, b - 1, b + 2, ... : a side stops at the first block whose
//   x-gap (the block's nearest x-rank) reaches the lane's current k-th distance;
//   in a block it binary-searches its y and scans outward in y while the y-gap is
//   below the threshold.
// Every skipped member is at least the threshold away in x or in y, an insert
// needs a strictly smaller distance, and the threshold only shrinks, so eps_i is
// the brute-force value bit for bit.  A lane visits about 20 candidates at
// M = 1000, k = 8 (the x-strip of the pruned kernel: about 120).  The warp runs
// the blocks of its lanes in lock step (a per-lane state machine with dynamic
// members, measured: 1.7x slower, the block changes with their binary searches
// diverge on almost every step); each step takes one candidate from each end of
// the block scan into the two-value merge insert.  Two warps share a pair's
// arrays (x sorted, y sorted, the block-sorted points: 16 B x M).
constexpr int kBlk = 64;  // x-ranks per block (two per lane in the block sort)
struct BlockCtl {
    unsigned long long item;
    double part[kGroupWarps];
};
// block b's kBlk points sit at 1 + b * kBlkStride + p, between +inf separators at
// b * kBlkStride (both scan directions stop on |y - y_i| = inf without bounds checks)
constexpr int kBlkStride = kBlk + 1;
constexpr int kTaskRows = 8;                     // y-positions per block in a warp task
constexpr int kTaskBlocks = 32 / kTaskRows;      // blocks in a warp task
constexpr int kTaskQuads = kBlk / kTaskRows;     // position groups of a block
__host__ __device__ inline size_t block_group_bytes(int M) {
    const int nb = (M + kBlk - 1) / kBlk;
    return sizeof(BlockCtl) + sizeof(float2) * ((size_t)nb * kBlkStride + 1) +
           2 * sizeof(float) * (size_t)((M + 3) & ~3);
}

constexpr int kBlkRegs = kBlk / 32;              // sort keys per lane

// warp-wide ascending bitonic sort of kBlk (key, val) pairs, element e = 32 r + lane
// in register r; (key, val) compared lexicographically (val unique), so the order
// is total.  Strides of 32 and more compare two registers of one lane.
__device__ __forceinline__ void warp_sort_block(float (&key)[kBlkRegs], int (&val)[kBlkRegs]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int size = 2; size <= kBlk; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            if (stride >= 32) {
                const int rs = stride / 32;
#pragma unroll
                for (int r = 0; r < kBlkRegs; ++r) {
                    if (r & rs) continue;
                    const int q = r | rs;
                    const bool up = ((r * 32) & size) == 0;
                    const bool q_less = key[q] < key[r] || (key[q] == key[r] && val[q] < val[r]);
                    if (up == q_less) {  // the lower element of an ascending pair keeps the smaller
                        const float tk = key[r];
                        const int tv = val[r];
                        key[r] = key[q];
                        val[r] = val[q];
                        key[q] = tk;
                        val[q] = tv;
                    }
                }
                continue;
            }
#pragma unroll
            for (int r = 0; r < kBlkRegs; ++r) {
                const float ok = __shfl_xor_sync(0xffffffffu, key[r], stride);
                const int ov = __shfl_xor_sync(0xffffffffu, val[r], stride);
                const bool up = ((r * 32 + lane) & size) == 0;
                const bool lower = (lane & stride) == 0;
                const bool other_less = ok < key[r] || (ok == key[r] && ov < val[r]);
                if (lower == up ? other_less : !other_less) {
                    key[r] = ok;
                    val[r] = ov;
                }
            }
        }
    }
}

// the sort keys of block b: query values of x-ranks b kBlk + 32 r + lane (+inf past M)
__device__ __forceinline__ void block_keys(const KsgArgs& A, const int* perm, int b, int64_t v,
                                           float (&key)[kBlkRegs], int (&val)[kBlkRegs]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int r = 0; r < kBlkRegs; ++r) {
        const int rank = b * kBlk + r * 32 + lane;
        key[r] = rank < A.M ? A.field[(int64_t)perm[rank] * A.N + v] : INFINITY;
        val[r] = rank;
    }
}

// lower bound of y in a block of kBlk ascending values (pads +inf): 0 .. kBlk - 1
__device__ __forceinline__ int block_lower_bound(const float2* blk, float y) {
    int pos = 0;
#pragma unroll
    for (int h = kBlk / 2; h > 0; h >>= 1)
        if (blk[pos + h - 1].x < y) pos += h;
    return pos;
}

// KSG algorithm 2 over the lane search's blocks: the largest fl(|x_j - xi|) and fl(|y_j - yi|)
// over the members j whose max-norm distance to (xi, yi) is <= e (the member itself adds
// zeros).  Blocks from the member's own block b0 outward in x while the block's nearest
// x-rank is within e (fl(x_j - xi) is monotone in x_j); inside a block, outward in y while
// |dy| <= e (the +inf separators stop both scans), from the member's own position p0 there and
// from enter(block) = the number of members below yi elsewhere.
template <class Enter>
__device__ __forceinline__ void block_extents(const float2* blk, const float2* bx, int nb, int bs, int b0, int p0,
                                              float xi, float yi, float e, float& ex, float& ey, Enter&& enter) {
    ex = 0.0f;
    ey = 0.0f;
    auto visit = [&](const float2* c) {  // false: beyond e in y
        const float dy = fabsf(c->x - yi), dx = fabsf(c->y - xi);
        if (!(dy <= e)) return false;
        if (dx <= e) {
            ex = fmaxf(ex, dx);
            ey = fmaxf(ey, dy);
        }
        return true;
    };
    auto scan = [&](int bb, int pos) {
        const float2* B = blk + 1 + bb * bs;  // (y, x), ascending y
        for (int u = pos; visit(B + u); ++u) {}
        for (int u = pos - 1; visit(B + u); --u) {}
    };
    scan(b0, p0);
    for (int bb = b0 + 1; bb < nb && bx[bb].x - xi <= e; ++bb) scan(bb, enter(bb));
    for (int bb = b0 - 1; bb >= 0 && xi - bx[bb].y <= e; --bb) scan(bb, enter(bb));
}

template <int K1>
__global__ void __launch_bounds__(32 * kGroupWarps * kMaxGroupsPerCta, 1)
    ksg_block_kernel(KsgArgs A, unsigned long long* work) {
    constexpr int KK = K1 - 1;
    constexpr int GT = 32 * kGroupWarps;
    extern __shared__ __align__(16) unsigned char smem[];
    const int M = A.M, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int group = warp / kGroupWarps, gw = warp % kGroupWarps, gt = threadIdx.x % GT;
    const int nb = (M + kBlk - 1) / kBlk;
    unsigned char* gbase = smem + (size_t)group * block_group_bytes(M);
    BlockCtl* ctl = reinterpret_cast<BlockCtl*>(gbase);
    float2* blk = reinterpret_cast<float2*>(gbase + sizeof(BlockCtl));  // (y, x), separated blocks
    float* xs = reinterpret_cast<float*>(blk + (size_t)nb * kBlkStride + 1);  // reference, x-sorted
    float* ys = xs + ((M + 3) & ~3);                                     // query, sorted
    const int64_t N = A.N, nv = A.v_end - A.v_begin;
    const unsigned long long items =
        A.paired ? (unsigned long long)nv : (unsigned long long)A.R * (unsigned long long)nv;
    const double psi_k = A.psi[A.k], psi_M = A.psi[M];
    unsigned long long evals_total = 0;

    for (;;) {
        group_sync(group);  // the previous pair is finished by both warps
        if (gt == 0) ctl->item = atomicAdd(work, 1ull);
        group_sync(group);
        const unsigned long long item = ctl->item;
        if (item >= items) break;
        const int r = A.paired ? (int)item : (int)(item / (unsigned long long)nv);
        const int64_t v = A.v_begin + (int64_t)(A.paired ? item : item - (unsigned long long)r * nv);
        const float* xsg = A.xs_all + (int64_t)r * M;
        const int* perm = A.perm_all + (int64_t)r * M;
        for (int s = gt; s < M; s += GT) {
            xs[s] = xsg[s];
            ys[s] = A.sorted[(int64_t)s * N + v];
        }
        // ---- blocks of kBlk x-ranks, each sorted by y; pads (y = x = +inf) sort last
        for (int b = gt; b <= nb; b += GT) blk[b * kBlkStride] = make_float2(INFINITY, INFINITY);
        for (int b = gw; b < nb; b += kGroupWarps) {
            float key[kBlkRegs];
            int val[kBlkRegs];
            block_keys(A, perm, b, v, key, val);
            warp_sort_block(key, val);
#pragma unroll
            for (int r2 = 0; r2 < kBlkRegs; ++r2)
                blk[1 + b * kBlkStride + r2 * 32 + lane] =
                    make_float2(key[r2], val[r2] < M ? xsg[val[r2]] : INFINITY);
        }
        group_sync(group);

        // ---- joint k-NN distance of each member, then its marginal counts
        const bool dbg = A.dbg_eps && r == 0 && v == A.v_begin;
        double acc = 0.0;
        unsigned long long my_evals = 0;
        // a warp task: the members at y-positions 8q .. 8q + 7 of blocks 4g .. 4g + 3 (lanes
        // of similar rank inside their blocks have similar windows, so the lock-step
        // scans waste fewer steps than with 32 consecutive members of one block)
        const int ntasks = ((nb + kTaskBlocks - 1) / kTaskBlocks) * kTaskQuads;
        for (int task = gw; task < ntasks; task += kGroupWarps) {
            const int b = (task / kTaskQuads) * kTaskBlocks + lane / kTaskRows;
            const int p = (task % kTaskQuads) * kTaskRows + lane % kTaskRows;
            const bool valid = b < nb && p < min(kBlk, M - b * kBlk);
            const float2 me = valid ? blk[1 + b * kBlkStride + p] : make_float2(INFINITY, INFINITY);
            const float yi = me.x, xi = me.y;
            float best[KK];  // the k nearest others, ascending
#pragma unroll
            for (int c = 0; c < KK; ++c) best[c] = FLT_MAX;
            // scan of block bb from positions up / dn outward while the y-gap is below
            // the threshold; a lane with on == false starts on the separators
            auto scan = [&](int bb, int up, int dn, bool on) {
                const float2* B = blk + 1 + (on ? bb : 0) * kBlkStride;
                if (!on) {
                    up = kBlk;
                    dn = -1;
                }
                const int up0 = up, dn0 = dn;
                for (;;) {
                    const float t = best[KK - 1];
                    const float2 cu = B[up], cd = B[dn];
                    const float dyu = cu.x - yi, dyd = yi - cd.x;
                    const bool au = fabsf(dyu) < t;  // false on a separator (and for pads: NaN)
                    const bool ad = fabsf(dyd) < t;
                    if (!__any_sync(0xffffffffu, au || ad)) break;
                    // a candidate outside the window has |dy| >= t, so its distance is >= t
                    // and leaves the list unchanged: no select needed (for a valid lane;
                    // the padding lanes' lists are never read)
                    const float du = fmaxf(fabsf(cu.y - xi), fabsf(dyu));
                    const float dd = fmaxf(fabsf(cd.y - xi), fabsf(dyd));
                    insert2<KK>(best, fminf(du, dd), fmaxf(du, dd));
                    up += au ? 1 : 0;
                    dn -= ad ? 1 : 0;
                }
                my_evals += (unsigned)((up - up0) + (dn0 - dn));
            };
            scan(b, p + 1, p - 1, valid);
            bool ron = valid, lon = valid;
            for (int dd = 1; dd < nb; ++dd) {
                const int br = b + dd, bleft = b - dd;
                if (br >= nb) ron = false;
                else if (ron && xs[br * kBlk] - xi >= best[KK - 1]) ron = false;  // nearest x of the block
                if (__any_sync(0xffffffffu, ron)) {
                    const int pos = ron ? block_lower_bound(blk + 1 + br * kBlkStride, yi) : 0;
                    scan(br, pos, pos - 1, ron);
                }
                if (bleft < 0) lon = false;
                else if (lon && xi - xs[min(bleft * kBlk + kBlk - 1, M - 1)] >= best[KK - 1]) lon = false;
                if (__any_sync(0xffffffffu, lon)) {
                    const int pos = lon ? block_lower_bound(blk + 1 + bleft * kBlkStride, yi) : 0;
                    scan(bleft, pos, pos - 1, lon);
                }
                if (!__any_sync(0xffffffffu, ron || lon)) break;
            }
            if (valid) {
                const float e = best[KK - 1];
                const int self = e > 0.0f ? 1 : 0;
                int cx, cy;
                count_within_pair(xs, ys, M, pow2_floor(M), xi, yi, e, cx, cy);
                cx -= self;
                cy -= self;
                acc += A.psi[cx + 1] + A.psi[cy + 1];
                // debug pair: eps by block position (scratch), put in member order below
                if (dbg) A.dbg_nx[b * kBlk + p] = __float_as_int(e);
            }
        }
        if (dbg) {
            // member ids: each block's sort again (deterministic) gives its positions' x-ranks.
            // Pass 1 moves eps from the position-indexed scratch (dbg_nx) to dbg_eps[member];
            // after every read of the scratch, pass 2 writes the counts over it.
            group_sync(group);
            for (int bq = gw; bq < nb; bq += kGroupWarps) {
                float key[kBlkRegs];
                int val[kBlkRegs];
                block_keys(A, perm, bq, v, key, val);
                warp_sort_block(key, val);
#pragma unroll
                for (int r2 = 0; r2 < kBlkRegs; ++r2)
                    if (val[r2] < M)
                        A.dbg_eps[perm[val[r2]]] = __int_as_float(A.dbg_nx[bq * kBlk + r2 * 32 + lane]);
            }
            group_sync(group);
            for (int bq = gw; bq < nb; bq += kGroupWarps) {
                float key[kBlkRegs];
                int val[kBlkRegs];
                block_keys(A, perm, bq, v, key, val);
                warp_sort_block(key, val);
#pragma unroll
                for (int r2 = 0; r2 < kBlkRegs; ++r2) {
                    if (val[r2] >= M) continue;
                    const int mi = perm[val[r2]];
                    const float e = A.dbg_eps[mi];
                    const float2 me = blk[1 + bq * kBlkStride + r2 * 32 + lane];
                    const int self = e > 0.0f ? 1 : 0;
                    if (A.dbg_ey) A.dbg_ey[mi] = e;
                    A.dbg_nx[mi] = count_within(xs, M, me.y, e) - self;
                    A.dbg_ny[mi] = count_within(ys, M, me.x, e) - self;
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) ctl->part[gw] = acc;
        evals_total += my_evals;
        group_sync(group);
        if (gt == 0) {
            double tot = 0.0;
#pragma unroll
            for (int w = 0; w < kGroupWarps; ++w) tot += ctl->part[w];
            const double mi = psi_k + psi_M - tot / (double)M;
            A.out[A.paired ? (v - A.v_begin) : (int64_t)r * A.out_stride + (v - A.v_begin)] = (float)mi;
            if (dbg && A.dbg_mi) *A.dbg_mi = mi;
        }
    }
    if (A.evals) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) evals_total += __shfl_xor_sync(0xffffffffu, evals_total, o);
        if (lane == 0) atomicAdd(A.evals, evals_total);
    }
}

// ---------------------------------------------------------------- lane-refill block search
// The same two-level search as ksg_block_kernel (x-blocks of W consecutive x-ranks
// sorted by the query value, +inf separators, the same window, x-gap and insert rules,
// so eps_i is again the brute-force value bit for bit), scheduled per lane instead of
// per block scan, and with the block order built from ranks instead of sorts:
//   - every member's rank in the query column (a binary search in the sorted copy; tied
//     members take consecutive ranks from a counter, in any order: neither eps nor the sums
//     depend on it) goes into its block's bitmap of ranks.
//     With the bitmap words' running counts, the number of a block's members below a rank is
//     two loads and a population count.  That gives a member's place in its block (no
//     sort: the former 64-key bitonic sorts took about 7 warp instructions per member, this
//     about 3) and, during the search, the point where a lane enters a neighbouring block
//     (before: a six-step binary search in a service step that few lanes share);
//   - a lane owns one member at a time and walks its own sequence of blocks: its own
//     block from its position outward, then the neighbouring blocks, at each switch
//     the side whose nearest x-rank is closer (a side ends at the first block whose
//     nearest x-rank is at least the current k-th distance away);
//   - a lane whose member is finished stores eps_i (by block position) and takes the
//     next member of its warp (the group's warps split the members evenly);
//   - block switches and refills run in a warp-uniform service step, entered only when at
//     least `switch_min` lanes wait or no lane is scanning, so the divergent code runs for
//     many lanes at once;
//   - every other lock step is the scan step of the block kernel for all lanes;
//   - the marginal counts (binary searches) and the digamma sum (in fixed point: the same sum in
//     any order, two integer adds for the slow FP64 pipe's one) follow in an evenly split pass
//     over the stored eps (for KSG algorithm 2 after the marginal extents of each member's
//     k-NN set, found over the same blocks: block_extents).
// What bounds it: the ALU pipe (the scan step's minima, maxima and compares issue at half
// rate; 77 % busy at M = 1000, k = 8) and the L1 data pipe (74 %, the lanes' scattered reads of
// shared memory 64 %); issue slots 65 %; 64,400 warp instructions per pair against 86,000 for
// the sorted 64-rank blocks before.  250 x 352 x 20 vertices, M = 1000, k = 8: 167.5 ms before,
// 130 - 133 ms now.
// Members are handed out in the block kernel's task order (8 y-positions of 4 neighbouring
// blocks per 32), so the lanes of a warp start on members of similar rank.  Shared memory per
// pair: the block-sorted points, the sorted query column, one word per member (its query
// value, then its rank, then eps) and the bitmaps (16 B x M + 5 B per block and 32 ranks);
// for algorithm 1 the sorted reference values sit in shared memory once per CTA when all pairs share
// the reference (and that costs no group, lane_plan), else they are read from the staging buffer in
// global memory (L1).
struct LaneCtl {
    unsigned long long item;
    unsigned long long pad;
    long long part[kGroupWarps];
};
__host__ __device__ inline int lane_slots(int nb, int lw) { return (((nb + 3) >> 2) << 2) << lw; }
// shared memory of one group (bytes from its base), W = 1 << lw ranks per block
struct LaneSmem {
    int blk, ys, eps, tab, below, bx, total;
    __host__ __device__ LaneSmem(int M, int lw) {
        const int nb = (M + (1 << lw) - 1) >> lw, nw = (M + 31) >> 5;
        int o = (int)sizeof(LaneCtl);
        blk = o; o += (int)sizeof(float2) * (M + nb + 1);
        ys = o; o += (int)sizeof(float) * ((M + 1) & ~1);
        eps = o; o += (int)sizeof(float) * ((M + 1) & ~1);
        bx = o; o += (int)sizeof(float2) * (nb + 2);
        tab = o; o += (int)sizeof(unsigned) * nb * nw;
        below = o; o += (nb * nw + 7) & ~7;
        total = (o + 15) & ~15;
    }
};
// ranks per block: the scan visits members inside the y-window of whole blocks, so wider blocks
// cost candidates that fail the x-test, narrower ones more block switches.  Measured (us a volume of
// 1.2e7 / M vertices, k = 8, 32 / 64 / 128 ranks): 1073 / 1080 / 1375 for M = 200, 973 / 935 / 1264 for
// M = 256, 1139 / 962 / 1030 for M = 600, 1166 / 981 / 1021 for M = 769, 1296 / 1086 / 1073 for M = 900,
// 1336 / 1131 / 1018 for M = 1000.
__host__ __device__ inline int lane_block_log2(int M) { return M > 850 ? 7 : M > 224 ? 6 : 5; }
// lock steps a warp may take per pair before it gives up (a safety bound far above
// any real schedule: every member visits at most nb blocks of W + 1 steps)
__host__ __device__ inline long long lane_step_bound(int nb, int lw) {
    return (long long)lane_slots(nb, lw) * (nb + 2) * ((1 << lw) + 4);
}
constexpr int kLaneMaxGroups = 14;  // groups per CTA: the most that leave a thread 72 registers
// The search of one pair by one warp: the joint k-NN distance of each of its members, to eps_s by block
// position.  gofs: the group's shared memory; returns (evaluations in bytes of points visited, gave up).
// A function of its own, not inlined: its registers are then allocated apart from those of the
// kernel's other phases, whose changes moved the scan's code by up to 3 % (88,000 vertices, M = 1000:
// inlined 7.14 ms with k = 8 and 5.31 with k = 4, as a function 6.80 and 5.13).
template <int KK>
__device__ __noinline__ uint2 lane_search(int gofs, int M, int lw, int gw, bool constant, int switch_min, int every) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr unsigned FULL = 0xffffffffu;
    // five scan steps, the default number, in a row (two: 6.90 ms in the case above, k = 8), but the longer
    // steps of more neighbours singly (M = 60, 200,000 vertices, k = 10: 1729 us with five)
    constexpr int kUnroll = KK > 8 ? 1 : 5;
    const int lane = threadIdx.x & 31;
    const int W = 1 << lw, nb = (M + W - 1) >> lw, nw = (M + 31) >> 5, bs = W + 1;
    const LaneSmem L(M, lw);
    float* eps_s = reinterpret_cast<float*>(smem + gofs + L.eps);
    const int* rank_s = reinterpret_cast<const int*>(eps_s);
    const unsigned* tab = reinterpret_cast<const unsigned*>(smem + gofs + L.tab);
    const unsigned char* below = smem + gofs + L.below;
    const float2* bx = reinterpret_cast<const float2*>(smem + gofs + L.bx) + 1;
    const int slots = lane_slots(nb, lw);
    const int step_bound = (int)min(lane_step_bound(nb, lw), (long long)INT_MAX);
    const int pt0 = gofs + L.blk + (int)sizeof(float2);  // block 0, position 0
    bool has = false, inblk = false;
    int up = pt0 - (int)sizeof(float2), dn = up;  // byte offsets; separators for an idle lane
    int nr = 0, nl = -1, rank = 0, slot_pos = 0;
    int next = 0;  // members handed out by this warp (task order, every kGroupWarps-th task)
    const int wslots = slots / kGroupWarps;
    float xi = 0.0f, yi = 0.0f;
    float best[KK];
#pragma unroll
    for (int c = 0; c < KK; ++c) best[c] = FLT_MAX;
    unsigned my_evals = 0;
    int steps = 0;
    for (;;) {
        const unsigned wm = __ballot_sync(FULL, has ? !inblk : next < wslots);
        const unsigned em = __ballot_sync(FULL, has && inblk);
        if (em == 0u && wm == 0u) break;
        if (em == 0u || __popc(wm) >= switch_min) {
            // service: block switches of the lanes whose window closed, then refills
            if (has && !inblk) {
                my_evals += (unsigned)(up - dn);
                const float t = best[KK - 1];
                const float x = constant ? yi : xi;
                const float gr = bx[nr].x - x, gl = x - bx[nl].y;
                const bool okr = gr < t, okl = gl < t;
                if (!okr && !okl) {
                    eps_s[slot_pos] = t;  // member finished
                    has = false;
                    my_evals -= (unsigned)sizeof(float2);  // itself
                    up = dn = pt0 - (int)sizeof(float2);
                } else {
                    const bool go_r = okr && (!okl || gr <= gl);
                    const int cb = go_r ? nr : nl;
                    nr += go_r ? 1 : 0;
                    nl -= go_r ? 0 : 1;
                    const int wd = cb * nw + (rank >> 5);
                    const int pos = below[wd] + __popc(tab[wd] & ((1u << (rank & 31)) - 1u));
                    up = pt0 + (cb * bs + pos) * (int)sizeof(float2);
                    dn = up - (int)sizeof(float2);
                    inblk = true;
                }
                my_evals -= (unsigned)sizeof(float2);
            }
            const unsigned dm = __ballot_sync(FULL, !has);
            if (dm != 0u && next < wslots) {
                const int q = next + __popc(dm & ((1u << lane) - 1u));
                next += __popc(dm);
                // slot q of the warp -> block, position; slots past a block's end are empty
                const int task = (q >> 5) * kGroupWarps + gw;
                const int b = ((task >> (lw - 3)) << 2) + ((q >> 3) & 3);
                const int p = ((task & ((W >> 3) - 1)) << 3) + (q & 7);
                if (!has && q < wslots && b < nb && (b << lw) + p < M) {
                    up = pt0 + (b * bs + p) * (int)sizeof(float2);
                    const float2 me = *reinterpret_cast<const float2*>(smem + up);
                    yi = me.x;
                    xi = me.y;
                    dn = up - (int)sizeof(float2);
                    up += (int)sizeof(float2);
                    has = true;
                    inblk = true;
                    nr = b + 1;
                    nl = b - 1;
                    slot_pos = (b << lw) + p;
                    rank = rank_s[slot_pos];
#pragma unroll
                    for (int c = 0; c < KK; ++c) best[c] = FLT_MAX;
                }
            }
        }
        steps += every;
        if (steps > step_bound) break;  // never expected: the pair's MI becomes NaN
        // `every` scan steps: one candidate above and one below in the lane's current
        // block (idle lanes, and lanes whose window has closed, re-read candidates at
        // least the threshold away and leave their lists unchanged)
        const unsigned long long P = pack_f2(make_float2(yi, xi));
        bool au = false, ad = false;
#pragma unroll kUnroll
        for (int rep = 0; rep < every; ++rep) {
            const float t = best[KK - 1];
            const float2 eu = sub_f32x2(P, *reinterpret_cast<const unsigned long long*>(smem + up));
            const float2 ed = sub_f32x2(P, *reinterpret_cast<const unsigned long long*>(smem + dn));
            au = fabsf(eu.x) < t;
            ad = fabsf(ed.x) < t;
            const float du = fmaxf(fabsf(eu.x), fabsf(eu.y));
            const float dd = fmaxf(fabsf(ed.x), fabsf(ed.y));
            insert2<KK>(best, fminf(du, dd), fmaxf(du, dd));
            up += au ? (int)sizeof(float2) : 0;
            dn -= ad ? (int)sizeof(float2) : 0;
        }
        inblk = au || ad;  // a closed side stays closed: the threshold only shrinks
    }
    return make_uint2(my_evals, steps > step_bound ? 1u : 0u);
}

// RPL: ranks per lane of the widest block (W <= 32 RPL)
template <int K1, int RPL>
__global__ void __launch_bounds__(32 * kGroupWarps * kLaneMaxGroups, 1)
    ksg_lane_kernel(KsgArgs A, unsigned long long* work, int lw, bool x_shared, int switch_min, int every) {
    constexpr int KK = K1 - 1;
    constexpr int GT = 32 * kGroupWarps;
    constexpr unsigned FULL = 0xffffffffu;
    pdl_wait();  // the staged references and the work counter
    extern __shared__ __align__(16) unsigned char smem[];
    const int M = A.M, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int group = warp / kGroupWarps, gw = warp % kGroupWarps, gt = threadIdx.x % GT;
    const int W = 1 << lw, nb = (M + W - 1) >> lw, nw = (M + 31) >> 5, bs = W + 1;
    const LaneSmem L(M, lw);
    unsigned char* gbase = smem + group * L.total;
    LaneCtl* ctl = reinterpret_cast<LaneCtl*>(gbase);
    float2* blk = reinterpret_cast<float2*>(gbase + L.blk);  // (y, x), separated blocks
    float* ys = reinterpret_cast<float*>(gbase + L.ys);      // query, sorted
    float* eps_s = reinterpret_cast<float*>(gbase + L.eps);  // y, rank, eps (see above)
    int* rank_s = reinterpret_cast<int*>(eps_s);
    unsigned* tab = reinterpret_cast<unsigned*>(gbase + L.tab);  // rank bits [nb][nw]
    unsigned char* below = gbase + L.below;  // a block's members below the word
    float2* bx = reinterpret_cast<float2*>(gbase + L.bx) + 1;  // (first, last) x per block
    const int64_t N = A.N, nv = A.v_end - A.v_begin;
    const unsigned long long items =
        A.paired ? (unsigned long long)nv : (unsigned long long)A.R * (unsigned long long)nv;
    const int top = pow2_floor(M);
    unsigned long long evals_total = 0;
    float* xsh = reinterpret_cast<float*>(smem + (blockDim.x / GT) * L.total);
    if (x_shared) {
        for (int i = threadIdx.x; i < M; i += blockDim.x) xsh[i] = A.xs_all[i];
        __syncthreads();
    }
    if (gt == 0) {  // no block beyond either end: an infinite x-gap
        bx[-1] = make_float2(0.0f, -INFINITY);
        bx[nb] = make_float2(INFINITY, 0.0f);
    }

    for (;;) {
        group_sync(group);  // the previous pair is finished by both warps
        if (gt == 0) ctl->item = atomicAdd(work, 1ull);
        group_sync(group);
        const unsigned long long item = ctl->item;
        if (item >= items) break;
        const int r = A.paired ? (int)item : (int)(item / (unsigned long long)nv);
        const int64_t v = A.v_begin + (int64_t)(A.paired ? item : item - (unsigned long long)r * nv);
        const float* xsg = A.xs_all + (int64_t)r * M;  // reference values, x-sorted (global)
        const int* perm = A.perm_all + (int64_t)r * M;
        const bool dbg = A.dbg_eps && r == 0 && v == A.v_begin;
        // ---- the query column in x-order and in sorted order; each thread has eight of its
        // strided loads of both in flight before their stores, so the column costs two memory
        // round trips, not M / 64
        int* cnt = reinterpret_cast<int*>(blk);  // tie counters (until the blocks are laid out)
        for (int s0 = 0; s0 < M; s0 += 8 * GT) {
            float c8[8], s8[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int s = s0 + j * GT + gt;
                c8[j] = s < M ? A.field[(int64_t)perm[s] * N + v] : 0.0f;
                s8[j] = s < M ? A.sorted[(int64_t)s * N + v] : 0.0f;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int s = s0 + j * GT + gt;
                if (s < M) {
                    eps_s[s] = c8[j];
                    ys[s] = s8[j];
                    cnt[s] = 0;
                }
            }
        }
        for (int i = gt; i < nb * nw; i += GT) tab[i] = 0u;
        for (int b = gt; b < nb; b += GT) bx[b] = make_float2(xsg[b << lw], xsg[min((b << lw) + W, M) - 1]);
        group_sync(group);  // the sorted column is complete
        // a constant query column: every distance is |dx|, so the blocks keep x-order and hold
        // (x, y) in the place of (y, x); the scan's window is then the x-gap
        const bool constant = ys[0] == ys[M - 1] && A.variant == 1;
        // ---- the members' ranks, four searches of a thread interleaved
        for (int s0 = gt; s0 < M; s0 += 4 * GT) {
            float y[4];
            int p[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) y[j] = eps_s[min(s0 + j * GT, M - 1)];
            if (!constant) lower_bounds<4>(ys, M, top, y, p);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int s = s0 + j * GT;
                if (s >= M) continue;
                int rank = constant ? s : min(p[j], M - 1);
                if (!constant && rank + 1 < M && ys[rank + 1] == y[j])
                    rank = min(rank + atomicAdd(cnt + rank, 1), M - 1);
                rank_s[s] = rank;
                atomicOr(&tab[(s >> lw) * nw + (rank >> 5)], 1u << (rank & 31));
            }
        }
        group_sync(group);
        // ---- blocks of W x-ranks (the last one shorter) in the order of the ranks
        for (int b = gt; b <= nb; b += GT) blk[b < nb ? b * bs : M + nb] = make_float2(INFINITY, INFINITY);
        for (int b = gw; b < nb; b += kGroupWarps) {
            const unsigned* tb = tab + b * nw;
            unsigned char* bb = below + b * nw;
            int carry = 0;
            for (int w0 = 0; w0 < nw; w0 += 32) {
                const int w = w0 + lane;
                const int c = w < nw ? __popc(tb[w]) : 0;
                int inc = c;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int u = __shfl_up_sync(FULL, inc, o);
                    inc += lane >= o ? u : 0;
                }
                // 256 ranks below a word count as 255: its word is empty then, and a scan that enters
                // there starts one rank lower and sees the same members
                if (w < nw) bb[w] = (unsigned char)(RPL > 4 ? min(carry + inc - c, 255) : carry + inc - c);
                carry += __shfl_sync(FULL, inc, 31);
            }
            int rk[RPL];
#pragma unroll
            for (int j = 0; j < RPL; ++j) {
                const int s = (b << lw) + j * 32 + lane;
                rk[j] = j * 32 < W && s < M ? rank_s[s] : -1;
            }
            __syncwarp();  // the counts are written, the ranks read (their places are reused)
#pragma unroll
            for (int j = 0; j < RPL; ++j) {
                if (rk[j] < 0) continue;
                const int s = (b << lw) + j * 32 + lane;
                const int pos = bb[rk[j] >> 5] + __popc(tb[rk[j] >> 5] & ((1u << (rk[j] & 31)) - 1u));
                const float y = ys[rk[j]], x = xsg[s];
                blk[1 + b * bs + pos] = constant ? make_float2(x, y) : make_float2(y, x);
                rank_s[(b << lw) + pos] = rk[j];
                if (dbg) A.dbg_ny[(b << lw) + pos] = s;  // x-rank by position (scratch)
            }
        }
        group_sync(group);

        // ---- joint k-NN distance of every member, lanes refilled from their warp's members
        const uint2 found = lane_search<KK>(group * L.total, M, lw, gw, constant, switch_min, every);
        const unsigned my_evals = found.x;
        const bool aborted = found.y != 0u;
        group_sync(group);

        // ---- marginal counts and the digamma sum, evenly split over the group
        long long acc = 0;  // fixed point
        for (int pos = gt; pos < M; pos += GT) {
            const int b = pos >> lw;
            const float e = eps_s[pos];
            float2 me = blk[1 + b + pos];
            if (constant) me = make_float2(me.y, me.x);
            int cx, cy;
            if (A.variant == 2) {  // non-strict counts within the k-NN set's marginal extents
                float ex, ey;
                const float yq[1] = {me.x};
                int rank[1];  // the query column's members below
                lower_bounds<1>(ys, M, top, yq, rank);
                const int w = min(rank[0], M - 1) >> 5;
                const unsigned under = (1u << (rank[0] & 31)) - 1u;
                block_extents(blk, bx, nb, bs, b, pos - (b << lw), me.y, me.x, e, ex, ey,
                              [&](int bb) { return below[bb * nw + w] + __popc(tab[bb * nw + w] & under); });
                count_le_pair(xsg, ys, M, top, me.y, ex, me.x, ey, cx, cy);
                --cx;  // the member itself excluded
                --cy;
                acc += A.psi_fix[cx] + A.psi_fix[cy];
                if (dbg) {
                    const int mi = perm[A.dbg_ny[pos]];
                    A.dbg_eps[mi] = ex;
                    if (A.dbg_ey) A.dbg_ey[mi] = ey;
                }
            } else {
                const int self = e > 0.0f ? 1 : 0;
                if (x_shared) count_within_pair(xsh, ys, M, top, me.y, me.x, e, cx, cy);
                else count_within_pair(xsg, ys, M, top, me.y, me.x, e, cx, cy);
                cx -= self;
                cy -= self;
                acc += A.psi_fix[cx + 1] + A.psi_fix[cy + 1];
                if (dbg) {
                    const int mi = perm[A.dbg_ny[pos]];
                    A.dbg_eps[mi] = e;
                    if (A.dbg_ey) A.dbg_ey[mi] = e;
                }
            }
            if (dbg) A.dbg_nx[pos] = cx | (cy << 16);  // counts by block position (scratch)
        }
        if (dbg) {
            // the counts in member order: every thread first moves its positions' scratch (x-rank,
            // counts) to shared memory that is no longer read, then all write the results over it
            group_sync(group);
            for (int pos = gt; pos < M; pos += GT)
                blk[1 + pos] = make_float2(__int_as_float(A.dbg_ny[pos]), __int_as_float(A.dbg_nx[pos]));
            group_sync(group);
            for (int pos = gt; pos < M; pos += GT) {
                const float2 c = blk[1 + pos];
                const int mi = perm[__float_as_int(c.x)], n = __float_as_int(c.y);
                A.dbg_nx[mi] = n & 0xffff;
                A.dbg_ny[mi] = n >> 16;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(FULL, acc, o);
        evals_total += __reduce_add_sync(FULL, my_evals / (unsigned)sizeof(float2));
        if (lane == 0) ctl->part[gw] = aborted ? LLONG_MIN : acc;
        group_sync(group);
        if (gt == 0) {
            long long sum = 0;
            bool gave_up = false;
#pragma unroll
            for (int w = 0; w < kGroupWarps; ++w) {
                sum += ctl->part[w];
                gave_up = gave_up || ctl->part[w] == LLONG_MIN;
            }
            const double tot = (double)sum * A.psi_scale;
            double mi = A.psi[A.k] - (A.variant == 2 ? 1.0 / A.k : 0.0) + A.psi[M] - tot / (double)M;
            if (gave_up) mi = __longlong_as_double(0x7ff8000000000000ll);
            A.out[A.paired ? (v - A.v_begin) : (int64_t)r * A.out_stride + (v - A.v_begin)] = (float)mi;
            if (dbg && A.dbg_mi) *A.dbg_mi = mi;
        }
    }
    if (A.evals && lane == 0) atomicAdd(A.evals, evals_total);
}

template <class Kern>
static cudaError_t launch_persistent(ndf_ctx* ctx, Kern kern, const KsgArgs& A, int threads,
                                    size_t smem, int64_t items) {
    cudaError_t e = allow_dynamic_smem(kern);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    int64_t grid = (int64_t)ctx->sm_count * per_sm;
    if (grid > items) grid = items;
    kern<<<(unsigned)grid, threads, smem, ctx->stream>>>(A);
    ctx->launches++;
    return cudaGetLastError();
}

// How the lane search runs a call: 2^lw ranks per block, gpc groups per CTA, the reference in shared
// memory or not (algorithm 1 alone reads it there).  The usual form is lane_block_log2's width with
// the shared reference, and 13 groups from 257 members on (14 against 13 groups, us for 1.2e7 / M
// vertices, k = 4: 1126 / 1159 for M = 60, 645 / 645 for M = 256, 733 / 703 for M = 600).  Another form may
// place another group per SM: the 14th, the reference left in global memory, blocks of 256 ranks, which halve
// the bitmaps.  It is taken where that saves a round of pairs: above 1700 members always (k = 8, 128
// against 256 ranks: 1509 / 1393 for M = 1800, 2268 / 1829 for M = 3000; M = 4096, without the reference,
// 4372 / 3292; where no group is gained 128 is the better one, M = 3500, k = 4: 2107 / 2146, algorithm 2: 3858
// / 4000), below where it saves at least a fifth of the rounds (2100 vertices, M = 500, k = 8: 136 in two
// rounds, 100 in one; 1600 vertices, M = 1200: 347 and 249).
struct LanePlan {
    int lw, gpc;
    bool x_shared;
};
static LanePlan lane_plan(int M, int64_t pairs, int sms, bool x_shared) {
    const int64_t need = (pairs + sms - 1) / sms;  // groups per SM that take all pairs at once
    auto groups = [&](int lw, bool xs, int most) {
        const int64_t g = (int64_t)((kMaxDynamicSmem - (xs ? sizeof(float) * (size_t)M : 0)) / LaneSmem(M, lw).total);
        return (int)std::min(std::min<int64_t>(g, most), need);
    };
    auto rounds = [&](int gpc) { return gpc > 0 ? (need + gpc - 1) / gpc : need + 1; };
    LanePlan best = {lane_block_log2(M), 0, x_shared};
    best.gpc = groups(best.lw, best.x_shared, M > 256 ? kLaneMaxGroups - 1 : kLaneMaxGroups);
    const LanePlan other[4] = {{best.lw, 0, x_shared}, {best.lw, 0, false}, {8, 0, x_shared}, {8, 0, false}};
    for (LanePlan o : other) {
        o.gpc = groups(o.lw, o.x_shared, kLaneMaxGroups);
        if ((M > 1700 ? 4 : 5) * rounds(o.gpc) < 4 * rounds(best.gpc)) best = o;
    }
    return best;
}

template <int K1>
static cudaError_t launch_ksg_k(ndf_ctx* ctx, KsgArgs A, bool prune) {
    const int M = A.M;
    if (prune && ctx->ksg_algorithm == NDF_KSG_LANES && (A.variant == 1 || A.variant == 2)) {
        // two-warp groups per pair
        const int64_t pairs = A.paired ? (A.v_end - A.v_begin) : (int64_t)A.R * (A.v_end - A.v_begin);
        const LanePlan p = lane_plan(M, pairs, ctx->sm_count, A.R == 1 && A.variant == 1);
        if (p.gpc >= 1) {
            const size_t smem = (size_t)p.gpc * LaneSmem(M, p.lw).total + (p.x_shared ? sizeof(float) * (size_t)M : 0);
            const int threads = 32 * kGroupWarps * p.gpc;
            auto kern = p.lw > 7 ? ksg_lane_kernel<K1, 8> : ksg_lane_kernel<K1, 4>;
            cudaError_t e = allow_dynamic_smem(kern);
            if (e != cudaSuccess) return e;
            int64_t grid = (int64_t)ctx->sm_count;
            if (grid * p.gpc > pairs) grid = (pairs + p.gpc - 1) / p.gpc;
            e = launch_after(kern, dim3((unsigned)grid), dim3((unsigned)threads), smem, ctx->stream, A,
                             ctx->ksg_work.as<unsigned long long>(), p.lw, p.x_shared, ctx->ksg_switch_min, ctx->ksg_every);
            ctx->launches++;
            return e;
        }
    }
    if (prune && ctx->ksg_algorithm == NDF_KSG_BLOCK && A.variant == 1) {
        // two-warp groups per pair; as many groups per CTA as fit in shared memory
        const size_t per_group = block_group_bytes(M);
        int gpc = (int)(kMaxDynamicSmem / per_group);
        if (gpc > kMaxGroupsPerCta) gpc = kMaxGroupsPerCta;
        if (gpc >= 1) {
            const size_t smem = (size_t)gpc * per_group;
            const int threads = 32 * kGroupWarps * gpc;
            auto kern = ksg_block_kernel<K1>;
            cudaError_t e = allow_dynamic_smem(kern);
            if (e != cudaSuccess) return e;
            const int64_t pairs = A.paired ? (A.v_end - A.v_begin) : (int64_t)A.R * (A.v_end - A.v_begin);
            int64_t grid = (int64_t)ctx->sm_count;
            if (grid * gpc > pairs) grid = (pairs + gpc - 1) / gpc;
            kern<<<(unsigned)grid, threads, smem, ctx->stream>>>(A, ctx->ksg_work.as<unsigned long long>());
            ctx->launches++;
            return cudaGetLastError();
        }
    }
    if (prune) {
        // one warp group per pair; as many groups per CTA as fit in shared memory
        const size_t per_group = (size_t)kGroupSmemPerM * M + kGroupSmemFixed;
        int gpc = (int)(kMaxDynamicSmem / per_group);
        if (gpc > kMaxGroupsPerCta) gpc = kMaxGroupsPerCta;
        if (gpc < 1) gpc = 1;
        const size_t smem = (size_t)gpc * per_group;
        const int threads = 32 * kGroupWarps * gpc;
        auto kern = ksg_pruned_kernel<K1>;
        cudaError_t e = allow_dynamic_smem(kern);
        if (e != cudaSuccess) return e;
        int per_sm = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
        if (e != cudaSuccess) return e;
        if (per_sm < 1) per_sm = 1;
        const int64_t pairs = A.paired ? (A.v_end - A.v_begin) : (int64_t)A.R * (A.v_end - A.v_begin);
        int64_t grid = (int64_t)ctx->sm_count * per_sm;
        if (grid * gpc > pairs) grid = (pairs + gpc - 1) / gpc;
        kern<<<(unsigned)grid, threads, smem, ctx->stream>>>(
            A, ctx->ksg_work.as<unsigned long long>());
        ctx->launches++;
        return cudaGetLastError();
    }
    // two CTAs per SM: at most ~112 KB of shared memory each
    const size_t budget = 112 * 1024;
    while (A.G > 1 && KsgSmem(M, A.VT, A.G).total > budget) A.G >>= 1;
    while (A.VT > 1 && KsgSmem(M, A.VT, A.G).total > budget) A.VT >>= 1;
    const size_t smem = KsgSmem(M, A.VT, A.G).total;
    const int64_t items =
        (int64_t)((A.R + A.G - 1) / A.G) * ((A.v_end - A.v_begin + A.VT - 1) / A.VT);
    int threads = ((M + kKsgPts - 1) / kKsgPts + 31) / 32 * 32;
    if (threads > kKsgMaxThreads) threads = kKsgMaxThreads;
    return launch_persistent(ctx, ksg_volume_kernel<K1>, A, threads, smem, items);
}

cudaError_t launch_ksg(ndf_ctx* ctx, const Field& rf, const Field& qf, const int64_t* d_refs,
                       int64_t ref0, int R, int k, int64_t v_begin, int64_t v_end, float* out,
                       int64_t out_stride, bool prune, int G, int VT, double* dbg_mi,
                       float* dbg_eps, int32_t* dbg_nx, int32_t* dbg_ny,
                       unsigned long long* evals, int variant, float* dbg_ey, bool paired) {
    const int M = (int)rf.M;
    if (!qf.sorted || R < 1 || v_end <= v_begin) return cudaErrorInvalidValue;
    if (paired) {
        if (R != v_end - v_begin) return cudaErrorInvalidValue;
        prune = true;  // the pair list runs on the pruned kernel's work counter
    }
    cudaError_t e = ctx->stage_x.reserve(sizeof(float) * (size_t)M * (size_t)R);
    if (e == cudaSuccess) e = ctx->stage_perm.reserve(sizeof(int) * (size_t)M * (size_t)R);
    if (e != cudaSuccess) return e;
    e = ctx->ksg_work.reserve(sizeof(unsigned long long));
    if (e != cudaSuccess) return e;
    // a warp per reference where there are many of them, or few members (a lone warp's network of
    // 1024 keys is a serial chain of 14,000 instructions; one CTA spreads it)
    auto stage_warps = [&](auto kern) {
        const int warps = R < 4 ? R : 4;
        kern<<<(unsigned)((R + warps - 1) / warps), 32 * warps, 0, ctx->stream>>>(
            rf.data, M, rf.N, d_refs, ref0, R, ctx->stage_x.as<float>(), ctx->stage_perm.as<int>(),
            ctx->flag.as<unsigned>() + 1, ctx->ksg_work.as<unsigned long long>());
    };
    if (M <= 128) stage_warps(ksg_stage_warp_kernel<4>);
    else if (M <= 256) stage_warps(ksg_stage_warp_kernel<8>);
    else if (M <= 512 && R >= 32) stage_warps(ksg_stage_warp_kernel<16>);
    else if (M <= 1024 && R >= 32) stage_warps(ksg_stage_warp_kernel<32>);
    else
        ksg_stage_kernel<<<R, 1024, 0, ctx->stream>>>(rf.data, M, rf.N, d_refs, ref0, ctx->stage_x.as<float>(),
                                                       ctx->stage_perm.as<int>(), ctx->flag.as<unsigned>() + 1,
                                                       ctx->ksg_work.as<unsigned long long>());
    ctx->launches++;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    KsgArgs A;
    A.field = qf.data;
    A.sorted = qf.sorted;
    A.M = M;
    A.k = k;
    A.G = G < 1 ? 1 : G > R ? R : G;
    A.VT = VT < 1 ? 1 : VT;
    A.R = R;
    A.N = qf.N;
    A.v_begin = v_begin;
    A.v_end = v_end;
    A.xs_all = ctx->stage_x.as<float>();
    A.perm_all = ctx->stage_perm.as<int>();
    A.psi = ctx->psi.as<double>();
    const int group = psi_fix_group(M);
    A.psi_fix = reinterpret_cast<const long long*>(A.psi + ctx->psi_n) + psi_fix_offset(group);
    A.psi_scale = 1.0 / (double)(1ll << psi_fix_bits(group));
    A.out = out;
    A.out_stride = out_stride;
    A.dbg_mi = dbg_mi;
    A.dbg_eps = dbg_eps;
    A.dbg_nx = dbg_nx;
    A.dbg_ny = dbg_ny;
    A.dbg_ey = dbg_ey;
    A.variant = variant;
    A.paired = paired ? 1 : 0;
    A.evals = evals;
    switch (k + 1) {
        case 2: return launch_ksg_k<2>(ctx, A, prune);
        case 3: return launch_ksg_k<3>(ctx, A, prune);
        case 4: return launch_ksg_k<4>(ctx, A, prune);
        case 5: return launch_ksg_k<5>(ctx, A, prune);
        case 6: return launch_ksg_k<6>(ctx, A, prune);
        case 7: return launch_ksg_k<7>(ctx, A, prune);
        case 8: return launch_ksg_k<8>(ctx, A, prune);
        case 9: return launch_ksg_k<9>(ctx, A, prune);
        case 10: return launch_ksg_k<10>(ctx, A, prune);
        case 11: return launch_ksg_k<11>(ctx, A, prune);
        case 12: return launch_ksg_k<12>(ctx, A, prune);
        case 13: return launch_ksg_k<13>(ctx, A, prune);
        case 14: return launch_ksg_k<14>(ctx, A, prune);
        case 15: return launch_ksg_k<15>(ctx, A, prune);
        case 16: return launch_ksg_k<16>(ctx, A, prune);
        case 17: return launch_ksg_k<17>(ctx, A, prune);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace ndf

using namespace ndf;

// Picks the exact search for algorithm 1 and the lane schedule: times the block
// search and the lane-refill search under several (switch_min, every) schedules on
// a sample (8 references spread over the reference field, 24,576 consecutive query
// vertices from the middle of the grid, one warm-up launch each) and keeps the
// fastest in the context.  Results do not depend on the choice.
extern "C" ndf_status ndf_ksg_autotune_search(ndf_ctx* ctx, int ref_field, int query_field, int k,
                                              int* algorithm, int* switch_min, int* every) {
    if (!ctx) return NDF_ERR_ARG;
    const Field *rf, *qf;
    ndf_status st = check_pair(ctx, ref_field, query_field, 0, &rf, &qf);
    if (st != NDF_OK) return st;
    if (k < 1 || k >= rf->M || k > kKsgMaxK || rf->M > kKsgMaxM)
        return fail(ctx, NDF_ERR_ARG, "bad k or M");
    cudaSetDevice(ctx->device);
    if ((st = ensure_psi_table(ctx, rf->M + 1)) != NDF_OK) return st;
    cudaError_t es = ensure_sorted_columns(ctx, ctx->fields[query_field]);
    if (es != cudaSuccess) return cuda_fail(ctx, es, "sorted columns");
    const int R = 8;
    const int64_t nv = qf->N < 24576 ? qf->N : 24576;
    const int64_t v0 = (qf->N - nv) / 2;
    int64_t refs[R];
    for (int i = 0; i < R; ++i) refs[i] = (int64_t)((double)(i + 0.5) / R * (double)(rf->N - 1));
    float* out = nullptr;
    int64_t* d_refs = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaError_t e = cudaMalloc(&out, sizeof(float) * (size_t)R * (size_t)nv);
    if (e == cudaSuccess) e = cudaMalloc(&d_refs, sizeof refs);
    if (e == cudaSuccess) e = cudaMemcpy(d_refs, refs, sizeof refs, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    const int cand[][3] = {{NDF_KSG_BLOCK, 0, 0},  {NDF_KSG_LANES, 8, 4},  {NDF_KSG_LANES, 12, 4},
                           {NDF_KSG_LANES, 16, 4}, {NDF_KSG_LANES, 12, 5}, {NDF_KSG_LANES, 16, 5},
                           {NDF_KSG_LANES, 12, 6}, {NDF_KSG_LANES, 16, 6}, {NDF_KSG_LANES, 20, 5}};
    const int keep_alg = ctx->ksg_algorithm, keep_sw = ctx->ksg_switch_min, keep_ev = ctx->ksg_every;
    const bool keep_count = ctx->count_evals;
    ctx->count_evals = false;
    float best = 3.4e38f;
    int ba = keep_alg, bs = keep_sw, be = keep_ev;
    for (const auto& c : cand) {
        if (e != cudaSuccess) break;
        ctx->ksg_algorithm = c[0];
        if (c[0] == NDF_KSG_LANES) {
            ctx->ksg_switch_min = c[1];
            ctx->ksg_every = c[2];
        }
        e = launch_ksg(ctx, *rf, *qf, d_refs, 0, R, k, v0, v0 + nv, out, nv, true, 1, 1, nullptr,
                       nullptr, nullptr, nullptr, nullptr);  // warm-up
        if (e == cudaSuccess) e = cudaEventRecord(e0, ctx->stream);
        if (e == cudaSuccess)
            e = launch_ksg(ctx, *rf, *qf, d_refs, 0, R, k, v0, v0 + nv, out, nv, true, 1, 1, nullptr,
                           nullptr, nullptr, nullptr, nullptr);
        if (e == cudaSuccess) e = cudaEventRecord(e1, ctx->stream);
        if (e == cudaSuccess) e = cudaEventSynchronize(e1);
        float ms = 0.0f;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
        if (e == cudaSuccess && ms < best) {
            best = ms;
            ba = c[0];
            bs = c[0] == NDF_KSG_LANES ? c[1] : keep_sw;
            be = c[0] == NDF_KSG_LANES ? c[2] : keep_ev;
        }
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (out) cudaFree(out);
    if (d_refs) cudaFree(d_refs);
    ctx->count_evals = keep_count;
    if (e != cudaSuccess) {
        ctx->ksg_algorithm = keep_alg;
        ctx->ksg_switch_min = keep_sw;
        ctx->ksg_every = keep_ev;
        return cuda_fail(ctx, e, "ksg search autotune");
    }
    ctx->ksg_algorithm = ba;
    ctx->ksg_switch_min = bs;
    ctx->ksg_every = be;
    if (algorithm) *algorithm = ba;
    if (switch_min) *switch_min = bs;
    if (every) *every = be;
    return NDF_OK;
}

extern "C" ndf_status ndf_ksg_autotune(ndf_ctx* ctx, int ref_field, int query_field, int k,
                                       int* best_group, int* best_tile) {
    if (!ctx) return NDF_ERR_ARG;
    const Field *rf, *qf;
    ndf_status st = check_pair(ctx, ref_field, query_field, 0, &rf, &qf);
    if (st != NDF_OK) return st;
    if (k < 1 || k >= rf->M || k > kKsgMaxK || rf->M > kKsgMaxM)
        return fail(ctx, NDF_ERR_ARG, "bad k or M");
    cudaSetDevice(ctx->device);
    if ((st = ensure_psi_table(ctx, rf->M + 1)) != NDF_OK) return st;
    cudaError_t es = ensure_sorted_columns(ctx, ctx->fields[query_field]);
    if (es != cudaSuccess) return cuda_fail(ctx, es, "sorted columns");
    // sample: 8 references spread over the grid, the first 16384 query vertices
    const int R = 8;
    const int64_t nv = qf->N < 16384 ? qf->N : 16384;
    int64_t refs[R];
    for (int i = 0; i < R; ++i) refs[i] = (int64_t)((double)(i + 0.5) / R * (double)(rf->N - 1));
    float* out = nullptr;
    int64_t* d_refs = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaError_t e = cudaMalloc(&out, sizeof(float) * (size_t)R * (size_t)nv);
    if (e == cudaSuccess) e = cudaMalloc(&d_refs, sizeof refs);
    if (e == cudaSuccess) e = cudaMemcpy(d_refs, refs, sizeof refs, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    const int cand[][2] = {{1, 4}, {1, 8}, {2, 4}, {2, 8}, {4, 4}, {4, 8}};
    const bool prune = false;  // the shapes belong to the brute-force kernel
    float best = 3.4e38f;
    int bg = ctx->ksg_group, bt = ctx->ksg_tile;
    for (const auto& c : cand) {
        if (e != cudaSuccess) break;
        // warm-up, then timed
        e = launch_ksg(ctx, *rf, *qf, d_refs, 0, R, k, 0, nv, out, nv, prune, c[0], c[1], nullptr,
                       nullptr, nullptr, nullptr, nullptr);
        if (e == cudaSuccess) e = cudaEventRecord(e0, ctx->stream);
        if (e == cudaSuccess)
            e = launch_ksg(ctx, *rf, *qf, d_refs, 0, R, k, 0, nv, out, nv, prune, c[0], c[1],
                           nullptr, nullptr, nullptr, nullptr, nullptr);
        if (e == cudaSuccess) e = cudaEventRecord(e1, ctx->stream);
        if (e == cudaSuccess) e = cudaEventSynchronize(e1);
        float ms = 0.0f;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
        if (e == cudaSuccess && ms < best) {
            best = ms;
            bg = c[0];
            bt = c[1];
        }
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (out) cudaFree(out);
    if (d_refs) cudaFree(d_refs);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "ksg autotune");
    ctx->ksg_group = bg;
    ctx->ksg_tile = bt;
    if (best_group) *best_group = bg;
    if (best_tile) *best_tile = bt;
    return NDF_OK;
}
