// The hash-grid network's dense layers in FP32 (Sec. 4.1-4.3, row f2): forward, data
// gradient and weight gradient, FP32 products and sums (the parity path of the network; the
// FP64 oracle checks it), deterministic: the weight gradients add fixed chunks of the batch in
// a fixed order.
//
// What bounds it: the FP32 pipe (a layer of 128 x 128 over 16,384 rows is 8.6 us of it on 152
// SMs), the last wave of tiles and, at these sizes, the number of launches.  So
//   - one launch per layer and direction: bias and activation are the forward's epilogue, the
//     activation's derivative the data gradient's, the bias gradient falls out of the weight
//     gradient's operand, and the weight and data gradients of a layer share a launch (their
//     tiles are independent; the longer weight tiles come first);
//   - a CTA of 128 threads computes a 64 x 128 tile in 16-deep slices (two CTAs per SM).  A
//     thread owns 8 rows x 8 columns, two columns per packed fma.rn.f32x2: a step of k is 32
//     FMA instructions (64 cycles of the pipe), four 16-byte shared loads and eight moves that
//     double an A value, so neither the issue slots nor the shared memory keep the pipe waiting
//     (4 x 8 values per thread from 256 threads needed as many loads for half the products:
//     25 us per forward layer of 16,384 rows).  The next slice is read into registers while the
//     present one is multiplied, and the slices alternate between two buffers (one barrier per
//     slice);
//   - each 16-deep slice is summed on its own and then added to the running sums (blocked
//     summation: rounding grows with 16 + K / 16 terms instead of K).
#include "gemm_f32.h"

#include "device_common.cuh"
#include "hash_common.cuh"

namespace ndf {

namespace {

constexpr int kBM = 64, kBN = 128, kBK = 16, kThreads = 128;
constexpr int kAStride = kBM + 4, kBStride = kBN + 4;  // floats per k

union Tile {
    struct {
        float a[2][kBK][kAStride];
        float b[2][kBK][kBStride];
    };
    float out[kBM][kBStride];  // the results, for a row-wise epilogue
};

typedef unsigned long long u64;
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
    u64 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ u64 twice(float a) {
    u64 d;
    asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(a));
    return d;
}

// four consecutive values p[0..3], the first n of them inside the matrix (vec: p is 16-byte
// aligned whenever n >= 4)
__device__ __forceinline__ float4 load4(const float* p, int n, bool vec) {
    if (n >= 4 && vec) return *reinterpret_cast<const float4*>(p);
    float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (n > 0) v.x = p[0];
    if (n > 1) v.y = p[1];
    if (n > 2) v.z = p[2];
    if (n > 3) v.w = p[3];
    return v;
}

// this thread's rows 4 ty + 32 h + i and columns 4 tx + 64 h + j (h < 2; i, j < 4) of the tile
__device__ __forceinline__ int tile_ty() { return ((threadIdx.x >> 5) & 1) * 4 + ((threadIdx.x & 31) >> 3); }
__device__ __forceinline__ int tile_tx() { return (threadIdx.x >> 6) * 8 + (threadIdx.x & 7); }

// acc[4 h + i][2 g + q] = the sums of row m0 + 4 ty + 32 h + i and the column pair
// n0 + 4 tx + 64 g + 2 q of A B over k in [k0, k1).  TA: A is [K][M] (else [M][K]); TB: B is
// [N][K] (else [K][N]).  With TA csum = this thread's sums of A over its rows k (every 8th),
// columns m0 + 4 (tid & 15) + 0 .. 3.
template <bool TA, bool TB>
__device__ __forceinline__ void tile_product(Tile& S, const float* A, const float* B,
                                             int64_t M, int64_t N, int64_t m0, int64_t n0, int64_t k0,
                                             int64_t k1, int64_t lda, int64_t ldb, bool avec, bool bvec,
                                             u64 (&acc)[8][4], float4& csum) {
    const int t = threadIdx.x, ty = tile_ty(), tx = tile_tx();
    float4 ra[2], rb[4];
    auto load = [&](int64_t k) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (TA) {  // 16 k x 64 m, threads along m
                const int64_t kk = k + (t >> 4) + 8 * h, m = m0 + (t & 15) * 4;
                ra[h] = load4(A + kk * lda + m, kk < k1 ? (int)min(M - m, (int64_t)4) : 0, avec);
            } else {  // 64 m x 16 k, threads along k
                const int64_t m = m0 + (t >> 2) + 32 * h, kk = k + (t & 3) * 4;
                ra[h] = load4(A + m * lda + kk, m < M ? (int)min(k1 - kk, (int64_t)4) : 0, avec);
            }
        }
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            if (TB) {  // 128 n x 16 k, threads along k
                const int64_t n = n0 + (t >> 2) + 32 * h, kk = k + (t & 3) * 4;
                rb[h] = load4(B + n * ldb + kk, n < N ? (int)min(k1 - kk, (int64_t)4) : 0, bvec);
            } else {  // 16 k x 128 n, threads along n
                const int64_t kk = k + (t >> 5) + 4 * h, n = n0 + (t & 31) * 4;
                rb[h] = load4(B + kk * ldb + n, kk < k1 ? (int)min(N - n, (int64_t)4) : 0, bvec);
            }
        }
    };
    auto store = [&](int buf) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (TA) {
                *reinterpret_cast<float4*>(&S.a[buf][(t >> 4) + 8 * h][(t & 15) * 4]) = ra[h];
                csum.x += ra[h].x;
                csum.y += ra[h].y;
                csum.z += ra[h].z;
                csum.w += ra[h].w;
            } else {
                const int m = (t >> 2) + 32 * h, k = (t & 3) * 4;
                S.a[buf][k][m] = ra[h].x;
                S.a[buf][k + 1][m] = ra[h].y;
                S.a[buf][k + 2][m] = ra[h].z;
                S.a[buf][k + 3][m] = ra[h].w;
            }
        }
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            if (TB) {
                const int n = (t >> 2) + 32 * h, k = (t & 3) * 4;
                S.b[buf][k][n] = rb[h].x;
                S.b[buf][k + 1][n] = rb[h].y;
                S.b[buf][k + 2][n] = rb[h].z;
                S.b[buf][k + 3][n] = rb[h].w;
            } else {
                *reinterpret_cast<float4*>(&S.b[buf][(t >> 5) + 4 * h][(t & 31) * 4]) = rb[h];
            }
        }
    };
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
    csum = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (k0 < k1) load(k0);
    int buf = 0;
    for (int64_t k = k0; k < k1; k += kBK, buf ^= 1) {
        store(buf);
        __syncthreads();  // also: every thread is done with this buffer's slice before last
        if (k + kBK < k1) load(k + kBK);
        u64 part[8][4] = {};
#pragma unroll
        for (int kk = 0; kk < kBK; ++kk) {
            const float4 a0 = *reinterpret_cast<const float4*>(&S.a[buf][kk][ty * 4]);
            const float4 a1 = *reinterpret_cast<const float4*>(&S.a[buf][kk][ty * 4 + 32]);
            const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(&S.b[buf][kk][tx * 4]);
            const ulonglong2 b1 = *reinterpret_cast<const ulonglong2*>(&S.b[buf][kk][tx * 4 + 64]);
            const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const u64 b[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const u64 aa = twice(a[i]);
#pragma unroll
                for (int j = 0; j < 4; ++j) part[i][j] = fma2(aa, b[j], part[i][j]);
            }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = add2(acc[i][j], part[i][j]);
    }
}

// the 8 x 8 results of this thread, four consecutive columns at a time: f(row, column, v)
template <class F>
__device__ __forceinline__ void for_results(const u64 (&acc)[8][4], int64_t m0, int64_t n0, F&& f) {
    const int64_t m = m0 + tile_ty() * 4, n = n0 + tile_tx() * 4;
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            const u64 p = acc[i][2 * g], q = acc[i][2 * g + 1];
            float v[4] = {__uint_as_float((unsigned)p), __uint_as_float((unsigned)(p >> 32)),
                          __uint_as_float((unsigned)q), __uint_as_float((unsigned)(q >> 32))};
            f(m + (i & 3) + 32 * (i >> 2), n + 64 * g, v);
        }
}

// The tile's results row by row: f(row, column, v, e) for four consecutive columns, a warp covering
// one row's 128 columns; e = fetch(row, column), read two iterations of the loop ahead of its use
// (its latency cost 6 us of a 28 us backward layer).  Two copies of f in a loop: with f inlined
// once per result of a thread the sine of the activations filled the instruction cache (26 us of
// a 43 us forward layer).
template <class Fetch, class F>
__device__ __forceinline__ void for_rows(Tile& S, const u64 (&acc)[8][4], int64_t m0, int64_t n0, Fetch&& fetch,
                                         F&& f) {
    const int n = (threadIdx.x & 31) * 4;
    int m = threadIdx.x >> 5;
    float4 e[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) e[r] = fetch(m0 + m + 4 * r, n0 + n);
    __syncthreads();  // the operand slices are done with
    for_results(acc, 0, 0, [&](int64_t mm, int64_t nn, float(&v)[4]) {
        *reinterpret_cast<float4*>(&S.out[mm][nn]) = make_float4(v[0], v[1], v[2], v[3]);
    });
    __syncthreads();
#pragma unroll 1
    for (; m < kBM; m += 8) {
        float4 next[2], q[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            next[r] = fetch(m0 + m + 8 + 4 * r, n0 + n);
            q[r] = *reinterpret_cast<const float4*>(&S.out[m + 4 * r][n]);
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            float v[4] = {q[r].x, q[r].y, q[r].z, q[r].w};
            f(m0 + m + 4 * r, n0 + n, v, e[r]);
            e[r] = next[r];
        }
    }
}

// stores v[0..3] at p, the first n of them inside the matrix (vec as in load4)
__device__ __forceinline__ void store4(float* p, const float (&v)[4], int64_t n, bool vec) {
    if (n >= 4 && vec) {
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (j < n) p[j] = v[j];
    }
}

// grid: (row tiles x column tiles, 1, batch)
__global__ void __launch_bounds__(kThreads, 2)
    dense_forward_kernel(DenseLayer L, const float* X, float* pre,
                         float* post, int act, bool xvec, bool wvec, bool yvec) {
    __shared__ __align__(16) Tile S;
    pdl_launch();
    pdl_wait();
    const int nt = (L.cout + kBN - 1) / kBN, z = blockIdx.z;
    const int64_t m0 = (int64_t)(blockIdx.x / nt) * kBM, n0 = (int64_t)(blockIdx.x % nt) * kBN;
    const int64_t row0 = (int64_t)z * L.rows;
    const float* W = L.W + z * L.wstride;
    const float* bias = L.b + z * L.wstride;
    u64 acc[8][4];
    float4 cs;
    tile_product<false, true>(S, X + row0 * L.cin, W, L.rows, L.cout, m0, n0, 0, L.cin, L.cin, L.cin, xvec, wvec,
                              acc, cs);
    const int64_t nb = n0 + (threadIdx.x & 31) * 4;
    float bn[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) bn[j] = nb + j < L.cout ? bias[nb + j] : 0.0f;
    auto nothing = [](int64_t, int64_t) { return make_float4(0.0f, 0.0f, 0.0f, 0.0f); };
    for_rows(S, acc, m0, n0, nothing, [&](int64_t m, int64_t n, float(&v)[4], const float4&) {
        if (m >= L.rows || n >= L.cout) return;
        const int64_t left = L.cout - n, o = (row0 + m) * L.cout + n;
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] += bn[j];
        store4(pre + o, v, left, yvec);
        if (post) {
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = act_f(act, v[j]);
            store4(post + o, v, left, yvec);
        }
    });
}

struct BackwardArgs {
    const float *X, *dY, *pre_in;
    float *dX, *wpart, *bpart;
    int col0, act, splits;
    int64_t chunk;
    unsigned wblocks, dblocks;  // per weight set
    bool xvec, yvec, wvec, dxvec;
};

// grid: (weight-gradient tiles x splits, then data-gradient tiles; 1; batch)
__global__ void __launch_bounds__(kThreads, 2) dense_backward_kernel(DenseLayer L, BackwardArgs a) {
    __shared__ __align__(16) Tile S;
    pdl_launch();
    pdl_wait();
    const int z = blockIdx.z;
    const int64_t row0 = (int64_t)z * L.rows;
    const float* dY = a.dY + row0 * L.cout;
    u64 acc[8][4];
    float4 cs;
    if (blockIdx.x < a.wblocks) {  // dW partial of a chunk of rows: dY^T X
        const int mt = (L.cout + kBM - 1) / kBM, nt = (L.cin + kBN - 1) / kBN;
        const int split = blockIdx.x / (mt * nt), tile = blockIdx.x % (mt * nt);
        const int64_t m0 = (int64_t)(tile / nt) * kBM, n0 = (int64_t)(tile % nt) * kBN;
        const int64_t k0 = split * a.chunk, k1 = min(k0 + a.chunk, L.rows);
        tile_product<true, false>(S, dY, a.X + row0 * L.cin, L.cout, L.cin, m0, n0, k0, k1, L.cout, L.cin, a.yvec,
                                  a.xvec, acc, cs);
        float* wp = a.wpart + ((int64_t)z * a.splits + split) * L.cout * L.cin;
        for_results(acc, m0, n0, [&](int64_t m, int64_t n, float(&v)[4]) {
            if (m < L.cout && n < L.cin) store4(wp + m * L.cin + n, v, L.cin - n, (L.cin & 3) == 0);
        });
        if (n0 != 0) return;
        // the bias gradient: 8 threads' sums per column, added in order
        __syncthreads();
        float* red = &S.b[0][0][0];  // [8][kBM]
        const int t = threadIdx.x;
        *reinterpret_cast<float4*>(red + (t >> 4) * kBM + (t & 15) * 4) = cs;
        __syncthreads();
        if (t < kBM && m0 + t < L.cout) {
            float s = 0.0f;
#pragma unroll
            for (int k = 0; k < 8; ++k) s += red[k * kBM + t];
            a.bpart[((int64_t)z * a.splits + split) * L.cout + m0 + t] = s;
        }
        return;
    }
    const int dn = L.cin - a.col0, nt = (dn + kBN - 1) / kBN;
    const unsigned tile = blockIdx.x - a.wblocks;
    const int64_t m0 = (int64_t)(tile / nt) * kBM, n0 = (int64_t)(tile % nt) * kBN;
    tile_product<false, false>(S, dY, L.W + z * L.wstride + a.col0, L.rows, dn, m0, n0, 0, L.cout, L.cout, L.cin,
                               a.yvec, a.wvec, acc, cs);
    const int64_t m_end = min(m0 + kBM, L.rows);
    auto fetch = [&](int64_t m, int64_t n) {
        const int left = a.pre_in && m < m_end ? (int)min(dn - n, (int64_t)4) : 0;
        return load4(a.pre_in + (row0 + m) * dn + n, left, a.dxvec);
    };
    for_rows(S, acc, m0, n0, fetch, [&](int64_t m, int64_t n, float(&v)[4], const float4& p) {
        if (m >= L.rows || n >= dn) return;
        const int64_t o = (row0 + m) * dn + n;
        if (a.pre_in) {
            v[0] *= dact_f(a.act, p.x);
            v[1] *= dact_f(a.act, p.y);
            v[2] *= dact_f(a.act, p.z);
            v[3] *= dact_f(a.act, p.w);
        }
        store4(a.dX + o, v, dn - n, a.dxvec);
    });
}

struct GradSegs {
    GradSeg s[kGradSegs];
};

// dst[i] += the sum of part[0 .. splits)[i]: a CTA of 32 columns and 8 row lanes (a warp reads 32
// consecutive columns of one partial); lane y sums the partials y, y + 8, .. in order, then the
// lanes' sums are added in order.  blockIdx.y: segment
__global__ void __launch_bounds__(256) grad_sums_kernel(GradSegs g) {
    __shared__ float red[8][32];
    pdl_launch();
    pdl_wait();
    const GradSeg s = g.s[blockIdx.y];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int64_t i0 = (int64_t)blockIdx.x * 32; i0 < s.n; i0 += (int64_t)gridDim.x * 32) {
        const int64_t i = i0 + tx;
        float a = 0.0f;
        if (i < s.n) {
#pragma unroll 8
            for (int z = ty; z < s.splits; z += 8) a += s.part[(int64_t)z * s.n + i];
        }
        red[ty][tx] = a;
        __syncthreads();
        if (ty == 0 && i < s.n) {
            float t = 0.0f;
#pragma unroll
            for (int y = 0; y < 8; ++y) t += red[y][tx];
            s.dst[i] += t;
        }
        __syncthreads();
    }
}

bool aligned16(const float* p, int64_t ld) { return ((uintptr_t)p & 15) == 0 && (ld & 3) == 0; }

}  // namespace

cudaError_t dense_forward(cudaStream_t s, const DenseLayer& L, const float* X, float* pre, float* post,
                          int act) {
    if (L.rows <= 0 || L.cout <= 0) return cudaSuccess;
    const int64_t tiles = (L.rows + kBM - 1) / kBM * ((L.cout + kBN - 1) / kBN);
    const bool wv = aligned16(L.W, L.cin) && (L.wstride & 3) == 0;
    const bool yv = aligned16(pre, L.cout) && (!post || aligned16(post, L.cout));
    return launch_after(dense_forward_kernel, dim3((unsigned)tiles, 1, (unsigned)L.batch), dim3(kThreads), 0, s, L, X,
                        pre, post, act, aligned16(X, L.cin), wv, yv);
}

int64_t dense_grad_floats(int64_t cin, int64_t cout, int64_t rows, int batch, int64_t max_splits) {
    return batch * dense_grad_splits(rows, max_splits) * cout * (cin + 1) + 16;
}

cudaError_t grad_sums_flush(cudaStream_t s, GradSums& g, uint64_t* launches) {
    if (g.count == 0) return cudaSuccess;
    GradSegs k;
    int64_t nmax = 0;
    for (int i = 0; i < g.count; ++i) {
        k.s[i] = g.seg[i];
        if (g.seg[i].n > nmax) nmax = g.seg[i].n;
    }
    int64_t bx = (nmax + 31) / 32;
    if (bx > 4096) bx = 4096;
    ++*launches;
    const dim3 grid((unsigned)bx, (unsigned)g.count);
    g.count = 0;
    g.used = 0;
    return launch_after(grad_sums_kernel, grid, dim3(256), 0, s, k);
}

cudaError_t dense_backward(cudaStream_t s, const DenseLayer& L, const float* X, const float* dY, float* dX,
                           int col0, const float* pre_in, int act, float* dW, float* db, GradSums& g,
                           uint64_t* launches) {
    if (L.rows <= 0 || L.cout <= 0 || L.cin <= 0) return cudaSuccess;
    BackwardArgs a;
    const int64_t splits = dense_grad_splits(L.rows, g.max_splits);
    a.chunk = ((L.rows + splits - 1) / splits + kBK - 1) / kBK * kBK;
    a.splits = (int)((L.rows + a.chunk - 1) / a.chunk);
    const int64_t wn = (int64_t)L.cin * L.cout, sb = (int64_t)a.splits * L.batch;
    if (g.count + 2 * L.batch > kGradSegs || g.used + sb * (wn + L.cout) + 8 > g.cap) {
        cudaError_t e = grad_sums_flush(s, g, launches);
        if (e != cudaSuccess) return e;
    }
    a.wpart = g.take(sb * wn);
    a.bpart = g.take(sb * L.cout);
    if (!a.wpart || !a.bpart) return cudaErrorInvalidValue;  // the workspace holds one layer
    for (int z = 0; z < L.batch; ++z) {
        g.seg[g.count++] = {a.wpart + z * a.splits * wn, dW + z * L.wstride, wn, a.splits};
        g.seg[g.count++] = {a.bpart + (int64_t)z * a.splits * L.cout, db + z * L.wstride, L.cout, a.splits};
    }
    a.X = X;
    a.dY = dY;
    a.dX = dX;
    a.pre_in = pre_in;
    a.col0 = col0;
    a.act = act;
    const int dn = L.cin - col0;
    a.wblocks = (unsigned)(a.splits * (int64_t)((L.cout + kBM - 1) / kBM) * ((L.cin + kBN - 1) / kBN));
    a.dblocks = dX ? (unsigned)((L.rows + kBM - 1) / kBM * ((dn + kBN - 1) / kBN)) : 0u;
    a.xvec = aligned16(X, L.cin);
    a.yvec = aligned16(dY, L.cout);
    a.wvec = aligned16(L.W + col0, L.cin) && (L.wstride & 3) == 0;
    a.dxvec = dX && aligned16(dX, dn) && (!pre_in || aligned16(pre_in, dn));
    ++*launches;
    return launch_after(dense_backward_kernel, dim3(a.wblocks + a.dblocks, 1, (unsigned)L.batch), dim3(kThreads), 0, s,
                        L, a);
}

}  // namespace ndf
