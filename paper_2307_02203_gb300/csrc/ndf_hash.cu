// The paper's neural dependence field architecture (Sec. 4.1-4.2, Fig. 2) on the
// GPU: input embedding = [p, Fourier features (Eq. 4), multi-resolution hash-grid
// features], MLP encoder(s) with Snake-family activations, element-wise product
// merge, MLP decoder, tanh / softplus output; L1 loss (Eq. 3) and Adam.
//
// Layout and definitions are those of the FP64 oracle (hash_net_oracle.h):
//   level l: R_l = base_res * 2^l points per axis, corner-aligned on [-1,1]^3,
//            E_l = min(2^T, R_l^3) entries of F features; dense index
//            x + R y + R^2 z when R^3 <= 2^T, else (x * 1 ^ y * 2654435761 ^
//            z * 805459861) mod 2^T (uint32)
//   params:  per encoder: level tables, then layers (W[out][in], b[out]); then
//            the decoder layers.  One encoder (self field, symmetric by
//            construction) or two (cross field: 0 reference, 1 query).
//
// GPU design: activations are sample-major ([rows][c]; the reference side's rows first, then
// the query side's, so a self field's shared encoder runs once over both).  The dense layers
// are this library's FP32 products (gemm_f32.cu: bias, activation and its derivative in their
// epilogues, deterministic weight-gradient sums), and the rest (embedding, merge, output layer
// with the loss and its gradients, the hash-table scatter of the backward, Adam) are the
// kernels below.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <chrono>
#include <new>
#include <numeric>
#include <vector>

#include "device_common.cuh"
#include "gemm_f32.h"
#include "hash_common.cuh"
#include "ndf_hash_tc.h"
#include "ndf_internal.h"

namespace ndf {

// initial scale of the first encoder layer's weights on the Fourier columns,
// relative to the He-uniform scale of the other weights (see ndf_hash_model_create)
constexpr double kFourierInit = 0.1;

// x0[row][din] = embed(position of the row): rows [0, B) from pos0 with the tables at enc0, rows
// [B, rows) from pos1 with those at enc1.  A CTA embeds 32 rows into shared memory and writes
// them coalesced; its warps split the features of a row (a Fourier axis and frequency or a grid
// level at a time: one row per lane, no divergence), so a batch of 8192 pairs fills the chip
// (one thread per row, measured: 15 us per 8192 rows; this: 6.5 us for all 16,384).
constexpr int kEmbedRows = 32;
__global__ void __launch_bounds__(256)
    hash_embed_kernel(const float* pos0, const float* pos1, int64_t B, int64_t rows,
                      const float* enc0, const float* enc1, EmbedArgs E,
                      float* x0) {
    extern __shared__ float xs[];  // [32][ld], ld odd: conflict-free by row
    pdl_launch();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, ld = E.din | 1;
    const int64_t r0 = (int64_t)blockIdx.x * kEmbedRows, r = r0 + lane;
    if (r < rows) {
        const float* pp = r < B ? pos0 + 3 * r : pos1 + 3 * (r - B);
        const float* enc = r < B ? enc0 : enc1;
        const float p[3] = {pp[0], pp[1], pp[2]};
        float* x = xs + lane * ld;
        for (int u = warp; u < E.levels + 3 * E.L + 1; u += 8) {
            if (u < E.levels) {
                embed_levels(E, enc, p, u, u + 1, [&](int k, float v) { x[3 + 6 * E.L + k] = v; });
            } else if (u < E.levels + 3 * E.L) {
                const int f = u - E.levels, j = f / E.L;
                float sn, cs;
                sincospif(ldexpf(p[j], f - j * E.L), &sn, &cs);
                x[3 + 2 * f] = sn;
                x[4 + 2 * f] = cs;
            } else {
                x[0] = p[0];
                x[1] = p[1];
                x[2] = p[2];
            }
        }
    }
    __syncthreads();
    const int n = (int)min((int64_t)kEmbedRows, rows - r0) * E.din;
    for (int i = threadIdx.x; i < n; i += 256) {
        const int q = i / E.din;
        x0[r0 * E.din + i] = xs[q * ld + (i - q * E.din)];
    }
}

// hash-table gradient: scatter dL/d(embedding) of the hash features, gx[row][ld] from its
// column 0 on (rows as in hash_embed_kernel), one thread per row and level
__global__ void hash_embed_backward_kernel(const float* pos0, const float* pos1,
                                           int64_t B, int64_t rows, const float* gx, int ld,
                                           EmbedArgs E, float* genc0, float* genc1) {
    pdl_launch();
    pdl_wait();
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int l = blockIdx.y;
    if (r >= rows) return;
    const float* pp = r < B ? pos0 + 3 * r : pos1 + 3 * (r - B);
    const float p[3] = {pp[0], pp[1], pp[2]};
    const float* g = gx + r * ld + l * E.F;
    const Cell cl = level_cell(E, l, p);
    float* tab = (r < B ? genc0 : genc1) + E.toff[l];
    for (int f = 0; f < E.F; ++f) {
        const float gv = g[f];
        if (gv == 0.0f) continue;
#pragma unroll
        for (int q = 0; q < 8; ++q) atomicAdd(tab + (int64_t)cl.idx[q] * E.F + f, cl.w[q] * gv);
    }
}

// z from the two latents (d features each, zr broadcast when zr_stride == 0):
// product (the paper's merge), sum, |difference|, or concatenation [zr; zq]
__global__ void merge_kernel(const float* zr, int64_t zr_stride,
                             const float* zq, int d, int64_t B, int mode,
                             float* z) {
    pdl_launch();
    pdl_wait();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)d * B) return;
    const int64_t b = i / d, o = i - b * d;
    const float a = zr[b * zr_stride + o], q = zq[i];
    if (mode == NDF_MERGE_CONCAT) {
        z[b * 2 * d + o] = a;
        z[b * 2 * d + d + o] = q;
    } else {
        z[i] = mode == NDF_MERGE_PRODUCT ? a * q : mode == NDF_MERGE_SUM ? a + q : fabsf(a - q);
    }
}

__global__ void merge_backward_kernel(const float* g, const float* zr,
                                      const float* zq, int d, int64_t B, int mode,
                                      float* gr, float* gq) {
    pdl_launch();
    pdl_wait();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)d * B) return;
    const int64_t b = i / d, o = i - b * d;
    if (mode == NDF_MERGE_CONCAT) {
        gr[i] = g[b * 2 * d + o];
        gq[i] = g[b * 2 * d + d + o];
    } else if (mode == NDF_MERGE_PRODUCT) {
        gr[i] = g[i] * zq[i];
        gq[i] = g[i] * zr[i];
    } else if (mode == NDF_MERGE_SUM) {
        gr[i] = g[i];
        gq[i] = g[i];
    } else {
        const float sg = zr[i] > zq[i] ? 1.0f : (zr[i] < zq[i] ? -1.0f : 0.0f);
        gr[i] = g[i] * sg;
        gq[i] = -g[i] * sg;
    }
}

// The output layer (one output: raw = w . in + bias), y = out_act(raw) and, when target is
// given, the L1 loss, its gradient through the layer and the layer's own gradients: in[B][cin]
// is read once, dX = dL/draw * w (* act'(pre), the pre-activations of `in`, when given), and
// every CTA's sums over its rows of dL/draw * in and dL/draw go to part[blockIdx.x][cin + 1]
// (added in order by grad_sums_flush).  The dot products in the layers' order (16 terms at a time,
// then the slices), eight lanes per row; then one thread
// per column (several row groups when there are fewer columns than threads), 32 rows at a
// time; a CTA takes `chunk` consecutive rows.
constexpr int kOutRows = 32;  // 8 warps x 4 rows
constexpr int64_t kOutMaxCtas = 256;  // partial sums to add
inline int64_t out_chunk(int64_t B) {
    const int64_t c = (B + kOutMaxCtas - 1) / kOutMaxCtas;
    return (c + kOutRows - 1) / kOutRows * kOutRows;
}
__global__ void __launch_bounds__(256)
    hash_out_kernel(const float* in, const float* w, const float* bias,
                    int cin, int64_t B, int64_t chunk, int measure, const float* target,
                    float* y, const float* pre, int act, float* dX, float* part,
                    double* loss) {
    __shared__ float gs[kOutRows];
    __shared__ float red[256];
    __shared__ double ls[8];
    pdl_launch();
    pdl_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t begin = (int64_t)blockIdx.x * chunk, end = min(begin + chunk, B);
    const int cw = cin > 128 ? 256 : cin > 64 ? 128 : 64, subs = 256 / cw;
    const int sub = threadIdx.x / cw, c = threadIdx.x % cw;
    float* pt = target ? part + (int64_t)blockIdx.x * (cin + 1) : nullptr;
    double l = 0.0;
    for (int64_t b0 = begin; b0 < end; b0 += kOutRows) {
        const int n = (int)min((int64_t)kOutRows, end - b0);
        {
            const int r = warp * 4 + (lane >> 3), ch = lane & 7;
            const float* x = in + (b0 + (r < n ? r : 0)) * cin;
            float acc = 0.0f;
            for (int c0 = 0; c0 < cin; c0 += 128) {
                float p = 0.0f;
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const int k = c0 + 16 * ch + i;
                    if (k < cin) p = fmaf(x[k], w[k], p);
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float q = __shfl_sync(0xffffffffu, p, (lane & 24) + j);
                    if (c0 + 16 * j < cin) acc += q;
                }
            }
            const float raw = acc + bias[0];
            const float v = out_act(measure, raw);
            if (r < n && ch == 0) {
                if (y) y[b0 + r] = v;
                if (target) {
                    const float d = v - target[b0 + r];
                    l += fabs((double)d);
                    const float sg = d > 0.0f ? 1.0f : (d < 0.0f ? -1.0f : 0.0f);
                    const float dv = measure == NDF_MEASURE_PEARSON ? 1.0f - v * v : 1.0f / (1.0f + expf(-raw));
                    gs[r] = sg / (float)B * dv;
                }
            }
        }
        if (!target) continue;
        __syncthreads();
        for (int i0 = 0; i0 < cin; i0 += cw) {
            const int i = i0 + c;
            float a = 0.0f;
            if (i < cin) {
                const float wi = w[i];
#pragma unroll 8
                for (int r = sub; r < n; r += subs) {
                    const int64_t o = (b0 + r) * cin + i;
                    const float g = gs[r];
                    a = fmaf(g, in[o], a);
                    float d = g * wi;
                    if (pre) d *= dact_f(act, pre[o]);
                    dX[o] = d;
                }
            }
            red[threadIdx.x] = a;
            __syncthreads();
            if (sub == 0 && i < cin) {
                for (int k = 1; k < subs; ++k) a += red[k * cw + c];
                pt[i] = b0 == begin ? a : pt[i] + a;
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            float a = 0.0f;
            for (int r = 0; r < n; ++r) a += gs[r];
            pt[cin] = b0 == begin ? a : pt[cin] + a;
        }
        __syncthreads();  // gs is rewritten by the next rows
    }
    if (!target) return;
    l += __shfl_xor_sync(0xffffffffu, l, 8);
    l += __shfl_xor_sync(0xffffffffu, l, 16);
    if (lane == 0) ls[warp] = l;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int k = 0; k < 8; ++k) t += ls[k];
        if (t != 0.0) atomicAdd(loss, t);
    }
}

__device__ __forceinline__ void adam_one(float& p, float g, float& m, float& v, float lr, float b1, float b2,
                                         float eps, float c1, float c2) {
    m = b1 * m + (1.0f - b1) * g;
    v = b2 * v + (1.0f - b2) * g * g;
    p -= lr * (m / c1) / (sqrtf(v / c2) + eps);
}

// HBM-bound (28 bytes per parameter).  Four parameters per thread with 16-byte accesses, every
// array streamed once (evict-first); the gradient may be the caller's buffer at any alignment
// (gvec: 16-byte aligned).
__global__ void __launch_bounds__(256)
    hash_adam_kernel(float* p, const float* g, float* m,
                     float* v, int64_t n, bool gvec, float lr, float b1, float b2, float eps,
                     float c1, float c2) {
    pdl_launch();
    pdl_wait();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, j = i << 2;
    if (j + 3 < n) {
        float4 P = __ldcs(reinterpret_cast<const float4*>(p) + i), M = __ldcs(reinterpret_cast<const float4*>(m) + i);
        float4 V = __ldcs(reinterpret_cast<const float4*>(v) + i);
        const float4 G = gvec ? __ldcs(reinterpret_cast<const float4*>(g) + i)
                              : make_float4(__ldcs(g + j), __ldcs(g + j + 1), __ldcs(g + j + 2), __ldcs(g + j + 3));
        adam_one(P.x, G.x, M.x, V.x, lr, b1, b2, eps, c1, c2);
        adam_one(P.y, G.y, M.y, V.y, lr, b1, b2, eps, c1, c2);
        adam_one(P.z, G.z, M.z, V.z, lr, b1, b2, eps, c1, c2);
        adam_one(P.w, G.w, M.w, V.w, lr, b1, b2, eps, c1, c2);
        __stcs(reinterpret_cast<float4*>(p) + i, P);
        __stcs(reinterpret_cast<float4*>(m) + i, M);
        __stcs(reinterpret_cast<float4*>(v) + i, V);
        return;
    }
    for (int64_t k = j; k < n; ++k) adam_one(p[k], g[k], m[k], v[k], lr, b1, b2, eps, c1, c2);
}

__global__ void vertex_positions_kernel(int64_t v0, int64_t n, int64_t X, int64_t Y, int64_t Z,
                                        float* __restrict__ pos) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    vertex_position(v0 + i, X, Y, Z, pos + 3 * i);
}

inline unsigned blocks_for(int64_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

}  // namespace ndf

namespace ndf {

// the tensor-core decoder covers width 128, an embedding of at most 128 inputs
// and the element-wise merges (not concatenation)
static bool hash_tc_eligible(const HashLayout& L) {
    const int nL = L.le + L.ld - 1;
    const int kin = 3 * hash_tc_f8(L.L) + 3 + L.levels * L.F;  // embedding columns in operand order
    return L.c == 128 && kin <= 128 && L.merge != NDF_MERGE_CONCAT && nL >= 1 && nL <= kHashTcMaxLayers;
}

// the query-latent cache needs a latent (an encoder layer) and a decoder layer after it
static bool hash_tc_cache_ok(const HashLayout& L) { return hash_tc_eligible(L) && L.le >= 1 && L.ld >= 2; }

}  // namespace ndf

using namespace ndf;

struct ndf_hash_model {
    ndf_ctx* ctx = nullptr;
    ndf_hash_arch arch{};
    int measure = 0;
    int64_t X = 1, Y = 1, Z = 1;
    HashLayout Ly;
    float *params = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
    int64_t t = 0;
    // workspace for a batch of up to cap samples (encoder buffers: both sides' rows), and of the
    // weight-gradient partial sums
    GradSums sums;
    int64_t cap = 0;
    float* ws = nullptr;
    float *x0 = nullptr, *pre_e[kHashMaxLayers] = {}, *post_e[kHashMaxLayers] = {};
    float *z = nullptr, *pre_d[kHashMaxLayers] = {}, *post_d[kHashMaxLayers] = {};
    float *ga = nullptr, *gb = nullptr, *gl = nullptr;
    float *y = nullptr, *tgt = nullptr, *pos = nullptr;
    double* loss = nullptr;
    // tensor-core decoding: packed BF16 weight images and biases of the parameter
    // version tc_ver, reference latents, per-axis Fourier features of the decode
    // grid, optional cache of the query latents
    int decode_tc = 0, cache_q = 0;
    int64_t ver = 0, tc_ver = -1, lat_ver = -1;
    unsigned char* tc_w = nullptr;
    float *tc_bias = nullptr, *tc_zr = nullptr, *tc_lat = nullptr, *tc_ftab = nullptr;
    // training record
    int passes = 0;
    double last_loss = 0.0, gen_seconds = 0.0, train_seconds = 0.0;
    int64_t n_triples = 0;
};

namespace ndf {

static cudaError_t hash_workspace(ndf_hash_model* m, int64_t B) {
    if (B <= m->cap) return cudaSuccess;
    if (m->ws) cudaFree(m->ws);
    m->ws = nullptr;
    m->cap = 0;
    const HashLayout& L = m->Ly;
    const int64_t c = L.c, wmax = std::max<int64_t>(std::max<int64_t>(L.din, c), L.ddec);
    // loss (2 doubles); both sides' x0 and encoder pre / post; z, decoder pre / post; ga, gb
    // (ping-pong gradients, both sides), gl (latent gradients, both sides); y, tgt, positions
    int64_t floats = 0;
    float* o = nullptr;
    auto take = [&](int64_t n) {
        float* r = o ? o + floats : nullptr;
        floats += (n + 3) & ~int64_t(3);
        return r;
    };
    auto carve = [&]() {
        floats = 0;
        m->loss = reinterpret_cast<double*>(take(4));
        m->x0 = take(2 * B * L.din);
        for (int k = 0; k < L.le; ++k) {
            m->pre_e[k] = take(2 * B * c);
            m->post_e[k] = k < L.le - 1 ? take(2 * B * c) : m->pre_e[k];  // the last layer is linear
        }
        m->z = take(B * L.ddec);
        for (int k = 0; k < L.ld - 1; ++k) {
            m->pre_d[k] = take(B * c);
            m->post_d[k] = take(B * c);
        }
        m->ga = take(2 * B * wmax);
        m->gb = take(2 * B * wmax);
        m->gl = take(2 * B * L.dlat);
        m->y = take(B);
        m->tgt = take(B);
        m->pos = take(6 * B);
    };
    carve();
    cudaError_t e = cudaMalloc(&o, sizeof(float) * (size_t)floats);
    if (e != cudaSuccess) return e;
    m->ws = o;
    carve();
    m->cap = B;
    return cudaSuccess;
}

// The weight gradients' partial sums for batches of up to B pairs (a step's alone: a forward call
// or a decode takes none): all layers where that stays within 128 MB (then one kernel adds them
// all at the end of a step), at least the largest one; with memory too short for that, fewer and
// longer chunks of rows.
static cudaError_t hash_grad_workspace(ndf_hash_model* m, int64_t B) {
    if (B <= m->sums.rows) return cudaSuccess;
    if (m->sums.work) cudaFree(m->sums.work);
    m->sums = GradSums();
    const HashLayout& L = m->Ly;
    const int64_t c = L.c, out_blocks = std::min<int64_t>((B + kOutRows - 1) / kOutRows, kOutMaxCtas);
    const int64_t out_part = out_blocks * (std::max<int64_t>(L.ddec, c) + 1) + 4;
    cudaError_t e = cudaErrorMemoryAllocation;
    for (int64_t splits = kGradSplits; splits >= 1 && e == cudaErrorMemoryAllocation; splits /= 2) {
        const int64_t enc =
            L.le > 0 ? dense_grad_floats(std::max<int64_t>(L.din, c), c, 2 * B / L.n_enc, L.n_enc, splits) : 0;
        const int64_t dec = dense_grad_floats(std::max<int64_t>(L.ddec, c), c, B, 1, splits);
        const int64_t one = std::max(std::max(enc, dec), out_part), all = L.le * enc + L.ld * dec + out_part;
        m->sums.max_splits = splits;
        for (int64_t cap : {std::max(one, std::min<int64_t>(all, int64_t(32) << 20)), one}) {
            m->sums.cap = cap;
            e = cudaMalloc(&m->sums.work, sizeof(float) * (size_t)cap);
            if (e != cudaErrorMemoryAllocation) break;
            cudaGetLastError();
        }
    }
    if (e != cudaSuccess) {
        m->sums = GradSums();
        return e;
    }
    m->sums.rows = B;
    return cudaSuccess;
}

// encoder layer k over `batch` weight sets from encoder e on, `rows` rows each
static DenseLayer enc_layer(const ndf_hash_model* m, int e, int k, int64_t rows, int batch) {
    const HashLayout& L = m->Ly;
    DenseLayer d;
    const float* enc = m->params + L.enc_size * e;
    d.W = enc + L.ew[k];
    d.b = enc + L.eb[k];
    d.cin = k == 0 ? L.din : L.c;
    d.cout = L.c;
    d.rows = rows;
    d.batch = batch;
    d.wstride = L.enc_size;
    return d;
}

static DenseLayer dec_layer(const ndf_hash_model* m, int k, int64_t rows) {
    const HashLayout& L = m->Ly;
    DenseLayer d;
    d.W = m->params + L.dw[k];
    d.b = m->params + L.db[k];
    d.cin = k == 0 ? L.ddec : L.c;
    d.cout = L.c;
    d.rows = rows;
    return d;
}

static const float* post_or_null(const float* pre, const float* post) { return pre == post ? nullptr : post; }

// The encoder chain over rows row0 .. row0 + rows of the workspace: rows [0, B) of them take
// their positions from pos0, the rest from pos1; `batch` weight sets from encoder e on share the
// rows evenly.  Leaves x0, pre and post of the rows.
static cudaError_t encode_rows(ndf_hash_model* m, int e, int batch, const float* pos0, const float* pos1,
                               int64_t B, int64_t rows, int64_t row0) {
    const HashLayout& L = m->Ly;
    ndf_ctx* ctx = m->ctx;
    const float* enc0 = m->params + L.enc_size * e;
    float* x0 = m->x0 + row0 * L.din;
    // an ordinary launch: the table reads (__ldg) must not start beside whatever wrote the tables
    hash_embed_kernel<<<blocks_for(rows, kEmbedRows), 256, sizeof(float) * kEmbedRows * (size_t)(L.din | 1),
                        ctx->stream>>>(pos0, pos1, B, rows, enc0, enc0 + L.enc_size * (batch - 1), embed_args(L), x0);
    ctx->launches++;
    cudaError_t st = cudaGetLastError();
    const float* in = x0;
    for (int k = 0; k < L.le && st == cudaSuccess; ++k) {
        float *pre = m->pre_e[k] + row0 * L.c, *post = m->post_e[k] + row0 * L.c;
        st = dense_forward(ctx->stream, enc_layer(m, e, k, rows / batch, batch), in, pre,
                           const_cast<float*>(post_or_null(pre, post)), L.act);
        ctx->launches++;
        in = post;
    }
    return st;
}

// the latents: the last encoder layer, or the embedding (grid-only), from row row0 on
static const float* latent(const ndf_hash_model* m, int64_t row0) {
    return (m->Ly.le > 0 ? m->post_e[m->Ly.le - 1] : m->x0) + row0 * m->Ly.dlat;
}

// decoder over m->z: the hidden layers, then the output layer (y; with target the loss and the
// gradient of the output layer's input in m->ga, its own gradients' partial sums listed)
static cudaError_t decode_z(ndf_hash_model* m, int64_t B, const float* target, float* y, float* grad) {
    const HashLayout& L = m->Ly;
    ndf_ctx* ctx = m->ctx;
    const float* in = m->z;
    cudaError_t e = cudaSuccess;
    for (int k = 0; k < L.ld - 1 && e == cudaSuccess; ++k) {
        e = dense_forward(ctx->stream, dec_layer(m, k, B), in, m->pre_d[k], m->post_d[k], L.act);
        ctx->launches++;
        in = m->post_d[k];
    }
    if (e != cudaSuccess) return e;
    const int k = L.ld - 1, cin = k == 0 ? L.ddec : L.c;
    const int64_t chunk = target ? out_chunk(B) : kOutRows;
    const unsigned blocks = (unsigned)((B + chunk - 1) / chunk);
    float* part = nullptr;
    if (target) {
        GradSums& g = m->sums;
        part = g.take((int64_t)blocks * (cin + 1));
        if (!part) return cudaErrorInvalidValue;  // the list is empty here and holds one layer
        // weights and bias are adjacent in the parameters: one segment
        g.seg[g.count++] = {part, grad + L.dw[k], cin + 1, (int)blocks};
    }
    launch_after(hash_out_kernel, dim3(blocks), dim3(256), 0, ctx->stream, in, m->params + L.dw[k],
                 m->params + L.db[k], cin, B, chunk, m->measure, target, y, k > 0 ? m->pre_d[k - 1] : nullptr,
                 L.act, m->ga, part, m->loss);
    ctx->launches++;
    return cudaGetLastError();
}

// full forward (and, with target, the L1 loss and the gradient, added to grad[total])
static cudaError_t hash_forward_backward(ndf_hash_model* m, const float* pr, const float* pq,
                                         const float* target, int64_t B, float* y, float* grad) {
    const HashLayout& L = m->Ly;
    ndf_ctx* ctx = m->ctx;
    cudaStream_t s = ctx->stream;
    GradSums& g = m->sums;
    g.count = 0;
    g.used = 0;
    const int batch = L.n_enc;  // a shared encoder sees both sides' rows at once
    cudaError_t e = encode_rows(m, 0, batch, pr, pq, B, 2 * B, 0);
    if (e != cudaSuccess) return e;
    const float *zr = latent(m, 0), *zq = latent(m, B);
    launch_after(merge_kernel, dim3(blocks_for((int64_t)L.dlat * B)), dim3(256), 0, s, zr, L.dlat, zq, L.dlat,
                 B, L.merge, m->z);
    ctx->launches++;
    if ((e = decode_z(m, B, target, y, grad)) != cudaSuccess || !target) return e;
    // ---- backward: decoder (ping-pong ga / gb), merge, then the encoder chain
    float *cur = m->ga, *other = m->gb;
    for (int k = L.ld - 2; k >= 0; --k) {
        e = dense_backward(s, dec_layer(m, k, B), k == 0 ? m->z : m->post_d[k - 1], cur, other, 0,
                           k > 0 ? m->pre_d[k - 1] : nullptr, L.act, grad + L.dw[k], grad + L.db[k], g,
                           &ctx->launches);
        if (e != cudaSuccess) return e;
        std::swap(cur, other);
    }
    launch_after(merge_backward_kernel, dim3(blocks_for((int64_t)L.dlat * B)), dim3(256), 0, s, cur, zr, zq,
                 L.dlat, B, L.merge, m->gl, m->gl + B * L.dlat);
    ctx->launches++;
    const float* gs = m->gl;
    cur = m->ga;
    other = m->gb;
    const int col0 = 3 + 6 * L.L;  // positions and Fourier features have no parameters behind them
    for (int k = L.le - 1; k >= 0; --k) {
        e = dense_backward(s, enc_layer(m, 0, k, 2 * B / batch, batch), k == 0 ? m->x0 : m->post_e[k - 1], gs, cur,
                           k == 0 ? col0 : 0, k > 0 ? m->pre_e[k - 1] : nullptr, L.act, grad + L.ew[k],
                           grad + L.eb[k], g, &ctx->launches);
        if (e != cudaSuccess) return e;
        gs = cur;
        std::swap(cur, other);
    }
    const bool grid_only = L.le == 0;
    launch_after(hash_embed_backward_kernel, dim3(blocks_for(2 * B), (unsigned)L.levels), dim3(256), 0, s, pr,
                 pq, B, 2 * B, grid_only ? gs + col0 : gs, grid_only ? L.din : L.din - col0, embed_args(L),
                 grad, grad + L.enc_size * (L.n_enc - 1));
    ctx->launches++;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return grad_sums_flush(s, g, &ctx->launches);
}


// ---------------------------------------------------------------- tensor-core decoding
// Packed images: [encoder 0 layers][encoder 1 layers (cross)][decoder hidden layers],
// so that a query-side chain (encoder eq, then the decoder) is contiguous.
static cudaError_t hash_tc_prepare(ndf_hash_model* m) {
    const HashLayout& L = m->Ly;
    const int n = L.n_enc * L.le + L.ld - 1;
    const size_t lb = hash_tc_layer_bytes();
    cudaError_t e = cudaSuccess;
    if (!m->tc_w) {
        e = cudaMalloc(&m->tc_w, lb * (size_t)n);
        if (e == cudaSuccess) e = cudaMalloc(&m->tc_bias, sizeof(float) * 128 * (size_t)n);
        if (e == cudaSuccess) e = cudaMalloc(&m->tc_zr, sizeof(float) * 128 * (size_t)kHashTcMaxRefs);
        const int f8 = hash_tc_f8(L.L);
        const size_t nf = (size_t)(m->X + m->Y + m->Z) * (size_t)f8;
        if (e == cudaSuccess) e = cudaMalloc(&m->tc_ftab, sizeof(float) * std::max<size_t>(nf, 4));
        if (e == cudaSuccess) e = launch_hash_tc_ftab(L.L, f8, m->X, m->Y, m->Z, m->tc_ftab, m->ctx->stream);
        m->ctx->launches++;
        if (e != cudaSuccess) return e;
    }
    if (m->tc_ver == m->ver) return cudaSuccess;
    HashTcPack pk;
    pk.L = L.L;
    pk.f8 = hash_tc_f8(L.L);
    pk.ngrid = L.levels * L.F;
    for (int en = 0; en < L.n_enc; ++en)
        for (int k = 0; k < L.le; ++k) {
            pk.perm[pk.n] = k == 0;
            pk.cin[pk.n] = k == 0 ? L.din : L.c;
            pk.w[pk.n] = L.enc_size * en + L.ew[k];
            pk.b[pk.n] = L.enc_size * en + L.eb[k];
            ++pk.n;
        }
    for (int k = 0; k < L.ld - 1; ++k) {
        pk.perm[pk.n] = k == 0 && L.le == 0;  // grid-only: the merged embedding
        pk.cin[pk.n] = k == 0 ? L.ddec : L.c;
        pk.w[pk.n] = L.dw[k];
        pk.b[pk.n] = L.db[k];
        ++pk.n;
    }
    e = launch_hash_tc_pack(m->params, pk, m->tc_w, m->tc_bias, m->ctx->stream);
    m->ctx->launches++;
    if (e == cudaSuccess) m->tc_ver = m->ver;
    return e;
}

static HashTcArgs hash_tc_base(const ndf_hash_model* m) {
    HashTcArgs a;
    a.E = embed_args(m->Ly);
    a.measure = m->measure;
    a.X = m->X;
    a.Y = m->Y;
    a.Z = m->Z;
    a.status = m->ctx->flag.as<unsigned>() + 1;
    a.ftab = m->tc_ftab;
    a.f8 = hash_tc_f8(m->Ly.L);
    a.foff[0] = 0;
    a.foff[1] = m->X * a.f8;
    a.foff[2] = (m->X + m->Y) * a.f8;
    return a;
}

// CTAs per reference: the SMs shared among the references (the launcher caps it at
// the tile groups there are)
static int hash_tc_ctas(const ndf_hash_model* m, int64_t rows, int R) {
    (void)rows;
    const int c = (m->ctx->sm_count + R - 1) / R;
    return c < 1 ? 1 : c;
}

// encode-only launch: the FP32 latents of encoder `en` for rows vertices
// (vlist when given, else 0 .. rows-1) into lat[rows][128]
static cudaError_t hash_tc_encode(ndf_hash_model* m, int en, const int64_t* vlist, int64_t rows, float* lat) {
    const HashLayout& L = m->Ly;
    HashTcArgs a = hash_tc_base(m);
    a.tables = m->params + L.enc_size * en;
    a.wimg = m->tc_w + hash_tc_layer_bytes() * (size_t)(en * L.le);
    a.bias = m->tc_bias + (size_t)128 * (en * L.le);
    a.nL = L.le;
    a.n_enc = L.le;
    a.merge = -1;
    a.N = rows;
    if (vlist) {
        a.vlist_n = (int)rows;
        for (int64_t i = 0; i < rows; ++i) a.vlist[i] = vlist[i];
    }
    a.lat = lat;
    m->ctx->launches++;
    return launch_hash_tc(a, L.act, hash_tc_ctas(m, rows, 1), 1, m->ctx->stream);
}

// volumes of R <= kHashTcMaxRefs references into out[R][N] (device)
static cudaError_t hash_tc_decode(ndf_hash_model* m, const int64_t* refs, int R, float* out) {
    const HashLayout& L = m->Ly;
    ndf_ctx* ctx = m->ctx;
    const int64_t N = m->X * m->Y * m->Z;
    cudaError_t e = hash_tc_prepare(m);
    if (e != cudaSuccess) return e;
    // reference latents (encoder 0)
    if (L.le == 0) {
        HashTcArgs a = hash_tc_base(m);
        a.tables = m->params;
        a.vlist_n = R;
        for (int i = 0; i < R; ++i) a.vlist[i] = refs[i];
        e = launch_hash_tc_embed_refs(a, m->tc_zr, ctx->stream);
        ctx->launches++;
    } else {
        e = hash_tc_encode(m, 0, refs, R, m->tc_zr);
    }
    if (e != cudaSuccess) return e;
    const int eq = L.n_enc - 1;
    const bool cached = m->cache_q && hash_tc_cache_ok(L);
    if (cached && m->lat_ver != m->ver) {
        if (!m->tc_lat && (e = cudaMalloc(&m->tc_lat, sizeof(float) * 128 * (size_t)N)) != cudaSuccess) return e;
        if ((e = hash_tc_encode(m, eq, nullptr, N, m->tc_lat)) != cudaSuccess) return e;
        m->lat_ver = m->ver;
    }
    HashTcArgs a = hash_tc_base(m);
    a.merge = L.merge;
    a.zr = m->tc_zr;
    a.w_last = m->params + L.dw[L.ld - 1];
    a.b_last = m->params + L.db[L.ld - 1];
    a.N = N;
    a.out = out;
    const int first = cached ? L.n_enc * L.le : eq * L.le;
    a.wimg = m->tc_w + hash_tc_layer_bytes() * (size_t)first;
    a.bias = m->tc_bias + (size_t)128 * first;
    if (cached) {
        a.lat_in = m->tc_lat;
        a.nL = L.ld - 1;
        a.n_enc = 0;
    } else {
        a.tables = m->params + L.enc_size * eq;
        a.nL = L.le + L.ld - 1;
        a.n_enc = L.le;
    }
    ctx->launches++;
    return launch_hash_tc(a, L.act, hash_tc_ctas(m, N, R), R, ctx->stream);
}

// the FP32 path for one reference: the reference encoded once, queries in chunks
static cudaError_t hash_fp32_decode(ndf_hash_model* m, int64_t ref_idx, float* dev_out) {
    ndf_ctx* ctx = m->ctx;
    const HashLayout& L = m->Ly;
    const int64_t N = m->X * m->Y * m->Z;
    const int64_t chunk = std::min<int64_t>(N, 65536);
    cudaError_t e = hash_workspace(m, chunk);
    if (e != cudaSuccess) return e;
    // rows of the workspace: the reference in row 0, a chunk of queries from row `chunk` on
    vertex_positions_kernel<<<1, 32, 0, ctx->stream>>>(ref_idx, 1, m->X, m->Y, m->Z, m->pos);
    ctx->launches++;
    e = encode_rows(m, 0, 1, m->pos, m->pos, 1, 1, 0);
    const float* zr = latent(m, 0);
    float* pq = m->pos + 3 * chunk;
    for (int64_t v0 = 0; v0 < N && e == cudaSuccess; v0 += chunk) {
        const int64_t n = std::min(chunk, N - v0);
        vertex_positions_kernel<<<blocks_for(n), 256, 0, ctx->stream>>>(v0, n, m->X, m->Y, m->Z, pq);
        ctx->launches++;
        e = encode_rows(m, L.n_enc - 1, 1, pq, pq, n, n, chunk);
        if (e != cudaSuccess) break;
        launch_after(merge_kernel, dim3(blocks_for((int64_t)L.dlat * n)), dim3(256), 0, ctx->stream, zr, 0,
                     latent(m, chunk), L.dlat, n, L.merge, m->z);
        ctx->launches++;
        e = decode_z(m, n, nullptr, dev_out + v0, nullptr);
    }
    return e;
}
}  // namespace ndf

extern "C" {

void ndf_hash_arch_default(ndf_hash_arch* a) {
    if (!a) return;
    a->levels = 6;
    a->base_res = 16;
    a->log2_table = 22;
    a->feat = 2;
    a->n_freq = 12;
    a->width = 128;
    a->enc_layers = 6;
    a->dec_layers = 6;
    a->act = NDF_ACT_SNAKEALT;
    a->merge = NDF_MERGE_PRODUCT;
}

ndf_status ndf_hash_model_create(ndf_ctx* ctx, const ndf_hash_arch* arch, int measure, int cross,
                                 uint64_t seed, int64_t X, int64_t Y, int64_t Z,
                                 ndf_hash_model** out) {
    if (!ctx || !arch || !out) return NDF_ERR_ARG;
    *out = nullptr;
    if (measure != NDF_MEASURE_PEARSON && measure != NDF_MEASURE_MI_KSG)
        return fail(ctx, NDF_ERR_ARG, "unknown measure %d", measure);
    if (X < 1 || Y < 1 || Z < 1 || X * Y * Z > (int64_t(1) << 31))
        return fail(ctx, NDF_ERR_ARG, "bad decode grid");
    ndf_hash_model* m = new (std::nothrow) ndf_hash_model();
    if (!m) return NDF_ERR_OOM;
    m->ctx = ctx;
    m->arch = *arch;
    m->measure = measure;
    m->X = X;
    m->Y = Y;
    m->Z = Z;
    if (!m->Ly.init(*arch, cross ? 2 : 1)) {
        delete m;
        return fail(ctx, NDF_ERR_ARG, "bad hash-network architecture");
    }
    cudaSetDevice(ctx->device);
    const size_t bytes = sizeof(float) * (size_t)m->Ly.total;
    cudaError_t e = cudaMalloc(&m->params, bytes);
    if (e == cudaSuccess) e = cudaMalloc(&m->grad, bytes);
    if (e == cudaSuccess) e = cudaMalloc(&m->m, bytes);
    if (e == cudaSuccess) e = cudaMalloc(&m->v, bytes);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->m, 0, bytes, ctx->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->v, 0, bytes, ctx->stream);
    if (e != cudaSuccess) {
        ndf_hash_model_free(m);
        return cuda_fail(ctx, e, "hash model allocation");
    }
    // initialisation: tables U(-0.1, 0.1), weights U(-sqrt(6/in), sqrt(6/in)), biases 0, and a
    // zero last decoder layer (the untrained field is constant: without it, the sin^2 term
    // of Snake-family activations drifts the output and L1 training collapses it).  The
    // first encoder layer's weights on the Fourier columns start at kFourierInit of that
    // scale: at full scale the frequencies up to 2^(L-1) pi reach every latent feature, the
    // untrained encoder maps positions a cell apart to unrelated latents, the product merge
    // carries no dependence signal, and on a field whose pairs are mostly uncorrelated the
    // L1 loss keeps the network at the constant predictor
    std::vector<float> h((size_t)m->Ly.total, 0.0f);
    uint64_t st = seed * 0x9e3779b97f4a7c15ULL + 0x1234567ULL;
    auto unif = [&]() {
        st += 0x9e3779b97f4a7c15ULL;
        uint64_t z = st;
        z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
        z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
        z ^= z >> 31;
        return (double)(z >> 11) * (1.0 / 9007199254740992.0) * 2.0 - 1.0;
    };
    const HashLayout& L = m->Ly;
    for (int e_i = 0; e_i < L.n_enc; ++e_i) {
        const int64_t base = L.enc_size * e_i;
        for (int64_t i = 0; i < L.tables; ++i) h[(size_t)(base + i)] = (float)(0.1 * unif());
        for (int k = 0; k < L.le; ++k) {
            const int64_t cin = k == 0 ? L.din : L.c;
            const double a = sqrt(6.0 / (double)cin);
            for (int64_t i = 0; i < cin * L.c; ++i) {
                const int64_t col = i % cin;  // W[out][in]
                const bool fourier = k == 0 && col >= 3 && col < 3 + 6 * (int64_t)L.L;
                h[(size_t)(base + L.ew[k] + i)] = (float)((fourier ? kFourierInit : 1.0) * a * unif());
            }
        }
    }
    for (int k = 0; k < L.ld - 1; ++k) {
        const int64_t cin = k == 0 ? L.ddec : L.c;
        const double a = sqrt(6.0 / (double)cin);
        for (int64_t i = 0; i < cin * L.c; ++i) h[(size_t)(L.dw[k] + i)] = (float)(a * unif());
    }
    e = cudaMemcpyAsync(m->params, h.data(), bytes, cudaMemcpyHostToDevice, ctx->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    if (e != cudaSuccess) {
        ndf_hash_model_free(m);
        return cuda_fail(ctx, e, "hash model initialisation");
    }
    m->decode_tc = hash_tc_eligible(m->Ly) ? 1 : 0;
    *out = m;
    return NDF_OK;
}

void ndf_hash_model_free(ndf_hash_model* m) {
    if (!m) return;
    if (m->ctx) cudaStreamSynchronize(m->ctx->stream);
    void* ps[] = {m->params, m->grad, m->m, m->v, m->ws, m->sums.work, m->tc_w, m->tc_bias,
                  m->tc_zr, m->tc_lat, m->tc_ftab};
    for (void* q : ps)
        if (q) cudaFree(q);
    delete m;
}

int64_t ndf_hash_model_param_count(const ndf_hash_model* m) { return m ? m->Ly.total : -1; }

ndf_status ndf_hash_model_get_params(ndf_hash_model* m, float* out) {
    if (!m || !out) return NDF_ERR_ARG;
    const size_t bytes = sizeof(float) * (size_t)m->Ly.total;
    cudaError_t e = cudaMemcpyAsync(out, m->params, bytes, cudaMemcpyDefault, m->ctx->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->ctx->stream);
    return e == cudaSuccess ? NDF_OK : cuda_fail(m->ctx, e, "hash params download");
}

ndf_status ndf_hash_model_set_params(ndf_hash_model* m, const float* in) {
    if (!m || !in) return NDF_ERR_ARG;
    const size_t bytes = sizeof(float) * (size_t)m->Ly.total;
    cudaError_t e = cudaMemcpyAsync(m->params, in, bytes, cudaMemcpyDefault, m->ctx->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->ctx->stream);
    ++m->ver;
    return e == cudaSuccess ? NDF_OK : cuda_fail(m->ctx, e, "hash params upload");
}

static cudaError_t hash_adam(ndf_hash_model* m, const float* grad, float lr) {
    ++m->t;
    ++m->ver;
    const float c1 = 1.0f - powf(0.9f, (float)m->t), c2 = 1.0f - powf(0.999f, (float)m->t);
    launch_after(hash_adam_kernel, dim3(blocks_for((m->Ly.total + 3) / 4)), dim3(256), 0, m->ctx->stream,
                 m->params, grad, m->m, m->v, m->Ly.total, ((uintptr_t)grad & 15) == 0, lr, 0.9f, 0.999f,
                 1e-8f, c1, c2);
    m->ctx->launches++;
    return cudaGetLastError();
}

// one training step on device batches (no copies, no host synchronisation): the
// summed |error| of the batch accumulates in m->loss
static cudaError_t hash_train_step(ndf_hash_model* m, const float* pr, const float* pq,
                                   const float* target, int64_t B, float lr) {
    ndf_ctx* ctx = m->ctx;
    cudaError_t e = cudaMemsetAsync(m->grad, 0, sizeof(float) * (size_t)m->Ly.total, ctx->stream);
    if (e == cudaSuccess) e = hash_forward_backward(m, pr, pq, target, B, nullptr, m->grad);
    if (e != cudaSuccess) return e;
    return hash_adam(m, m->grad, lr);
}

ndf_status ndf_hash_model_step(ndf_hash_model* m, const float* pr, const float* pq,
                               const float* target, int64_t B, float lr, int apply,
                               float* grad_out, double* loss_out) {
    if (!m || !pr || !pq || !target || B < 1) return NDF_ERR_ARG;
    ndf_ctx* ctx = m->ctx;
    cudaSetDevice(ctx->device);
    cudaError_t e = hash_workspace(m, B);
    if (e == cudaSuccess) e = hash_grad_workspace(m, B);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "hash workspace");
    const size_t pb = sizeof(float) * 3 * (size_t)B;
    e = cudaMemcpyAsync(m->pos, pr, pb, cudaMemcpyDefault, ctx->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(m->pos + 3 * B, pq, pb, cudaMemcpyDefault, ctx->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(m->tgt, target, sizeof(float) * B, cudaMemcpyDefault, ctx->stream);
    // a gradient buffer of the caller on this device serves as the step's own (no copy of it)
    const size_t gb = sizeof(float) * (size_t)m->Ly.total;
    float* grad = grad_out && device_writable(ctx, grad_out) ? grad_out : m->grad;
    if (e == cudaSuccess) e = cudaMemsetAsync(grad, 0, gb, ctx->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->loss, 0, sizeof(double), ctx->stream);
    if (e == cudaSuccess) e = hash_forward_backward(m, m->pos, m->pos + 3 * B, m->tgt, B, nullptr, grad);
    if (e == cudaSuccess && apply) e = hash_adam(m, grad, lr);
    double l = 0.0;
    if (e == cudaSuccess && grad_out && grad != grad_out)
        e = cudaMemcpyAsync(grad_out, grad, gb, cudaMemcpyDefault, ctx->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&l, m->loss, sizeof(double), cudaMemcpyDeviceToHost, ctx->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "hash step");
    if (loss_out) *loss_out = l / (double)B;
    return NDF_OK;
}

ndf_status ndf_hash_model_forward(ndf_hash_model* m, const float* pr, const float* pq, int64_t B,
                                  float* out) {
    if (!m || !pr || !pq || !out || B < 1) return NDF_ERR_ARG;
    ndf_ctx* ctx = m->ctx;
    cudaSetDevice(ctx->device);
    cudaError_t e = hash_workspace(m, B);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "hash workspace");
    const size_t pb = sizeof(float) * 3 * (size_t)B;
    e = cudaMemcpyAsync(m->pos, pr, pb, cudaMemcpyDefault, ctx->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(m->pos + 3 * B, pq, pb, cudaMemcpyDefault, ctx->stream);
    if (e == cudaSuccess) e = hash_forward_backward(m, m->pos, m->pos + 3 * B, nullptr, B, m->y, nullptr);
    if (e == cudaSuccess) e = cudaMemcpyAsync(out, m->y, sizeof(float) * B, cudaMemcpyDefault, ctx->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    return e == cudaSuccess ? NDF_OK : cuda_fail(ctx, e, "hash forward");
}

// the volume of one reference vertex (tensor-core decoder or the FP32 chain)
ndf_status ndf_hash_infer(ndf_hash_model* m, int64_t ref_idx, float* out) {
    return ndf_hash_infer_batch(m, &ref_idx, 1, out);
}

ndf_status ndf_hash_infer_batch(ndf_hash_model* m, const int64_t* refs, int32_t R, float* out) {
    if (!m || !refs || !out || R < 1) return NDF_ERR_ARG;
    ndf_ctx* ctx = m->ctx;
    const int64_t N = m->X * m->Y * m->Z;
    for (int32_t i = 0; i < R; ++i)
        if (refs[i] < 0 || refs[i] >= N) return fail(ctx, NDF_ERR_ARG, "ref_idx out of range");
    cudaSetDevice(ctx->device);
    void* dev_out;
    bool is_host;
    const size_t bytes = sizeof(float) * (size_t)N * (size_t)R;
    ndf_status st = resolve_out(ctx, out, bytes, &dev_out, &is_host);
    if (st != NDF_OK) return st;
    float* o = static_cast<float*>(dev_out);
    cudaError_t e = cudaSuccess;
    if (m->decode_tc) {
        for (int32_t r0 = 0; r0 < R && e == cudaSuccess; r0 += kHashTcMaxRefs)
            e = hash_tc_decode(m, refs + r0, std::min<int32_t>(kHashTcMaxRefs, R - r0), o + (size_t)r0 * N);
    } else {
        for (int32_t r = 0; r < R && e == cudaSuccess; ++r) e = hash_fp32_decode(m, refs[r], o + (size_t)r * N);
    }
    if (e != cudaSuccess) return cuda_fail(ctx, e, "hash decode");
    return finish_out(ctx, out, dev_out, bytes, is_host);
}

ndf_status ndf_hash_set_decode(ndf_hash_model* m, int32_t mode, int32_t cache_queries) {
    if (!m) return NDF_ERR_ARG;
    if (mode != NDF_HASH_DECODE_FP32 && mode != NDF_HASH_DECODE_TC)
        return fail(m->ctx, NDF_ERR_ARG, "unknown decode mode %d", mode);
    if (mode == NDF_HASH_DECODE_TC && !hash_tc_eligible(m->Ly))
        return fail(m->ctx, NDF_ERR_ARG,
                    "the tensor-core decoder needs width 128, at most 128 embedding inputs and a "
                    "product / sum / |difference| merge");
    if (cache_queries && (mode != NDF_HASH_DECODE_TC || !hash_tc_cache_ok(m->Ly)))
        return fail(m->ctx, NDF_ERR_ARG,
                    "the query-latent cache needs the tensor-core decoder, an encoder layer and two "
                    "decoder layers");
    m->decode_tc = mode;
    m->cache_q = cache_queries ? 1 : 0;
    if (!m->cache_q && m->tc_lat) {
        cudaStreamSynchronize(m->ctx->stream);
        cudaFree(m->tc_lat);
        m->tc_lat = nullptr;
        m->lat_ver = -1;
    }
    return NDF_OK;
}

int32_t ndf_hash_get_decode(const ndf_hash_model* m) { return m ? m->decode_tc : -1; }

// training on continuous samples renewed every pass (Sec. 4.3)
ndf_status ndf_hash_train(ndf_ctx* ctx, int ref_field, int query_field, int measure, int k,
                          const ndf_hash_arch* arch, const ndf_train_cfg* cfg_in,
                          ndf_hash_model** out) {
    if (!ctx || !arch || !out) return NDF_ERR_ARG;
    ndf_train_cfg cfg;
    if (cfg_in) cfg = *cfg_in;
    else ndf_train_cfg_default(&cfg);
    const Field *rf, *qf;
    ndf_status st = check_pair(ctx, ref_field, query_field, 0, &rf, &qf);
    if (st != NDF_OK) return st;
    if (measure == NDF_MEASURE_MI_KSG && (k < 1 || k >= rf->M || k > kKsgMaxK || rf->M > kKsgMaxM))
        return fail(ctx, NDF_ERR_ARG, "bad k or M for the KSG targets");
    if (cfg.n_triples < 1 || cfg.batch < 1 || cfg.max_passes < 1 || cfg.n_triples > (int64_t(1) << 31))
        return fail(ctx, NDF_ERR_ARG, "bad training configuration");
    ndf_hash_model* m = nullptr;
    if ((st = ndf_hash_model_create(ctx, arch, measure, ref_field != query_field, cfg.seed, qf->X,
                                    qf->Y, qf->Z, &m)) != NDF_OK)
        return st;
    if (measure == NDF_MEASURE_MI_KSG && (st = ensure_psi_table(ctx, rf->M + 1)) != NDF_OK) {
        ndf_hash_model_free(m);
        return st;
    }
    const int64_t T = cfg.n_triples, B = std::min(cfg.batch, T);
    float *pref = nullptr, *pq = nullptr, *tgt = nullptr;
    cudaError_t e = cudaMalloc(&pref, sizeof(float) * 3 * (size_t)T);
    if (e == cudaSuccess) e = cudaMalloc(&pq, sizeof(float) * 3 * (size_t)T);
    if (e == cudaSuccess) e = cudaMalloc(&tgt, sizeof(float) * (size_t)T);
    if (e == cudaSuccess) e = hash_workspace(m, B);
    if (e == cudaSuccess) e = hash_grad_workspace(m, B);
    SampleScratch sc;
    auto cleanup = [&]() {
        if (pref) cudaFree(pref);
        if (pq) cudaFree(pq);
        if (tgt) cudaFree(tgt);
        sc.release();
    };
    const auto t_start = std::chrono::steady_clock::now();
    float lr = cfg.lr;
    double best = 1e300;
    int bad = 0, decays = 0;
    for (int pass = 0; pass < cfg.max_passes && e == cudaSuccess; ++pass) {
        const auto g0 = std::chrono::steady_clock::now();
        e = sample_triples_dev(ctx, *rf, *qf, measure, k, T, cfg.seed + (uint64_t)pass, pref, pq, tgt, sc);
        m->gen_seconds += std::chrono::duration<double>(std::chrono::steady_clock::now() - g0).count();
        if (e != cudaSuccess) break;
        // the pass's steps run back to back; its summed |error| is read once
        e = cudaMemsetAsync(m->loss, 0, sizeof(double), ctx->stream);
        for (int64_t b0 = 0; b0 < T && e == cudaSuccess; b0 += B)
            e = hash_train_step(m, pref + 3 * b0, pq + 3 * b0, tgt + b0, std::min(B, T - b0), lr);
        double pass_sum = 0.0;
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(&pass_sum, m->loss, sizeof(double), cudaMemcpyDeviceToHost, ctx->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
        if (e != cudaSuccess) break;
        const double pass_loss = pass_sum / (double)T;
        m->last_loss = pass_loss;
        m->passes = pass + 1;
        if (pass_loss < best * (1.0 - 1e-4)) {
            best = pass_loss;
            bad = 0;
        } else if (++bad > cfg.patience) {
            lr *= 0.1f;
            bad = 0;
            if (++decays > cfg.max_decays) break;
        }
        const double el = std::chrono::duration<double>(std::chrono::steady_clock::now() - t_start).count();
        if (cfg.time_budget_s > 0.0 && el > cfg.time_budget_s) break;
    }
    m->train_seconds =
        std::chrono::duration<double>(std::chrono::steady_clock::now() - t_start).count() - m->gen_seconds;
    m->n_triples = T;
    cleanup();
    if (e != cudaSuccess) {
        ndf_hash_model_free(m);
        return cuda_fail(ctx, e, "hash training");
    }
    *out = m;
    return NDF_OK;
}

ndf_status ndf_hash_model_info(const ndf_hash_model* m, int* passes, double* last_loss,
                               double* gen_seconds, double* train_seconds, int64_t* adam_steps) {
    if (!m) return NDF_ERR_ARG;
    if (passes) *passes = m->passes;
    if (last_loss) *last_loss = m->last_loss;
    if (gen_seconds) *gen_seconds = m->gen_seconds;
    if (train_seconds) *train_seconds = m->train_seconds;
    if (adam_steps) *adam_steps = m->t;
    return NDF_OK;
}

}  // extern "C"
