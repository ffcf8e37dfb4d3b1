// Neural dependence field volume decoding (Sec. 5) on the 5th-generation tensor
// cores, R references per launch.
//
// For reference r and query vertex v the network computes
//   x  = [f(p_r) * f(v) ; f(p_r) + f(v)]          (the merge, rounded to BF16)
//   h1 = ReLU(W1 x + b1), h2 = ReLU(W2 h1 + b2), h3 = ReLU(W3 h2 + b3),
//   y  = act(w4 . h3 + b4)
// -- the arithmetic of the training forward.  The reference enters only through
// the layer-1 operand x, so W1, W2 and W3 are the same for every reference and
// stay in shared memory for the launch, and the query encoding f(v) (the grid
// gathers, most of a vertex's cost) is computed once per vertex for all R
// references of the launch.
//
// A persistent CTA per SM decodes 128-vertex tiles (the MMA M dimension) in two
// slots so that one slot's epilogue overlaps the other slot's MMAs:
//   warps 0-7 (slot 0) and 8-15 (slot 1): thread i of a slot's two halves owns row i of the
//     tile (TMEM lane i) and 64 of its columns.  The halves encode the vertex once per tile
//     (two levels each; 64 FP32 features in shared memory); then for each reference, after
//     each layer, they load their columns of the FP32 accumulator with tcgen05.ld, add the
//     bias, round, apply ReLU and write the next layer's operand (after layer 3 the columns stay as BF16
//     pairs in registers).  All other work sits where the slot would wait for an MMA: the
//     output layer's dot product under the next reference's layer 1, its halves' exchange and
//     the output function under layer 2, and the reference after that one's x (one half the
//     products, the other the sums; an operand of its own) under layer 3.
//   warp 16: allocates TMEM; one lane issues tcgen05.mma (M = 128, N = 128, K = 128) for
//     whichever slot is ready and commits to that slot's mbarrier.
// The A operands live in TMEM (two times 64 columns of BF16 pairs per slot, x and h, beside its
// 128 accumulator columns), not in shared memory: a layer's operand write and read would each be
// 32 KB of shared-memory bandwidth (256 cycles) on top of the weights' 32 KB.  What bounds the
// kernel is the chain of a slot (MMA of 512 cycles, commit, epilogue, MMA) with two slots per SM,
// so what counts is what stands between a commit and the next hand-over (with x, dot product and
// output there too it was 2,900 cycles after layer 3, and 3,800 per layer with one warp per 128
// columns and operands in shared memory).  16 references on 1.76M vertices: 4.29 ms before,
// 2.90 ms now (3.66 with the biases in shared memory; with the biases as a ninth K step of
// three BF16 terms each 2.83 ms, but the sums before the rounding to BF16 are then added in another
// order.)
// The references' features f(p_r) (FP32) sit in shared memory, the biases in constant memory.
#include <cuda_bf16.h>

#include <map>
#include <mutex>
#include <vector>

#include "ndf_net.h"
#include "tc_common.cuh"

namespace ndf {

namespace {

using namespace tc;

constexpr int kTile = 128;
constexpr int kEpiWarps = 16;
constexpr int kTcThreads = 32 * kEpiWarps + 32;  // + 1 MMA warp

struct TcGrid {
    const __nv_bfloat16* grid;
    int res[kLevels];
    int64_t off[kLevels];
};

// interpolated 16 features of one level at p (corner-aligned grid on [-1,1]^3)
__device__ __forceinline__ void encode_level(const TcGrid& G, int l, const float* p, float (&o)[kFeat]) {
    const int R = G.res[l];
    int i[3];
    float f[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        float u = (p[a] + 1.0f) * 0.5f * (float)(R - 1);
        int k = (int)floorf(u);
        k = k < 0 ? 0 : (k > R - 2 ? R - 2 : k);
        i[a] = k;
        f[a] = u - (float)k;
    }
#pragma unroll
    for (int q = 0; q < kFeat; ++q) o[q] = 0.0f;
    const uint4* base = reinterpret_cast<const uint4*>(G.grid + G.off[l]);
    uint4 g[8][2];
#pragma unroll
    for (int c = 0; c < 8; ++c) {  // all 16 loads first, then the weighted sums
        const int dx = c & 1, dy = (c >> 1) & 1, dz = (c >> 2) & 1;
        const int64_t idx = ((int64_t)(i[2] + dz) * R + (i[1] + dy)) * R + (i[0] + dx);
        g[c][0] = __ldg(base + idx * 2);
        g[c][1] = __ldg(base + idx * 2 + 1);
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const int dx = c & 1, dy = (c >> 1) & 1, dz = (c >> 2) & 1;
        const float w = (dx ? f[0] : 1.0f - f[0]) * (dy ? f[1] : 1.0f - f[1]) * (dz ? f[2] : 1.0f - f[2]);
        const uint32_t uu[8] = {g[c][0].x, g[c][0].y, g[c][0].z, g[c][0].w,
                                g[c][1].x, g[c][1].y, g[c][1].z, g[c][1].w};
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float2 v = unbf2(uu[j]);
            o[2 * j] = fmaf(w, v.x, o[2 * j]);
            o[2 * j + 1] = fmaf(w, v.y, o[2 * j + 1]);
        }
    }
}

__device__ __forceinline__ float pos_axis(int64_t i, int64_t n) {
    return n > 1 ? -1.0f + 2.0f * (float)i / (float)(n - 1) : 0.0f;
}

}  // namespace

struct TcInferArgs {
    TcGrid G;
    const int64_t* refs;       // [R] reference vertices
    int R;
    const __nv_bfloat16* w;    // [3][128][128] W1..W3 ([out][in])
    const float* params;
    int64_t offb1, offb2, offb3, offw4, offb4;
    int64_t N, X, Y, Z;
    int measure;
    int slot;                  // of the model in c_net
    float* out;                // [R][N]
    unsigned* status;
};

// shared memory: W1, W2, W3 (2 atoms each), then biases / output weights (4 x 128 FP32), the
// output layer's halves, the references' features [R][64], the rows' features and the barriers
constexpr int kMaxRefsPerLaunch = 64;
constexpr uint32_t kOffW = 0, kOffVec = 6 * kAtom;
// TMEM columns: accumulators at 0 and 128, the slots' h at 256 and 320, their x at 384 and 448
constexpr uint32_t kTmemCols = 512, kTmemH = 256, kTmemX = 384;
constexpr uint32_t kOffPart = kOffVec + 4 * kHid * 4;  // [2 slots][128] output-layer halves
constexpr uint32_t kOffFr = kOffPart + 2 * 128 * 4;
constexpr uint32_t kOffFq = kOffFr + kMaxRefsPerLaunch * kLF * 4;  // [16][256 rows] float4
constexpr uint32_t kOffBar = kOffFq + 256 * kLF * 4;
constexpr uint32_t kTcSmem = kOffBar + 256 /*barriers*/ + 1024 /*align*/;

// Biases and output weights of up to kConstSlots live models in constant memory: an epilogue thread
// reads 64 of each per layer and reference, the same for its whole warp; from shared memory these
// broadcasts took 1,100 cycles of its pipe per tile and reference (of 4,900), beside the tensor
// cores' operand reads.  A model holds a slot from its creation to its end (one past the
// kConstSlots-th decodes from shared memory); the decoder refreshes it after a parameter update.
constexpr int kConstSlots = 16;
__constant__ ulonglong2 c_net[kConstSlots][kHid];  // b1, b2, b3, w4

// ---- encode / epilogue: slot s, row i = TMEM lane i, columns of half H
template <bool CB, int H>
__device__ __forceinline__ void decode_rows(const TcInferArgs& a, unsigned char* smem, uint32_t tmem, int64_t tiles,
                                            int64_t step, volatile int* abort_flag) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, s = warp >> 3, R = a.R;
    const float* vec = reinterpret_cast<const float*>(smem + kOffVec);
    float* part_s = reinterpret_cast<float*>(smem + kOffPart);
    const float* fr_all = reinterpret_cast<const float*>(smem + kOffFr);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kOffBar);
    uint64_t *a_ready = bars, *d_ready = bars + 2, *enc_ready = bars + 4, *part_ready = bars + 6;
    // four consecutive values of (b1, b2, b3, w4)
    auto vec4 = [&](int i) {
        return CB ? c_net[a.slot][i >> 2] : reinterpret_cast<const ulonglong2*>(vec)[i >> 2];
    };
    const int i = (warp & 3) * 32 + lane;
    const uint32_t tl = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t taddr = tl + (uint32_t)(s * 128 + H * 64);
    const uint32_t haddr = tl + kTmemH + (uint32_t)(s * 64 + H * 32);
    const uint32_t xaddr = tl + kTmemX + (uint32_t)(s * 64 + H * 32);
    const float b4 = a.params[a.offb4];
    // this row's query features, four per 16 bytes
    ulonglong2* fq = reinterpret_cast<ulonglong2*>(smem + kOffFq) + s * 128 + i;
    uint32_t nd = 0, ne = 0, np = 0;
    for (int64_t t = (int64_t)blockIdx.x * 2 + s; t < tiles; t += step) {
        const int64_t v = t * kTile + i;
        // this row's vertex, encoded once for every reference (rows past N encode
        // position 0: harmless, never written out)
        {
            const int64_t vv = v < a.N ? v : 0;
            const int64_t x = vv % a.X, y = (vv / a.X) % a.Y, z = vv / (a.X * a.Y);
            const float p[3] = {pos_axis(x, a.X), pos_axis(y, a.Y), pos_axis(z, a.Z)};
#pragma unroll 1
            for (int l = H * (kLevels / 2); l < (H + 1) * (kLevels / 2); ++l) {
                float f[kFeat];
                encode_level(a.G, l, p, f);
#pragma unroll
                for (int q = 0; q < kFeat / 4; ++q)
                    fq[(l * (kFeat / 4) + q) * 256] =
                        make_ulonglong2(pair2(f[4 * q], f[4 * q + 1]), pair2(f[4 * q + 2], f[4 * q + 3]));
            }
        }
        arrive_warp(&enc_ready[s]);
        if (!__all_sync(0xffffffffu, wait_bounded(&enc_ready[s], ne & 1u, abort_flag))) return;
        ++ne;
        // x = [fr * fq ; fr + fq]: operand columns 0-31 the products, 32-63 the sums
        auto put_x = [&](int r) {
            const ulonglong2* fr = reinterpret_cast<const ulonglong2*>(fr_all + r * kLF);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint32_t o[8];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const ulonglong2 f = fr[4 * c + j], q = fq[(4 * c + j) * 256];
                    if (H == 0) {
                        o[2 * j] = bf2(mul_pair(f.x, q.x));
                        o[2 * j + 1] = bf2(mul_pair(f.y, q.y));
                    } else {
                        o[2 * j] = bf2(add_pair(f.x, q.x));
                        o[2 * j + 1] = bf2(add_pair(f.y, q.y));
                    }
                }
                tmem_st8(xaddr + (uint32_t)(8 * c), o);
            }
            tmem_wait_st();
        };
        // 32 accumulator columns d of layer l, from this half's column 32 c on: + bias, rounded, ReLU
        auto hidden = [&](int l, int c, const uint32_t* d, uint32_t* o) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const ulonglong2 b = vec4(l * kHid + 64 * H + 32 * c + 4 * j);
                o[2 * j] = relu2(bf2(add_pair(pair2(d[4 * j], d[4 * j + 1]), b.x)));
                o[2 * j + 1] = relu2(bf2(add_pair(pair2(d[4 * j + 2], d[4 * j + 3]), b.y)));
            }
        };
        // the output of reference r from this half's sum of the output layer
        float sum = 0.0f;
        auto put_out = [&](int r) {
            if (H == 1) return true;
            if (!__all_sync(0xffffffffu, wait_bounded(&part_ready[s], np & 1u, abort_flag))) return false;
            ++np;
            const float o = (sum + part_s[s * 128 + i]) + b4;
            if (v < a.N)
                a.out[(int64_t)r * a.N + v] = a.measure == 0 ? tanhf(o) : (o > 20.f ? o : log1pf(expf(o)));
            return true;
        };
        put_x(0);
        tc_fence_before();
        arrive_warp(&a_ready[s]);
        for (int r = 0; r < R; ++r) {
#pragma unroll
            for (int layer = 0; layer < 2; ++layer) {
                if (!__all_sync(0xffffffffu, wait_bounded(&d_ready[s], nd & 1u, abort_flag))) return;
                ++nd;
                tc_fence_after();
                uint32_t d[64], o[16];
                tmem_ld64(taddr, d);
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    hidden(layer, c, d + 32 * c, o);
                    tmem_st16(haddr + (uint32_t)(16 * c), o);
                }
                tmem_wait_st();
                tc_fence_before();
                arrive_warp(&a_ready[s]);
                if (layer == 0) {
                    if (r > 0 && !put_out(r - 1)) return;
                } else if (r + 1 < R) {
                    put_x(r + 1);  // layer 1 of this reference, which read x, has completed
                }
            }
            if (!__all_sync(0xffffffffu, wait_bounded(&d_ready[s], nd & 1u, abort_flag))) return;
            ++nd;
            tc_fence_after();
            uint32_t h3[32];
            {
                uint32_t d[64];
                tmem_ld64(taddr, d);
                hidden(2, 0, d, h3);
                hidden(2, 1, d + 32, h3 + 16);
            }
            if (r + 1 < R) {  // x is in place and the accumulator read: the next reference's layer 1
                tc_fence_before();
                arrive_warp(&a_ready[s]);
            }
            uint64_t acc[4] = {0ull, 0ull, 0ull, 0ull};  // output layer on the BF16-rounded h3
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const ulonglong2 w = vec4(3 * kHid + 64 * H + 4 * j);
                const float2 u0 = unbf2(h3[2 * j]), u1 = unbf2(h3[2 * j + 1]);
                acc[2 * (j & 1)] = fma_pair(w.x, pair2(u0.x, u0.y), acc[2 * (j & 1)]);
                acc[2 * (j & 1) + 1] = fma_pair(w.y, pair2(u1.x, u1.y), acc[2 * (j & 1) + 1]);
            }
            const float2 s0 = unpair2(add_pair(add_pair(acc[0], acc[1]), add_pair(acc[2], acc[3])));
            sum = s0.x + s0.y;
            // the second half's sum meets the first half's here; it is rewritten only after the
            // next reference's three layers, to which the first half contributes after reading it
            if (H == 1) {
                part_s[s * 128 + i] = sum;
                arrive_warp(&part_ready[s]);
            }
        }
        if (!put_out(R - 1)) return;
    }
}

template <bool CB>
__global__ void __launch_bounds__(kTcThreads, 1) infer_tc_kernel(const TcInferArgs a) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    float* vec = reinterpret_cast<float*>(smem + kOffVec);  // b1, b2, b3, w4
    float* fr_all = reinterpret_cast<float*>(smem + kOffFr);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kOffBar);
    uint64_t* a_ready = bars;         // [2] epilogue -> MMA (8 warps)
    uint64_t* d_ready = bars + 2;     // [2] MMA -> epilogue (commit)
    uint64_t* enc_ready = bars + 4;   // [2] the tile's features are written (8 warps)
    uint64_t* part_ready = bars + 6;  // [2] the second half's output sums are written (4 warps)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 8);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int R = a.R;

    // ---- weights into the swizzled K-major layout (rows = output features),
    // biases and output weights, the references' features
    for (int i = threadIdx.x; i < 3 * kHid * 16; i += blockDim.x) {  // 3 layers x 128 rows x 16 chunks
        const int l = i / (kHid * 16), row = (i >> 4) % kHid, c = i & 15;
        const uint32_t o = (uint32_t)(2 * l + (c >> 3)) * kAtom + swz(row, c & 7);
        *reinterpret_cast<uint4*>(smem + kOffW + o) =
            reinterpret_cast<const uint4*>(a.w + ((size_t)l * kHid + row) * kHid)[c];
    }
    for (int i = threadIdx.x; i < 4 * kHid; i += blockDim.x) {
        const int64_t off = i < kHid ? a.offb1 : i < 2 * kHid ? a.offb2 : i < 3 * kHid ? a.offb3 : a.offw4;
        vec[i] = a.params[off + (i % kHid)];
    }
    for (int i = threadIdx.x; i < R * kLevels; i += blockDim.x) {
        const int64_t v = a.refs[i / kLevels];
        const int64_t x = v % a.X, y = (v / a.X) % a.Y, z = v / (a.X * a.Y);
        const float p[3] = {pos_axis(x, a.X), pos_axis(y, a.Y), pos_axis(z, a.Z)};
        float f[kFeat];
        encode_level(a.G, i % kLevels, p, f);
#pragma unroll
        for (int q = 0; q < kFeat; ++q) fr_all[(i / kLevels) * kLF + (i % kLevels) * kFeat + q] = f[q];
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(&a_ready[s], 8);
            mbar_init(&d_ready[s], 1);
            mbar_init(&enc_ready[s], 8);
            mbar_init(&part_ready[s], 4);
        }
        *abort_flag = 0;
    }
    if (warp == kEpiWarps) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tmem_slot)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    proxy_fence();  // weights written by threads are read by the tensor cores
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const int64_t tiles = (a.N + kTile - 1) / kTile;
    const int64_t step = (int64_t)gridDim.x * 2;
    // instruction descriptor: D FP32, A/B BF16, K-major, N = 128, M = 128
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kHid >> 3) << 17) |
                           ((uint32_t)(kTile >> 4) << 24);

    if (warp == kEpiWarps) {
        if (lane == 0) {  // ---- MMA issuer: serve whichever slot is ready
            // operands per slot: (its tiles) x R references x 3 layers
            int64_t left[2];
            for (int s = 0; s < 2; ++s) {
                const int64_t t0 = (int64_t)blockIdx.x * 2 + s;
                left[s] = t0 < tiles ? ((tiles - 1 - t0) / step + 1) * (int64_t)R * 3 : 0;
            }
            int layer[2] = {0, 0};
            uint32_t na[2] = {0, 0};
            const uint32_t sw = smem_u32(smem + kOffW);
            uint32_t polls = 0;
            uint64_t t0 = 0;
            while ((left[0] > 0 || left[1] > 0) && !*abort_flag) {
                bool progressed = false;
                for (int s = 0; s < 2; ++s) {
                    if (left[s] == 0 || !test_wait(&a_ready[s], na[s] & 1u)) continue;
                    progressed = true;
                    ++na[s];
                    tc_fence_after();
                    const uint32_t ta = tmem + (layer[s] == 0 ? kTmemX : kTmemH) + (uint32_t)(s * 64);
                    const uint32_t wl = sw + (uint32_t)(2 * layer[s]) * kAtom;
                    const uint32_t d = tmem + (uint32_t)(s * 128);
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk) {  // K = 128: two atoms, 4 steps of 16 each
                        const uint32_t at = (uint32_t)(kk >> 2) * kAtom;
                        tc_mma_ts(d, ta + (uint32_t)(kk * 8), desc_sw128(wl + at) + (uint64_t)((kk & 3) * 2), idesc,
                                  kk > 0 ? 1u : 0u);
                    }
                    tc_commit(&d_ready[s]);
                    layer[s] = layer[s] == 2 ? 0 : layer[s] + 1;
                    --left[s];
                }
                if (progressed) {
                    polls = 0;
                    t0 = 0;
                } else if (++polls > kWaitPolls) {
                    *abort_flag = 1;
                } else if ((polls & 1023u) == 0u) {  // and at most kWaitNs of wall time
                    const uint64_t t = global_ns();
                    if (t0 == 0) t0 = t;
                    else if (t - t0 > kWaitNs) *abort_flag = 1;
                }
            }
        }
    } else if (((warp >> 2) & 1) == 0) {
        decode_rows<CB, 0>(a, smem, tmem, tiles, step, abort_flag);
    } else {
        decode_rows<CB, 1>(a, smem, tmem, tiles, step, abort_flag);
    }
    if (*abort_flag && threadIdx.x == 0) report(a.status, kDevTimeout);
    tc_fence_before();
    __syncthreads();
    if (warp == kEpiWarps) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols)
                     : "memory");
    }
}

static std::mutex g_slot_mutex;
static std::map<int, std::vector<char>> g_slots;  // per device: slots in use

int const_slot_acquire(int device) {
    std::lock_guard<std::mutex> lock(g_slot_mutex);
    std::vector<char>& used = g_slots[device];
    used.resize(kConstSlots, 0);
    for (int i = 0; i < kConstSlots; ++i)
        if (!used[(size_t)i]) {
            used[(size_t)i] = 1;
            return i;
        }
    return -1;
}

void const_slot_release(int device, int slot) {
    if (slot < 0) return;
    std::lock_guard<std::mutex> lock(g_slot_mutex);
    g_slots[device][(size_t)slot] = 0;
}

cudaError_t launch_infer_tc(ndf_model* m, const int64_t* d_refs, int R, float* out) {
    ndf_ctx* ctx = m->ctx;
    // from 100,000 values on (40 us) the constant copy after a parameter update (2 us) is repaid by
    // its first call; a captured call reads the parameters themselves (its copy would not run now)
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(ctx->stream, &capture);
    if (e != cudaSuccess) return e;
    const bool constant = m->cslot >= 0 && capture == cudaStreamCaptureStatusNone &&
                          (double)R * (double)(m->X * m->Y * m->Z) >= 1e5;
    auto kern = constant ? infer_tc_kernel<true> : infer_tc_kernel<false>;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTcSmem);
    if (e != cudaSuccess) return e;
    if (constant && m->cslot_stale) {
        void* base = nullptr;
        e = cudaGetSymbolAddress(&base, c_net);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(static_cast<char*>(base) + (size_t)m->cslot * sizeof(c_net[0]), m->mlp_vec(),
                                sizeof(c_net[0]), cudaMemcpyDeviceToDevice, ctx->stream);
        if (e == cudaSuccess) e = cudaEventRecord(m->cslot_ready, ctx->stream);
        if (e != cudaSuccess) return e;
        m->cslot_stale = false;
    } else if (constant) {
        // the copy may have run on another stream, which this call need not follow
        e = cudaStreamWaitEvent(ctx->stream, m->cslot_ready, 0);
        if (e != cudaSuccess) return e;
    }
    TcInferArgs a;
    a.G.grid = m->grid_bf;
    for (int l = 0; l < kLevels; ++l) {
        a.G.res[l] = m->L.res[l];
        a.G.off[l] = m->L.grid_off[l];
    }
    a.w = m->wbf;
    a.params = m->params;
    a.offb1 = m->L.b1;
    a.offb2 = m->L.b2;
    a.offb3 = m->L.b3;
    a.offw4 = m->L.w4;
    a.offb4 = m->L.b4;
    a.N = m->X * m->Y * m->Z;
    a.X = m->X;
    a.Y = m->Y;
    a.Z = m->Z;
    a.measure = m->measure;
    a.slot = m->cslot;
    a.status = ctx->flag.as<unsigned>() + 1;
    const int64_t tiles = (a.N + kTile - 1) / kTile;
    int64_t grid = ctx->sm_count;  // one persistent CTA per SM, two tiles in flight each
    if (grid > (tiles + 1) / 2) grid = (tiles + 1) / 2;
    if (grid < 1) grid = 1;
    for (int r0 = 0; r0 < R; r0 += kMaxRefsPerLaunch) {
        a.refs = d_refs + r0;
        a.R = R - r0 < kMaxRefsPerLaunch ? R - r0 : kMaxRefsPerLaunch;
        a.out = out + (int64_t)r0 * a.N;
        kern<<<(unsigned)grid, kTcThreads, kTcSmem, ctx->stream>>>(a);
        ctx->launches++;
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace ndf
