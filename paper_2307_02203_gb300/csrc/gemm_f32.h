// FP32 matrix products of the hash-grid network's training (gemm_f32.cu).  All
// matrices are row-major; every call is enqueued on stream s.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace ndf {

// A dense layer over `batch` independent weight sets (one, or one per encoder of a cross
// field): rows [i * rows, (i + 1) * rows) of the activations belong to weight set i, whose
// parameters start i * wstride floats after W and b.
struct DenseLayer {
    const float* W = nullptr;  // [cout][cin]
    const float* b = nullptr;  // [cout]
    int cin = 0, cout = 0;
    int64_t rows = 0;
    int batch = 1;
    int64_t wstride = 0;
};

// pre = X W^T + b; post = act(pre) when post is given (activation code as in act_f)
cudaError_t dense_forward(cudaStream_t s, const DenseLayer& L, const float* X, float* pre, float* post,
                          int act);

// The weight and bias gradients are sums over the rows: every chunk of rows writes a partial
// sum, and one kernel at the end adds the partials of all layers in a fixed order
// (deterministic).  GradSums holds the list of partials and their workspace.
constexpr int kGradSegs = 40;
constexpr int64_t kGradSplits = 64;   // most chunks of one layer
struct GradSeg {
    const float* part;  // [splits][n]
    float* dst;         // dst[i] += sum over the splits
    int64_t n;
    int splits;
};
struct GradSums {
    float* work = nullptr;
    int64_t cap = 0, used = 0;
    int64_t rows = 0;  // the batch that it was sized for
    int64_t max_splits = kGradSplits;
    GradSeg seg[kGradSegs];
    int count = 0;
    float* take(int64_t floats) {  // nullptr: flush first
        if (used + floats > cap) return nullptr;
        float* r = work + used;
        used += (floats + 3) & ~int64_t(3);
        return r;
    }
};
// chunks of a layer's rows: of at least 128 rows (eight slices, the length of a 128-wide
// data-gradient tile), at most max_splits of them
inline int64_t dense_grad_splits(int64_t rows, int64_t max_splits) {
    const int64_t s = (rows + 127) / 128;
    return s < 1 ? 1 : s > max_splits ? max_splits : s;
}
// workspace one layer needs for up to `rows` rows of each of its `batch` weight sets
int64_t dense_grad_floats(int64_t cin, int64_t cout, int64_t rows, int batch, int64_t max_splits);
// adds every listed partial to its destination and empties the list (counts one launch)
cudaError_t grad_sums_flush(cudaStream_t s, GradSums& g, uint64_t* launches);

// One launch: the weight and bias gradients' partials of the layer (dW, db += ...; gradients of
// weight set i at dW + i * wstride) and, when dX is given, the data gradient of its input
// columns [col0, cin): dX[rows][cin - col0] = (dY W)[.., col0..] (* act'(pre_in), the layer
// input's pre-activations [rows][cin], when given; col0 = 0 then).
cudaError_t dense_backward(cudaStream_t s, const DenseLayer& L, const float* X, const float* dY, float* dX,
                           int col0, const float* pre_in, int act, float* dW, float* db, GradSums& g,
                           uint64_t* launches);

}  // namespace ndf
