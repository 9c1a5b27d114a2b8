// Training kernels of the learned warm start (tpf_mlp_train.cu).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>

#include "tpf_internal.h"

namespace tpf {

constexpr int kTrainN = 32;       // batch columns (or inputs) per tile of the products
constexpr int kWgradMax = 8;      // layers per launch of the weight gradients
constexpr int kTrainLayers = 17;  // weight layers at most (tpf_mlp_create's limit)

// One layer's product D[unit m][column b] and what becomes of it.
struct LayerArgs {
    CUtensorMap a, b;  // weights [M][K] in 128 x 64 boxes, columns [B][K] in kTrainN x 64 boxes
    int chunks;        // K / 64
    int M, B, real;    // padded units, columns of the batch, units
    const float *bias;
    float *Z;                  // [B][M] pre-activations (written forward, read backward)
    __nv_bfloat16 *o, *oT;     // [B][M] and [M][B]
    // output layer: the targets (Re V - 1, Im V), z-scored
    const double2 *V;
    int n;
    const float *mean, *sd;
    double *loss;
    int *err;
};
enum LayerKind : int { kHidden = 0, kOutput = 1, kBackward = 2 };
tpf_status launch_layer(int kind, const LayerArgs &g, cudaStream_t st);

// Weight and bias gradients of up to kWgradMax layers.
struct WgradArgs {
    CUtensorMap a[kWgradMax], b[kWgradMax];  // dZ^T [Po][B] in 128 x 64, inputs^T [Pi][B] in kTrainN x 64 boxes
    int first[kWgradMax + 1];                // first tile of each layer
    int m_tiles[kWgradMax];
    float *D[kWgradMax];                     // [Pi][Po]
    int ld[kWgradMax];                       // Po
    const __nv_bfloat16 *zT[kWgradMax];      // dZ^T again
    float *gb[kWgradMax];
    int layers, chunks;                      // chunks: B / 64
    int *err;
};
tpf_status launch_wgrad(const WgradArgs &g, cudaStream_t st);

// Adam on every layer, or (update == 0) only the BF16 copies W and W^T of the master weights.
struct AdamLayer {
    float *W, *m, *v, *b, *mb, *vb;
    const float *gWT, *gb;  // gradients [Pi][Po], [Po]
    __nv_bfloat16 *Wb, *WTb;
    int Po, Pi, ro, ri, tile0;
};
struct AdamArgs {
    AdamLayer l[kTrainLayers];
    int L, update;
    float lr, b1, b2, eps, c1, c2;
};
tpf_status launch_adam(AdamArgs &g, cudaStream_t st);

// Features of B columns in both layouts, X [B][P] and X^T [P][B], BF16; clears the error flag and the loss.
tpf_status launch_train_features(const double2 *S, int B, int n, int P, const float *mean, const float *sd,
                                 __nv_bfloat16 *X, __nv_bfloat16 *XT, int *err, double *loss, cudaStream_t st);

// Parameters or gradients of every layer to or from a flat array: per layer
// W [out][in], then b [out].
struct FlatLayer {
    float *W, *b;  // masters
    const float *gWT, *gb;
    int Po, Pi, ro, ri;
    int64_t off;
};
struct FlatArgs {
    FlatLayer l[kTrainLayers];
    int L;
    int64_t total;
    float *flat;
    int mode;  // 0: masters -> flat, 1: flat -> masters, 2: gradients -> flat
};
tpf_status launch_flat(const FlatArgs &g, cudaStream_t st);

}  // namespace tpf
