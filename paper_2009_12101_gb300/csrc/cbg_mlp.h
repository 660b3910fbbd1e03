// cbg_mlp.h -- shape and parameter layout of the learned preconditioner's per-row network
// (7 stencil features -> 64 -> 64 -> 7, ReLU), shared by its host code and its kernels.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "cbg_tc.cuh"

namespace cbg {

constexpr int NIN = 7, NH = 64, NOUT = 7;
// parameters, row-major (out x in): W1[64][7], b1[64], W2[64][64], b2[64], W3[7][64], b3[7]
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + NH * NIN, OFF_W2 = OFF_B1 + NH, OFF_B2 = OFF_W2 + NH * NH,
              OFF_W3 = OFF_B2 + NH, OFF_B3 = OFF_W3 + NOUT * NH, NPARAM = OFF_B3 + NOUT;   // 5127
constexpr int MLP_ROWS = 128;   // rows per tile of the tensor-core kernel (one per tensor-memory lane)

constexpr int MLP_PARTS = 3;    // warpgroups of a CTA (tiles in flight)

// entry (k, l), k <= l, of a symmetric 7 x 7 matrix stored as 28 values
__host__ __device__ constexpr int spai_sym(int k, int l) { return k * 7 - k * (k - 1) / 2 + (l - k); }

// The weights as the network kernel reads them, in bytes: the five BF16 operands in their
// K-major swizzled layouts (unused places zero), then the biases b1[64], b2[64], b3[7] in FP32.
// Written once per change of the weights, so that a CTA only copies it.
constexpr int IMG_W1 = 0;                              // [64 o][K 0-15: W1 row, copy at K 8] B of layer 1
constexpr int IMG_W3T = IMG_W1;                        // [64 o][K 16-31: W3 column, copy at K 24] B of dH2
constexpr int IMG_W2 = IMG_W1 + 64 * TC_ROWB;          // [64 o][64 q]                 B of layer 2
constexpr int IMG_W2T = IMG_W2 + 64 * TC_ROWB;         // [64 q][64 o]                 B of dH1
constexpr int IMG_W3 = IMG_W2T + 64 * TC_ROWB;         // [16 k][64 o] (rows 7-15 zero) B of layer 3
constexpr int MLP_IMAGE_OPS = IMG_W3 + 16 * TC_ROWB;
constexpr int MLP_IMAGE = MLP_IMAGE_OPS + (2 * NH + 16) * 4;

// parameter idx, rounded to BF16, into its places of the image
__device__ __forceinline__ void mlp_pack(unsigned char* img, int idx, float w)
{
    const __nv_bfloat16 b = __float2bfloat16_rn(w);
    auto put = [&](int at, int m, int k) {
        *reinterpret_cast<__nv_bfloat16*>(img + at + tc_swz(m, k >> 3) + (k & 7) * 2) = b;
    };
    float* bias = reinterpret_cast<float*>(img + MLP_IMAGE_OPS);
    if (idx < OFF_B1) {
        put(IMG_W1, idx / NIN, idx % NIN);
        put(IMG_W1, idx / NIN, 8 + idx % NIN);
    } else if (idx < OFF_W2) {
        bias[idx - OFF_B1] = __bfloat162float(b);
    } else if (idx < OFF_B2) {
        const int q = idx - OFF_W2;
        put(IMG_W2, q / NH, q % NH);
        put(IMG_W2T, q % NH, q / NH);
    } else if (idx < OFF_W3) {
        bias[NH + idx - OFF_B2] = __bfloat162float(b);
    } else if (idx < OFF_B3) {
        const int q = idx - OFF_W3;
        put(IMG_W3, q / NH, q % NH);
        put(IMG_W3T, q % NH, 16 + q / NH);
        put(IMG_W3T, q % NH, 24 + q / NH);
    } else {
        bias[2 * NH + idx - OFF_B3] = __bfloat162float(b);
    }
}

// What one launch of the tensor-core network kernel computes.
enum MlpMode { MLP_FWD = 0, MLP_BWD = 1, MLP_TRAIN = 2 };

struct MlpArgs {
    long long n;                  // rows
    const float* feat;            // n x 7 features (16-byte aligned)
    const unsigned char* image;   // [MLP_IMAGE] the weights (mlp_pack), 16-byte aligned
    float* out;                   // MLP_FWD: n x 7 outputs
    const float* gout;            // MLP_BWD: n x 7, dL/dout (16-byte aligned)
    // MLP_TRAIN: per-row statistics of the (r, e) pairs, one array of `stride` rows per entry:
    // G (28 entries, spai_sym), c (7), d; 1 / a_ii in FP32; the pattern mask
    const float* G;
    const float* c;
    const float* d;
    const float* idiag;
    const unsigned char* mask;
    long long stride;
    double inv_npairs;
    float* gpart;                 // MLP_BWD / MLP_TRAIN: [gridDim.x][NPARAM] gradient partials
    double* lpart;                // MLP_TRAIN: [gridDim.x] loss partials
    int* fault;                   // set when a wait on the tensor core ran out (may be null)
};

// Launch the tensor-core network kernel (one CTA per SM at most).
cudaError_t mlp_tc_launch(int mode, int grid, cudaStream_t s, const MlpArgs& a);
int mlp_tc_grid(long long n);

}  // namespace cbg
