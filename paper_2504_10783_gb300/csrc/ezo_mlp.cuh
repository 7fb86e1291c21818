// Training of the learned surrogate: the operand images and the arguments of
// the kernels in ezo_mlp_gemm_tc.cu.
//
// An operand image holds rows of 64 BF16 values (one K-chunk) in the K-major
// 128-byte swizzled layout of the tensor cores (sw128, ezo_tc.cuh), so a
// range of its rows is one contiguous copy. Transposed operands (batch rows
// are the product's K) are [chunk of 64 batch rows][feature], weights
// [K-chunk][256 rows].
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

namespace ezo {

constexpr int kMlpChunk = 256 * 128;                 // bytes of a K-chunk of 256 rows
constexpr int kMlpWeights = 2 * 65536 + 256 * 64;    // hidden weights: W3, W2, W1 in a workspace
// flat parameter layout: W1 [256 x 64] | b1 | W2 [256 x 256] | b2 | W3 | b3 | w4 [256] | b4 [1]
constexpr long long kOffW1 = 0, kOffB1 = kOffW1 + 256 * 64, kOffW2 = kOffB1 + 256, kOffB2 = kOffW2 + 65536,
                    kOffW3 = kOffB2 + 256, kOffB3 = kOffW3 + 65536, kOffW4 = kOffB3 + 256, kOffB4 = kOffW4 + 256,
                    kNumParams = kOffB4 + 1;
constexpr int kOutPart = 258;    // partial sums of the output layer: dw4, db4, loss
constexpr int kOutBlocks = 256;  // of them at most

inline int mlp_splits(int rows) { return (rows + 127) / 128; }
inline int mlp_out_blocks(int rows) { return rows / 8 < kOutBlocks ? rows / 8 : kOutBlocks; }

struct ChainArgs {
  int rows;           // batch rows, a multiple of 64
  const float* q;     // configurations, value j of row i at q[j * ldq + i]
  long long ldq;
  int n;
  const float* t;     // targets
  const uint8_t *img, *timg;  // weight images
  const float *bias[3], *w4, *b4;
  uint8_t *Xt;        // transposed feature image, 64 features a chunk
  uint8_t* Ht[6];     // transposed images of H1, H2, H3, dZ3, dZ2, dZ1
  float* e;           // output minus target
  int* err;           // set when a bounded wait gave up
};
struct WgradArgs {
  const uint8_t *Xt, *H1t, *H2t, *H3t, *dZ1t, *dZ2t, *dZ3t;
  const float* e;
  int rows, splits, out_blocks;
  float* ws;    // [128 batch rows][kMlpWeights]
  float* part;  // [out_blocks][kOutPart]
  int* err;
};
struct UpdateArgs {
  const float* ws;
  int splits;
  const uint8_t *dZ1t, *dZ2t, *dZ3t;
  int rows;
  const float* part;
  int out_blocks;
  float *g, *loss;
  float lr;  // 0: gradients only
  float beta1, beta2, eps, c1, c2;
  float *p, *m, *v;
  uint8_t *img, *timg;  // weight images
};

cudaError_t mlp_chain(const ChainArgs& g, cudaStream_t s);
cudaError_t mlp_wgrad(const WgradArgs& g, cudaStream_t s);
cudaError_t mlp_update(const UpdateArgs& u, cudaStream_t s);
cudaError_t mlp_weight_images(const float* p, void* img, void* timg, cudaStream_t s);

}  // namespace ezo
