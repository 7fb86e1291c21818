// Learned signed-distance surrogate: a small MLP sd_hat(q) from the features
// [sin q_1 .. sin q_n, cos q_1 .. cos q_n] (zero-padded to F = 64) through
// three hidden layers of width H = 256 with SiLU to one output. Not part of
// the paper: it only orders and prefilters bisection candidates; every
// certification sample is still checked exactly.
//
// Weights are kept in FP32 (master, Adam moments) and as BF16 operand images
// that feed the tensor cores. Training runs on the kernels of
// ezo_mlp_gemm_tc.cu; inference runs the whole network in one tensor-core
// kernel (ezo_mlp_tc.cu) from the same weight image.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/ezo.h"
#include "ezo_engine.cuh"
#include "ezo_mlp.cuh"

namespace ezo {

// tensor-core forward pass (ezo_mlp_tc.cu)
size_t mlp_tc_image_bytes();
cudaError_t mlp_tc_forward(const float* q, long long ldq, int n, long long rows_cap, const int* m_dev,
                           const void* img, const float* b1, const float* b2, const float* b3, const float* w4,
                           const float* b4, float* y, int* err, cudaStream_t s);
cudaError_t mlp_tc_bisect(int n, long long rows_cap, const int* m_dev, const void* img, const float* b1,
                          const float* b2, const float* b3, const float* w4, const float* b4, const float* s_p32,
                          const float* s_d32, float* s_lo, float* s_hi, uint32_t* s_bits, int n_b, float margin,
                          int* err, cudaStream_t s);

constexpr int kF = 64;   // padded input features
constexpr int kH = 256;  // hidden width


// ------------------------------------------------------------ small kernels --
__global__ void k_clamp_labels(float* __restrict__ t, long long N, float lo, float hi) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x)
    t[i] = fminf(fmaxf(t[i], lo), hi);
}

// configuration i of a training set: uniform in the joint box from Philox
// (counter (i, j, 0x5355, seed word), key (seed low, seed high))
__global__ void k_uniform_q(float* __restrict__ q, long long N, int n, const float* __restrict__ lo,
                            const float* __restrict__ hi, uint32_t k0, uint32_t k1) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
    for (int j = 0; j < n; j += 4) {
      const u32x4 r = philox4x32_10(u32x4{(uint32_t)i, (uint32_t)(i >> 32), (uint32_t)j, 0x5355u}, k0, k1);
      const uint32_t w[4] = {r.x, r.y, r.z, r.w};
      for (int c = 0; c < 4 && j + c < n; ++c) q[(long long)(j + c) * N + i] = lo[j + c] + (hi[j + c] - lo[j + c]) * u01_co(w[c]);
    }
  }
}


}  // namespace ezo

// ------------------------------------------------------------------ host side --
namespace {

using namespace ezo;

template <typename T>
cudaError_t dal(T** p, size_t n) {
  return cudaMalloc((void**)p, std::max<size_t>(1, n) * sizeof(T));
}

}  // namespace

extern "C" int ezo_internal_robot_boxes(const ezo_robot* r);
extern "C" int ezo_internal_env_boxes(const ezo_env* e);
extern "C" int ezo_internal_sd_lane(const ezo_robot* r, const ezo_env* e, long long N);
extern "C" int ezo_internal_env_dev(const ezo_robot* r, const ezo_env* e, ezo::EnvDevFull* out);
extern "C" ezo::WideGrid ezo_internal_sd_grid(const ezo_env* e, long long N, cudaStream_t s);
extern "C" int ezo_internal_robot_prismatic(const ezo_robot* r);
extern "C" void ezo_internal_set_error(const char* msg);
extern "C" const ezo::RobotDev* ezo_internal_robot_dev(const ezo_robot* r, int* n, int* nsp_pad, double* q_lo,
                                                       double* q_hi);

struct ezo_surrogate {
  int n = 0;
  const ezo_robot* robot = nullptr;
  uint8_t* mem = nullptr;                                        // what follows, in one block
  float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;  // flat FP32
  long long step = 0;
  // weight images: the forward kernel's (and training's), and W2, W3 transposed
  uint8_t *wimg = nullptr, *wtimg = nullptr;
  int* tc_err = nullptr;
  float* loss = nullptr;
  // one block for a training batch of up to cap rows: operand images, the
  // outputs' errors, the partial sums of the gradients
  int cap = 0;
  uint8_t* train = nullptr;
};

namespace {

using namespace ezo;

int blocks_for(long long n, int t) { return (int)std::max<long long>(1, std::min<long long>((n + t - 1) / t, 4096)); }

// The training block's parts for `rows` batch rows.
struct TrainBufs {
  uint8_t *Xt, *H1t, *H2t, *H3t, *dZ1t, *dZ2t, *dZ3t;
  float *e, *part, *ws;
  size_t bytes;
};
TrainBufs train_bufs(uint8_t* base, int rows) {
  const size_t tiles = (rows + 127) / 128, op = tiles * 128 * 512;  // an operand of 256 features
  TrainBufs b{};
  size_t at = 0;
  auto take = [&](size_t n) {
    uint8_t* p = base + at;
    at += n;
    return p;
  };
  b.Xt = take(tiles * 128 * 128);
  for (uint8_t** p : {&b.H1t, &b.H2t, &b.H3t, &b.dZ1t, &b.dZ2t, &b.dZ3t}) *p = take(op);
  b.e = reinterpret_cast<float*>(take(tiles * 128 * sizeof(float)));
  b.ws = reinterpret_cast<float*>(take(tiles * kMlpWeights * sizeof(float)));
  b.part = reinterpret_cast<float*>(take(sizeof(float) * kOutBlocks * kOutPart));
  b.bytes = at;
  return b;
}

cudaError_t ensure_train_cap(ezo_surrogate* S, int B, cudaStream_t s) {
  if (B <= S->cap) return cudaSuccess;
  cudaFree(S->train);
  S->train = nullptr;
  S->cap = 0;
  const TrainBufs b = train_bufs(nullptr, B);
  cudaError_t e = dal(&S->train, b.bytes);
  // the transposed feature image comes first; its padding features stay zero
  if (e == cudaSuccess) e = cudaMemsetAsync(S->train, 0, (size_t)(B + 127) / 128 * 128 * 128, s);
  if (e == cudaSuccess) S->cap = B;
  return e;
}

// One batch (q: n x B, stride ldq; t: B targets): gradients into S->g, the
// loss into S->loss and, for lr > 0, the Adam step of all parameters.
cudaError_t train_step(ezo_surrogate* S, const float* q, long long ldq, const float* t, int B, float lr,
                       cudaStream_t s) {
  cudaError_t e = ensure_train_cap(S, B, s);
  if (e != cudaSuccess) return e;
  const TrainBufs b = train_bufs(S->train, S->cap);
  const ChainArgs c{B, q, ldq, S->n, t, S->wimg, S->wtimg, {S->p + kOffB1, S->p + kOffB2, S->p + kOffB3},
                    S->p + kOffW4, S->p + kOffB4, b.Xt, {b.H1t, b.H2t, b.H3t, b.dZ3t, b.dZ2t, b.dZ1t}, b.e, S->tc_err};
  if ((e = mlp_chain(c, s)) != cudaSuccess) return e;
  const WgradArgs w{b.Xt, b.H1t, b.H2t, b.H3t, b.dZ1t, b.dZ2t, b.dZ3t, b.e, B, mlp_splits(B), mlp_out_blocks(B),
                    b.ws, b.part, S->tc_err};
  if ((e = mlp_wgrad(w, s)) != cudaSuccess) return e;
  UpdateArgs u{};
  u.ws = b.ws; u.splits = w.splits;
  u.dZ1t = b.dZ1t; u.dZ2t = b.dZ2t; u.dZ3t = b.dZ3t;
  u.rows = B;
  u.part = b.part; u.out_blocks = w.out_blocks;
  u.g = S->g; u.loss = S->loss;
  u.p = S->p; u.m = S->m; u.v = S->v;
  u.img = S->wimg; u.timg = S->wtimg;
  if (lr > 0.f) {
    S->step += 1;
    u.lr = lr; u.beta1 = 0.9f; u.beta2 = 0.999f; u.eps = 1e-8f;
    u.c1 = 1.f - std::pow(u.beta1, (float)S->step);
    u.c2 = 1.f - std::pow(u.beta2, (float)S->step);
  }
  return mlp_update(u, s);
}

}  // namespace

// n_b surrogate bisection steps on the brackets of the rows below the device
// count *m_dev, in one tensor-core launch. Internal.
extern "C" __attribute__((visibility("hidden"))) cudaError_t ezo_internal_mlp_bisect(
    ezo_surrogate* S, long long rows_cap, const int* m_dev, const float* s_p32, const float* s_d32, float* s_lo,
    float* s_hi, uint32_t* s_bits, int n_b, float margin, cudaStream_t s) {
  return mlp_tc_bisect(S->n, rows_cap, m_dev, S->wimg, S->p + kOffB1, S->p + kOffB2, S->p + kOffB3, S->p + kOffW4,
                       S->p + kOffB4, s_p32, s_d32, s_lo, s_hi, s_bits, n_b, margin, S->tc_err, s);
}

extern "C" __attribute__((visibility("hidden"))) int ezo_internal_surrogate_dof(const ezo_surrogate* S) {
  return S ? S->n : 0;
}

extern "C" {

int64_t ezo_surrogate_num_params(void) { return kNumParams; }

ezo_status ezo_surrogate_create(const ezo_robot* robot, uint64_t seed, ezo_surrogate** out) {
  if (!robot || !out) {
    ezo_internal_set_error("ezo_surrogate_create: null argument");
    return EZO_ERR_INVALID_ARG;
  }
  int n = 0, nsp = 0;
  double lo[EZO_MAX_DOF], hi[EZO_MAX_DOF];
  ezo_internal_robot_dev(robot, &n, &nsp, lo, hi);
  if (2 * n > kF) {
    ezo_internal_set_error("ezo_surrogate_create: 2 n features must fit in 64");
    return EZO_ERR_INVALID_ARG;
  }
  if (ezo_internal_robot_prismatic(robot)) {
    // the features sin q, cos q identify revolute joint angles only
    ezo_internal_set_error("ezo_surrogate_create: prismatic joints are not supported by the [sin q, cos q] features");
    return EZO_ERR_INVALID_ARG;
  }
  ezo_surrogate* S = new ezo_surrogate();
  S->n = n;
  S->robot = robot;
  // one block: the weight images, then the flat FP32 vectors, the loss and
  // the error flag
  const size_t vec = ((size_t)kNumParams + 63) / 64 * 64 * sizeof(float), img = mlp_tc_image_bytes(),
               timg = (size_t)8 * kMlpChunk;
  cudaError_t e = dal(&S->mem, img + timg + 4 * vec + 256);
  if (e == cudaSuccess) e = cudaMemset(S->mem + img + timg, 0, 4 * vec + 256);
  S->wimg = S->mem;
  S->wtimg = S->mem + img;
  S->p = reinterpret_cast<float*>(S->mem + img + timg);
  S->g = S->p + vec / sizeof(float);
  S->m = S->g + vec / sizeof(float);
  S->v = S->m + vec / sizeof(float);
  S->loss = S->v + vec / sizeof(float);
  S->tc_err = reinterpret_cast<int*>(S->loss + 32);
  if (e != cudaSuccess) {
    ezo_surrogate_free(S);
    ezo_internal_set_error((std::string("ezo_surrogate_create: ") + cudaGetErrorString(e)).c_str());
    return EZO_ERR_CUDA;
  }
  // uniform(-1/sqrt(fan_in), 1/sqrt(fan_in)) weights and biases from a
  // 64-bit LCG (Knuth's MMIX constants), so the start is reproducible
  std::vector<float> h(kNumParams);
  uint64_t st = seed * 6364136223846793005ull + 1442695040888963407ull;
  auto uni = [&]() {
    st = st * 6364136223846793005ull + 1442695040888963407ull;
    return (float)((st >> 40) * (1.0 / 16777216.0));
  };
  auto fill = [&](long long off, long long cnt, int fan_in) {
    const float a = 1.f / std::sqrt((float)fan_in);
    for (long long i = 0; i < cnt; ++i) h[off + i] = (2.f * uni() - 1.f) * a;
  };
  fill(kOffW1, (long long)kH * kF, 2 * n);
  fill(kOffB1, kH, 2 * n);
  for (long long i = 0; i < kH; ++i)
    for (int c = 2 * n; c < kF; ++c) h[kOffW1 + i * kF + c] = 0.f;  // padding features carry no weight
  fill(kOffW2, (long long)kH * kH, kH);
  fill(kOffB2, kH, kH);
  fill(kOffW3, (long long)kH * kH, kH);
  fill(kOffB3, kH, kH);
  fill(kOffW4, kH, kH);
  h[kOffB4] = 0.f;
  cudaMemcpy(S->p, h.data(), sizeof(float) * kNumParams, cudaMemcpyHostToDevice);
  mlp_weight_images(S->p, S->wimg, S->wtimg, nullptr);
  e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    ezo_surrogate_free(S);
    ezo_internal_set_error((std::string("ezo_surrogate_create: ") + cudaGetErrorString(e)).c_str());
    return EZO_ERR_CUDA;
  }
  *out = S;
  return EZO_OK;
}

void ezo_surrogate_free(ezo_surrogate* S) {
  if (!S) return;
  cudaFree(S->mem);
  cudaFree(S->train);
  delete S;
}

ezo_status ezo_surrogate_get_params(const ezo_surrogate* S, float* out) {
  if (!S || !out) return EZO_ERR_INVALID_ARG;
  if (cudaMemcpy(out, S->p, sizeof(float) * kNumParams, cudaMemcpyDeviceToHost) != cudaSuccess) return EZO_ERR_CUDA;
  return EZO_OK;
}

ezo_status ezo_surrogate_set_params(ezo_surrogate* S, const float* in) {
  if (!S || !in) return EZO_ERR_INVALID_ARG;
  if (cudaMemcpy(S->p, in, sizeof(float) * kNumParams, cudaMemcpyHostToDevice) != cudaSuccess) return EZO_ERR_CUDA;
  mlp_weight_images(S->p, S->wimg, S->wtimg, nullptr);
  return cudaDeviceSynchronize() == cudaSuccess ? EZO_OK : EZO_ERR_CUDA;
}

ezo_status ezo_surrogate_grad(ezo_surrogate* S, const float* q_dev, int64_t ldq, const float* t_dev, int32_t N,
                              float* grad, float* loss, void* stream) {
  if (!S || !q_dev || !t_dev || N < 64 || N % 64 || ldq < N) {
    ezo_internal_set_error("ezo_surrogate_grad: need N a positive multiple of 64 and ldq >= N");
    return EZO_ERR_INVALID_ARG;
  }
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e = train_step(S, q_dev, ldq, t_dev, N, 0.f, s);
  if (e == cudaSuccess && grad) e = cudaMemcpyAsync(grad, S->g, sizeof(float) * kNumParams, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess && loss) e = cudaMemcpyAsync(loss, S->loss, sizeof(float), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    ezo_internal_set_error((std::string("ezo_surrogate_grad: ") + cudaGetErrorString(e)).c_str());
    return EZO_ERR_CUDA;
  }
  return EZO_OK;
}

ezo_status ezo_surrogate_predict(ezo_surrogate* S, const float* q_dev, int64_t ldq, int64_t N, float* out_dev,
                                 void* stream) {
  if (!S || (N > 0 && (!q_dev || !out_dev)) || N < 0 || ldq < N) {
    ezo_internal_set_error("ezo_surrogate_predict: bad argument");
    return EZO_ERR_INVALID_ARG;
  }
  if (N == 0) return EZO_OK;
  cudaStream_t s = (cudaStream_t)stream;
  // features computed inside the forward kernel from the configurations
  mlp_tc_forward(q_dev, ldq, S->n, N, nullptr, S->wimg, S->p + kOffB1, S->p + kOffB2, S->p + kOffB3, S->p + kOffW4, S->p + kOffB4,
                 out_dev, S->tc_err, s);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    ezo_internal_set_error((std::string("ezo_surrogate_predict: ") + cudaGetErrorString(e)).c_str());
    return EZO_ERR_CUDA;
  }
  return EZO_OK;
}

ezo_status ezo_surrogate_status(ezo_surrogate* S, int32_t* timed_out, int32_t reset, void* stream) {
  if (!S || !timed_out) {
    ezo_internal_set_error("ezo_surrogate_status: null argument");
    return EZO_ERR_INVALID_ARG;
  }
  cudaStream_t s = (cudaStream_t)stream;
  int v = 0;
  cudaError_t e = cudaMemcpyAsync(&v, S->tc_err, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess && reset) e = cudaMemsetAsync(S->tc_err, 0, sizeof(int), s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    ezo_internal_set_error((std::string("ezo_surrogate_status: ") + cudaGetErrorString(e)).c_str());
    return EZO_ERR_CUDA;
  }
  *timed_out = v != 0 ? 1 : 0;
  ezo_internal_set_error("");
  return EZO_OK;
}

ezo_status ezo_surrogate_train(ezo_surrogate* S, const ezo_env* env, int64_t n_samples, int32_t epochs, int32_t batch,
                               float lr, uint64_t data_seed, float label_lo, float label_hi, float* epoch_loss,
                               void* stream) {
  if (!S || !env || n_samples < batch || batch < 64 || batch % 64 || epochs < 1 || !(lr > 0.f)) {
    ezo_internal_set_error("ezo_surrogate_train: need batch a multiple of 64, n_samples >= batch, epochs >= 1");
    return EZO_ERR_INVALID_ARG;
  }
  if (ezo_internal_robot_boxes(S->robot) || ezo_internal_env_boxes(env)) {
    // the labels come from the sphere signed-distance kernel
    ezo_internal_set_error("ezo_surrogate_train: sphere geometries only (the robot or env has boxes)");
    return EZO_ERR_INVALID_ARG;
  }
  cudaStream_t s = (cudaStream_t)stream;
  int n = 0, nsp = 0;
  double lo[EZO_MAX_DOF], hi[EZO_MAX_DOF];
  const RobotDev* rd = ezo_internal_robot_dev(S->robot, &n, &nsp, lo, hi);
  EnvDevFull ef{};
  ezo_internal_env_dev(S->robot, env, &ef);
  const long long N = n_samples / batch * batch;
  const int lane = ezo_internal_sd_lane(S->robot, env, N);
  // one block: the configurations, their labels, the joint limits
  float* q = nullptr;
  cudaError_t e = dal(&q, (size_t)(n + 1) * N + 2 * EZO_MAX_DOF);
  float *t = q + (size_t)n * N, *bnd = t + N;
  if (e == cudaSuccess) {
    float hb[2 * EZO_MAX_DOF];
    for (int j = 0; j < n; ++j) {
      hb[j] = (float)lo[j];
      hb[EZO_MAX_DOF + j] = (float)hi[j];
    }
    cudaMemcpyAsync(bnd, hb, sizeof(hb), cudaMemcpyHostToDevice, s);
    // training set: uniform configurations labelled by the exact FP32
    // signed distance, clamped to [label_lo, label_hi]
    k_uniform_q<<<blocks_for(N, 256), 256, 0, s>>>(q, N, n, bnd, bnd + EZO_MAX_DOF, (uint32_t)data_seed,
                                                     (uint32_t)(data_seed >> 32));
    e = launch_sd_flat(rd, n, nsp, lane, ef.e, lane >= 0 ? ezo_internal_sd_grid(env, N, s) : WideGrid{}, q, N, N, t, s, label_hi);
    k_clamp_labels<<<blocks_for(N, 256), 256, 0, s>>>(t, N, label_lo, label_hi);
  }
  for (int ep = 0; ep < epochs && e == cudaSuccess; ++ep) {
    float sum = 0.f;
    const long long steps = N / batch;
    for (long long st = 0; st < steps && e == cudaSuccess; ++st) {
      e = train_step(S, q + st * batch, N, t + st * batch, batch, lr, s);
      if (epoch_loss && e == cudaSuccess && (st % 64 == 63 || st == steps - 1)) {
        float l = 0.f;
        cudaMemcpyAsync(&l, S->loss, sizeof(float), cudaMemcpyDeviceToHost, s);
        cudaStreamSynchronize(s);
        sum = l;  // loss of the latest batch
      }
    }
    if (epoch_loss) epoch_loss[ep] = sum;
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFree(q);
  if (e != cudaSuccess) {
    ezo_internal_set_error((std::string("ezo_surrogate_train: ") + cudaGetErrorString(e)).c_str());
    return EZO_ERR_CUDA;
  }
  return EZO_OK;
}

}  // extern "C"
