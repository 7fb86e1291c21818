// The grid over an obstacle set that the collision kernels look spheres up in
// (ObsGrid, ezo_device.cuh).
//
// One block of 64 threads per brick of 4 x 4 x 4 fine cells. The block first
// keeps the obstacles that can be the nearest to some point of the brick
// (lower bound of the distance over the brick at most the smallest upper
// bound), then each thread does the same for its cell from that list, so an
// obstacle is read once per brick and a cell looks at the few that are left:
// 1024 obstacles cost about as much as 64. Built once per obstacle set, in
// one launch.
#include "ezo_kernels_common.cuh"

namespace ezo {

namespace {

// Bounds of the surface distance of obstacle o over the box [lo, hi]: lower
// less the margin, upper plus it.
__device__ __forceinline__ void surface_bounds(const float (&lo)[3], const float (&hi)[3], float4 o, float margin,
                                               float& lower, float& upper) {
  const float c[3] = {o.x, o.y, o.z};
  float near2 = 0.f, far2 = 0.f;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float a = lo[k] - c[k], b = c[k] - hi[k];
    const float n = fmaxf(fmaxf(a, b), 0.f), f = fmaxf(-a, -b);
    near2 = fmaf(n, n, near2);
    far2 = fmaf(f, f, far2);
  }
  lower = sqrtf(near2) - o.w - margin;
  upper = sqrtf(far2) - o.w + margin;
}

__global__ void __launch_bounds__(64) k_grid_build(GridBuild g) {
  __shared__ uint16_t list[EZO_MAX_OBS];
  __shared__ int s_count;
  __shared__ float s_min[2];
  __shared__ int s_lb[64];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int sub = g.sub, stride = sub * kGridC;
  const int n_fine[3] = {sub * g.n[0], sub * g.n[1], sub * g.n[2]};
  const int b0[3] = {(int)blockIdx.x * 4, (int)blockIdx.y * 4, (int)blockIdx.z * 4};
  const float hf = sub == 2 ? 0.5f * g.h : g.h;
  float lo[3], hi[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    lo[k] = (float)(sub * g.k0[k] + b0[k]) * hf;
    hi[k] = (float)(sub * g.k0[k] + b0[k] + 4) * hf;
  }
  if (t == 0) s_count = 0;
  s_lb[t] = 255;
  float best = 3.0e38f;
  for (int j = t; j < g.n_obs; j += 64) {
    float l, u;
    surface_bounds(lo, hi, g.obs[j], g.margin, l, u);
    best = fminf(best, u);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) best = fminf(best, __shfl_xor_sync(0xffffffffu, best, o));
  if (lane == 0) s_min[warp] = best;
  __syncthreads();
  best = fminf(s_min[0], s_min[1]);
  for (int j0 = 0; j0 < g.n_obs; j0 += 64) {
    const int j = j0 + t;
    float l = 3.0e38f, u;
    if (j < g.n_obs) surface_bounds(lo, hi, g.obs[j], g.margin, l, u);
    const unsigned keep = __ballot_sync(0xffffffffu, l <= best);
    int at = 0;
    if (lane == 0 && keep) at = atomicAdd(&s_count, __popc(keep));
    at = __shfl_sync(0xffffffffu, at, 0);
    if (l <= best) list[at + __popc(keep & ((1u << lane) - 1u))] = (uint16_t)j;
  }
  __syncthreads();
  const int cnt = s_count;
  const int x = b0[0] + (t & 3), y = b0[1] + ((t >> 2) & 3), z = b0[2] + (t >> 4);
  const bool in = x < n_fine[0] && y < n_fine[1] && z < n_fine[2];
  if (in) {
    const int cell[3] = {x, y, z};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      lo[k] = (float)(sub * g.k0[k] + cell[k]) * hf;
      hi[k] = (float)(sub * g.k0[k] + cell[k] + 1) * hf;
    }
    float up = 3.0e38f, low = 3.0e38f;
    for (int i = 0; i < cnt; ++i) {
      float l, u;
      surface_bounds(lo, hi, __ldg(g.obs + list[i]), g.margin, l, u);
      up = fminf(up, u);
      low = fminf(low, l);
    }
    const int lb8 = (int)fminf(fmaxf(floorf(low / g.step), 0.f), 255.f);
    // the ids, the first kGridInline of them in the cell's word
    unsigned long long w = 0ull;
    int m = 0;
    for (int i = 0; i < cnt; ++i) {
      float l, u;
      surface_bounds(lo, hi, __ldg(g.obs + list[i]), g.margin, l, u);
      if (l <= up) {
        if (m < (int)kGridInline) w |= (unsigned long long)list[i] << (16 + 12 * m);
        ++m;
      }
    }
    unsigned kind = (unsigned)m;
    if (m > (int)kGridInline) {
      // the collision grid's cells farther from every obstacle than its edge
      // need no list: a sphere that large is tested against every obstacle
      kind = kGridAll;
      if (low <= g.far) {
        const unsigned off = atomicAdd(g.used, (unsigned)m);
        if (off + (unsigned)m <= g.ids_cap) {
          kind = kGridList;
          w = ((unsigned long long)off << 32) | ((unsigned long long)m << 16);
          int at = 0;
          for (int i = 0; i < cnt; ++i) {
            float l, u;
            surface_bounds(lo, hi, __ldg(g.obs + list[i]), g.margin, l, u);
            if (l <= up) g.ids[off + at++] = list[i];
          }
        }
      }
      if (kind == kGridAll) w = 0ull;
    }
    g.cell[(z * stride + y) * stride + x] = w | ((unsigned long long)kind << 8) | (unsigned long long)lb8;
    // the coarse cell's bound, at its first fine cell's place
    atomicMin(&s_lb[sub == 2 ? t & 0x2a : t], lb8);
  }
  __syncthreads();
  if (in && g.lb && (sub == 1 || (t & ~0x2a) == 0))
    g.lb[((z / sub) * kGridC + y / sub) * kGridC + x / sub] = (uint8_t)s_lb[t];
}

}  // namespace

cudaError_t launch_grid_build(const GridBuild& g, cudaStream_t s) {
  if (g.n_obs <= 0) return cudaSuccess;
  const dim3 grid((g.sub * g.n[0] + 3) / 4, (g.sub * g.n[1] + 3) / 4, (g.sub * g.n[2] + 3) / 4);
  k_grid_build<<<grid, 64, 0, s>>>(g);
  return cudaGetLastError();
}

}  // namespace ezo
