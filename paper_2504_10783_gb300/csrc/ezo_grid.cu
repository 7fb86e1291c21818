// The grid over an obstacle set that the collision kernels look spheres up in
// (ObsGrid, ezo_device.cuh).
//
// One block per brick of 4 x 4 x 4 fine cells. The block first keeps the
// obstacles that can be the nearest to some point of the brick (lower bound of
// the distance over the brick at most the smallest upper bound), then four
// threads a cell do the same for the cell from that list, so an obstacle is
// read once per brick and a cell looks at the few that are left. Latency of
// the bricks with the longest lists bounds it (hundreds of obstacles above a
// dense layer): one thread a cell and an atomic a list took 12 us for 64
// spheres, 111 for 1024 on a table and 168 for 4096 where this takes 8, 57 and
// 106 (eight threads a cell: 9, 55, 113). Built once per obstacle set, in one
// launch.
#include "ezo_kernels_common.cuh"

namespace ezo {

namespace {

constexpr int kParts = 4;  // threads a cell
constexpr int kThreads = 64 * kParts;

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

__global__ void __launch_bounds__(kThreads) k_grid_build(GridBuild g) {
  __shared__ uint16_t list[EZO_MAX_OBS];
  __shared__ int s_count;
  __shared__ float s_min[kThreads / 32];
  __shared__ int s_lb[64];
  __shared__ float s_up[kParts][64], s_low[kParts][64];
  __shared__ int s_kept[kParts][64];
  __shared__ unsigned s_off[64];
  __shared__ unsigned long long s_word[64];
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
  if (t < 64) {
    s_lb[t] = 255;
    s_word[t] = 0ull;
  }
  float best = 3.0e38f;
  for (int j = t; j < g.n_obs; j += kThreads) {
    float l, u;
    surface_bounds(lo, hi, g.obs[j], g.margin, l, u);
    best = fminf(best, u);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) best = fminf(best, __shfl_xor_sync(0xffffffffu, best, o));
  if (lane == 0) s_min[warp] = best;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kThreads / 32; ++k) best = fminf(best, s_min[k]);
  for (int j0 = 0; j0 < g.n_obs; j0 += kThreads) {
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
  // thread (part, c): every kParts-th obstacle of the list for cell c
  const int part = t >> 6, c = t & 63;
  const int x = b0[0] + (c & 3), y = b0[1] + ((c >> 2) & 3), z = b0[2] + (c >> 4);
  const bool in = x < n_fine[0] && y < n_fine[1] && z < n_fine[2];
  const int cell[3] = {x, y, z};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    lo[k] = (float)(sub * g.k0[k] + cell[k]) * hf;
    hi[k] = (float)(sub * g.k0[k] + cell[k] + 1) * hf;
  }
  float up = 3.0e38f, low = 3.0e38f;
#pragma unroll 4
  for (int i = part; i < cnt; i += kParts) {
    float l, u;
    surface_bounds(lo, hi, __ldg(g.obs + list[i]), g.margin, l, u);
    up = fminf(up, u);
    low = fminf(low, l);
  }
  s_up[part][c] = up;
  s_low[part][c] = low;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kParts; ++k) {
    up = fminf(up, s_up[k][c]);
    low = fminf(low, s_low[k][c]);
  }
  int kept = 0;
#pragma unroll 4
  for (int i = part; i < cnt; i += kParts) {
    float l, u;
    surface_bounds(lo, hi, __ldg(g.obs + list[i]), g.margin, l, u);
    kept += l <= up ? 1 : 0;
  }
  s_kept[part][c] = kept;
  __syncthreads();
  int m = 0, at = 0;  // the cell's ids, and those of the parts before this one
#pragma unroll
  for (int k = 0; k < kParts; ++k) {
    at += k < part ? s_kept[k][c] : 0;
    m += s_kept[k][c];
  }
  // The first kGridInline ids go into the cell's word, more into a list; the
  // collision grid's cells farther from every obstacle than its edge need no
  // list: a sphere that large is tested against every obstacle.
  const bool listed = in && m > (int)kGridInline && low <= g.far;
  if (part == 0) {  // a warp takes its cells' room together
    int sum = listed ? m : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, sum, o);
      if (lane >= o) sum += v;
    }
    unsigned base = 0u;
    if (lane == 31 && sum) base = atomicAdd(g.used, (unsigned)sum);
    s_off[c] = __shfl_sync(0xffffffffu, base, 31) + (unsigned)(sum - (listed ? m : 0));
  }
  __syncthreads();
  const unsigned off = s_off[c];
  const bool fits = listed && off + (unsigned)m <= g.ids_cap;
  if (in && kept && (fits || m <= (int)kGridInline)) {
    for (int i = part; i < cnt; i += kParts) {
      float l, u;
      surface_bounds(lo, hi, __ldg(g.obs + list[i]), g.margin, l, u);
      if (!(l <= up)) continue;
      if (fits) g.ids[off + (unsigned)at] = list[i];
      else atomicOr(&s_word[c], (unsigned long long)list[i] << (16 + 12 * at));
      ++at;
    }
  }
  const int lb8 = (int)fminf(fmaxf(floorf(low / g.step), 0.f), 255.f);
  // the coarse cell's bound, at its first fine cell's place
  if (in && part == 0) atomicMin(&s_lb[sub == 2 ? c & 0x2a : c], lb8);
  __syncthreads();
  if (!in || part != 0) return;
  unsigned long long w = s_word[c];
  unsigned kind = (unsigned)m;
  if (m > (int)kGridInline) {
    kind = fits ? kGridList : kGridAll;
    w = fits ? ((unsigned long long)off << 32) | ((unsigned long long)m << 16) : 0ull;
  }
  g.cell[(z * stride + y) * stride + x] = w | ((unsigned long long)kind << 8) | (unsigned long long)lb8;
  if (g.lb && (sub == 1 || (c & ~0x2a) == 0))
    g.lb[((z / sub) * kGridC + y / sub) * kGridC + x / sub] = (uint8_t)s_lb[c];
}

}  // namespace

cudaError_t launch_grid_build(const GridBuild& g, cudaStream_t s) {
  if (g.n_obs <= 0) return cudaSuccess;
  const dim3 grid((g.sub * g.n[0] + 3) / 4, (g.sub * g.n[1] + 3) / 4, (g.sub * g.n[2] + 3) / 4);
  k_grid_build<<<grid, kThreads, 0, s>>>(g);
  return cudaGetLastError();
}

}  // namespace ezo
