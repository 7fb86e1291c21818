// Device-side building blocks of the EI-ZO hot path (sm_103a).
//
// * Philox4x32-10 counter-based generator (Salmon et al., SC'11), used by the
//   hit-and-run walks of Sec. IV-B / IV-D.
// * Forward kinematics of a standard DH chain in FP32 and the sphere
//   collision test (robot vs obstacle spheres and listed self pairs) that the
//   paper's GPU collision checker performs (Sec. IV-D, Sec. V-B).
//
// Collision test, per robot sphere i and obstacle j: the pair collides when
// |c_i - o_j|^2 < (r_i + R_j)^2, evaluated in FP32 differences. Which
// obstacles a sphere is tested against comes from a grid over the obstacle
// set (ObsGrid): per cell only those that can be the nearest to a point of
// the cell. Self pairs use a four-FMA form of the same test with a rounding
// bound, and the direct form inside the bound.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#define EZO_MAX_DOF 16
#define EZO_MAX_SPHERES 256
#define EZO_MAX_OBS 4096
#define EZO_CH 8
#define EZO_MAX_SBLK 32
#define EZO_MAX_BOX 32    // robot boxes
#define EZO_MAX_EBOX 64   // obstacle boxes per environment

namespace ezo {

// ------------------------------------------------------------------ Philox --
struct u32x4 {
  uint32_t x, y, z, w;
};

__device__ __forceinline__ u32x4 philox4x32_10(u32x4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    // each 32 x 32 -> 64-bit product gives both halves at once
    const uint64_t p0 = (uint64_t)0xD2511F53u * c.x, p1 = (uint64_t)0xCD9E8D57u * c.z;
    const uint32_t lo0 = (uint32_t)p0, hi0 = (uint32_t)(p0 >> 32);
    const uint32_t lo1 = (uint32_t)p1, hi1 = (uint32_t)(p1 >> 32);
    c = u32x4{hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0};
  }
  return c;
}

// The ten round keys of Philox4x32-10 for one seed: (k0 + r 0x9E3779B9,
// k1 + r 0xBB67AE85) for r = 0..9, computed on the host and passed in kernel
// parameters, so the rounds read them as constant operands.
struct PhiloxKeys {
  uint32_t k0[10], k1[10];
};

inline PhiloxKeys philox_keys(uint64_t seed) {
  PhiloxKeys ks;
  uint32_t a = (uint32_t)(seed & 0xffffffffu), b = (uint32_t)(seed >> 32);
  for (int r = 0; r < 10; ++r) {
    ks.k0[r] = a;
    ks.k1[r] = b;
    a += 0x9E3779B9u;
    b += 0xBB67AE85u;
  }
  return ks;
}

// philox4x32_10 with the round keys given (the same bits).
__device__ __forceinline__ u32x4 philox4x32_10(u32x4 c, const PhiloxKeys& ks) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint64_t p0 = (uint64_t)0xD2511F53u * c.x, p1 = (uint64_t)0xCD9E8D57u * c.z;
    const uint32_t lo0 = (uint32_t)p0, hi0 = (uint32_t)(p0 >> 32);
    const uint32_t lo1 = (uint32_t)p1, hi1 = (uint32_t)(p1 >> 32);
    c = u32x4{hi1 ^ c.y ^ ks.k0[r], lo1, hi0 ^ c.w ^ ks.k1[r], lo0};
  }
  return c;
}

// [0, 1): top 24 bits times 2^-24 (exact in FP32).
__device__ __forceinline__ float u01_co(uint32_t x) { return (float)(x >> 8) * 5.9604644775390625e-8f; }
// (0, 1]: (top 24 bits + 1) times 2^-24 (exact in FP32).
__device__ __forceinline__ float u01_oc(uint32_t x) { return (float)((x >> 8) + 1u) * 5.9604644775390625e-8f; }

// ------------------------------------------------------------------ robot --
// The robot as collide_lane walks it. axis[f] = 1, 2, 3 when every sphere of
// frame f lies on its x, y or z axis, else 0; slot[f] numbers the frames with
// spheres (-1: none), whose poses a group of lanes keeps: the axis and the
// origin, or three axes and the origin where some frame is general. The chain
// is walked to frame `last`, the last with spheres. The self pairs are a list
// of links, runs of spheres on one frame each (a0, na on frame fa; b0, nb on
// fb), every sphere of one against every sphere of the other, each run with
// the segment p + t u through it (in its frame): axes of two capsules whose
// radii together are sqrt(r2), so links whose segments are farther apart than
// that have no colliding pair; nor have those where the middle mb of the
// shorter segment b is farther than sqrt(m2), r2's root and half of b, from
// segment a (inv = 1/|ua|^2).
constexpr int kLinkPairs = 32;
struct LinkPair {
  short fa, fb, a0, na, b0, nb;
  float r2, m2, inv, ra;  // ra: how far a's spheres reach from its segment, with the slack of r2
  float pa[3], ua[3], pb[3], ub[3], mb[3];
};
struct LaneRobot {
  int ok, n_link, n_slot, general, last;
  int axis[EZO_MAX_DOF + 2], slot[EZO_MAX_DOF + 2];
  LinkPair link[kLinkPairs];
  int frame[EZO_MAX_SPHERES];  // of each sorted sphere
};

// Device image of a robot: DH chain plus spheres sorted by the frame they are
// attached to. Lives in global memory; kernels stage the small part in smem.
struct RobotDev {
  int n;              // degrees of freedom (<= EZO_MAX_DOF)
  int n_spheres;      // real spheres
  int n_spheres_pad;  // multiple of EZO_CH; padding spheres never collide
  int n_self;         // listed self pairs
  float ca[EZO_MAX_DOF], sa[EZO_MAX_DOF], a[EZO_MAX_DOF], d[EZO_MAX_DOF], toff[EZO_MAX_DOF];
  // joint j turns by kth_j q_j + toff_j and slides by d_j + kd_j q_j:
  // (kth, kd) = (1, 0) for a revolute joint, (0, 1) for a prismatic one
  float kth[EZO_MAX_DOF], kd[EZO_MAX_DOF];
  int frame_first[EZO_MAX_DOF + 2];  // sorted spheres of frame f: [frame_first[f], frame_first[f+1])
  float4 sph[EZO_MAX_SPHERES];       // local x, y, z and radius (sorted by frame)
  const ushort2* self_pairs;         // [n_self] indices into the sorted spheres
  const float* self_rr;              // [n_self] (r_i + r_j)^2
  // Self pairs as work items (r0, nr, k0, nk): sorted spheres [r0, r0 + nr),
  // nr <= EZO_CH, each against the partners [k0, k0 + nk), when the pair
  // list is a union of such blocks (n_sblk > 0, then the n_self pairs are
  // not used); swept like obstacles with band E_self.
  int n_sblk;
  float E_self;
  int4 sblk[EZO_MAX_SBLK];
  // Oriented boxes fixed to frames (sorted by frame, box_first like
  // frame_first), four float4 each in the frame: (centre, h_x), (axis 0, h_y),
  // (axis 1, h_z), (axis 2, 0); self pairs sphere x box and box x box
  int n_box;
  int box_first[EZO_MAX_DOF + 2];
  float4 box_l[4 * EZO_MAX_BOX];
  int n_sbp, n_bbp;
  const ushort2* sb_pairs;  // (sorted sphere, sorted box)
  const ushort2* bb_pairs;  // (sorted box, sorted box)
  LaneRobot lane;
};

// The chain and the spheres in FP64 as given at creation (spheres sorted as
// in RobotDev), for the FP64 reference kinematics that the forward-kinematics
// error of the FP32 checker is measured against.
struct RobotFK64 {
  int n, n_spheres;
  double ca[EZO_MAX_DOF], sa[EZO_MAX_DOF], a[EZO_MAX_DOF], d[EZO_MAX_DOF], toff[EZO_MAX_DOF];
  double kth[EZO_MAX_DOF], kd[EZO_MAX_DOF];
  int frame_first[EZO_MAX_DOF + 2];
  double sx[EZO_MAX_SPHERES], sy[EZO_MAX_SPHERES], sz[EZO_MAX_SPHERES];
};

// The part of RobotDev a block keeps in shared memory.
struct RobotSmem {
  float ca[EZO_MAX_DOF], sa[EZO_MAX_DOF], a[EZO_MAX_DOF], d[EZO_MAX_DOF], toff[EZO_MAX_DOF];
  float kth[EZO_MAX_DOF], kd[EZO_MAX_DOF];
  int frame_first[EZO_MAX_DOF + 2];
  int box_first[EZO_MAX_DOF + 2];
  int n_box, n_sbp, n_bbp;
  int n, n_spheres, n_spheres_pad, n_self;
  int n_sblk;
  float E_self;
  int4 sblk[EZO_MAX_SBLK];
};

__device__ __forceinline__ void stage_robot(RobotSmem& rs, float4* sph_s, const RobotDev* __restrict__ rd) {
  for (int i = threadIdx.x; i < EZO_MAX_DOF; i += blockDim.x) {
    rs.ca[i] = rd->ca[i];
    rs.sa[i] = rd->sa[i];
    rs.a[i] = rd->a[i];
    rs.d[i] = rd->d[i];
    rs.toff[i] = rd->toff[i];
    rs.kth[i] = rd->kth[i];
    rs.kd[i] = rd->kd[i];
  }
  for (int i = threadIdx.x; i < EZO_MAX_DOF + 2; i += blockDim.x) {
    rs.frame_first[i] = rd->frame_first[i];
    rs.box_first[i] = rd->box_first[i];
  }
  for (int i = threadIdx.x; i < EZO_MAX_SBLK; i += blockDim.x) rs.sblk[i] = rd->sblk[i];
  if (threadIdx.x == 0) {
    rs.n = rd->n;
    rs.n_spheres = rd->n_spheres;
    rs.n_spheres_pad = rd->n_spheres_pad;
    rs.n_self = rd->n_self;
    rs.n_sblk = rd->n_sblk;
    rs.E_self = rd->E_self;
    rs.n_box = rd->n_box;
    rs.n_sbp = rd->n_sbp;
    rs.n_bbp = rd->n_bbp;
  }
  const int np = rd->n_spheres_pad;
  for (int i = threadIdx.x; i < np; i += blockDim.x) sph_s[i] = rd->sph[i];
}

// The robot's boxes in their frames (4 float4 per box) into shared memory.
__device__ __forceinline__ void stage_robot_boxes(float4* rbox_l, const RobotDev* __restrict__ rd) {
  const int nb = 4 * rd->n_box;
  for (int i = threadIdx.x; i < nb; i += blockDim.x) rbox_l[i] = rd->box_l[i];
}

// Grid over an obstacle set (built once per set by k_grid_build): up to 32
// coarse cells an axis and as many or twice as many fine ones. For a point of coarse
// cell i, lb[i] step is a lower bound of its distance to the nearest obstacle
// surface; a point outside the grid is at least as far from all of them as from
// the box around them. A fine cell
// lists the obstacles that can be the nearest to some point of it: obstacle j
// is left out when another one is nearer to every point of the cell, so a
// sphere of any radius whose centre lies in the cell collides with the set
// exactly when it collides with a listed obstacle. Bounds are built with a
// margin of 4e-6 of the coordinates' size, some thirty roundings of the FP32
// pair test, so labels equal the FP32 test over all pairs.
// cell[i]: bits 0-7 the fine cell's bound in units of step, bits 8-15 the
// count of ids in bits 16 + 12 k (count <= kGridInline), or kGridList: a list
// of (bits 16-31) ids from ids[bits 32-63], or kGridAll: every obstacle.
constexpr int kGridC = 32;             // coarse cells an axis (row stride)
constexpr int kGridLbBytes = kGridC * kGridC * kGridC;
constexpr unsigned kGridInline = 4, kGridList = 0xFE, kGridAll = 0xFF;

struct ObsGrid {
  // before the bounds, two float4: the box around the obstacles (its least and
  // largest coordinates; the first one's w is added to a radius that is
  // compared with the distance to the box)
  const uint8_t* lb;
  const unsigned long long* cell;
  const uint16_t* ids;
  // x inv is the coarse cell coordinate; fma_rd(x, inv, bx) has floor(x inv)
  // less the first cell's index in its low mantissa bits (bx = 2^23 - index,
  // so the sum's unit is 1 and rounding down is the floor), fma_rd(x, finv,
  // fx) likewise for the fine cells
  float inv, finv, inv_step;
  float bx, by, bz, fx, fy, fz;
  float ex, ey, ez;  // 2^23 + fine cells
  int fbits;         // log2 of the fine cells' row stride: 5 or 6
  int large;         // whether the robot has spheres that can be hit with their centres outside the grid
  float step;        // metres a unit of lb
};

// The signed distance's grid: 32 cells an axis over the obstacles and their
// extent all around, each with its candidates (cell words as in ObsGrid, the
// bound in units of step), and the box it covers; or, with cell null, the
// collision grid's coarse cells, which have a bound but no candidates.
struct WideGrid {
  const unsigned long long* cell;
  const uint16_t* ids;
  float inv, step, r_obs;           // r_obs: the largest obstacle radius
  float fx, fy, fz, ex, ey, ez;     // as in ObsGrid
  float lx, ly, lz, hx, hy, hz;
};

// Obstacle set in global memory: (x, y, z, R), padded to a multiple of EZO_CH.
struct EnvDev {
  const float4* obs;
  int n_obs;
  int n_obs_pad;
  const float4* box;  // obstacle boxes, 4 float4 each: (centre, h_x), (axis 0, h_y), (axis 1, h_z), (axis 2, 0)
  int n_box;
  // first robot sphere of the obstacle tests: the spheres before it sit on the
  // fixed base frame, so their pairs with these obstacles are the same for
  // every configuration, and they were found clear of every obstacle by more
  // than any rounding band when the pair (robot, obstacle set) was set up
  int s_first;
  ObsGrid grid;
};

constexpr float kGridBias = 8388608.f;  // 2^23

__device__ __forceinline__ void stage_env_boxes(float4* ebox_s, const EnvDev& e) {
  for (int i = threadIdx.x; i < 4 * e.n_box; i += blockDim.x) ebox_s[i] = e.box[i];
}

// Box geometry of one collision group (all in shared memory).
struct BoxCtx {
  const float4* rbox_l;  // robot boxes in their frames
  const float4* ebox;    // obstacle boxes of the current environment
  float4* rbox_w;        // this group's robot boxes in the world
  int n_ebox;
  const ushort2* sb_pairs;
  const ushort2* bb_pairs;
};

// Sphere (centre c.xyz, radius r) against an oriented box B (4 float4): the
// centre in box coordinates p_k = axis_k . (c - centre), q_k = abs(p_k) - h_k;
// overlap iff the centre is strictly inside (every q_k < 0) or the squared
// norm of max(q, 0) is below r^2.
__device__ __forceinline__ bool sphere_box_hit(float4 c, float r, const float4* __restrict__ B) {
  const float4 b0 = B[0], b1 = B[1], b2 = B[2], b3 = B[3];
  const float dx = c.x - b0.x, dy = c.y - b0.y, dz = c.z - b0.z;
  const float q0 = fabsf(fmaf(dx, b1.x, fmaf(dy, b1.y, dz * b1.z))) - b0.w;
  const float q1 = fabsf(fmaf(dx, b2.x, fmaf(dy, b2.y, dz * b2.z))) - b1.w;
  const float q2 = fabsf(fmaf(dx, b3.x, fmaf(dy, b3.y, dz * b3.z))) - b2.w;
  if (q0 < 0.f && q1 < 0.f && q2 < 0.f) return true;
  const float m0 = fmaxf(q0, 0.f), m1 = fmaxf(q1, 0.f), m2 = fmaxf(q2, 0.f);
  return fmaf(m0, m0, fmaf(m1, m1, m2 * m2)) < r * r;
}

// Separating-axis test of two oriented boxes, written in A's frame: with
// t = A^T (c_B - c_A) and R = A^T B, a candidate axis L separates when
// abs(t . L) - sum_k hA_k abs(L_k) - sum_k hB_k abs(r_k . L) >= 0 (r_k the
// columns of R); the candidates are A's axes, B's axes and e_i x r_j, the
// latter skipped when abs(L)^2 < 1e-4 (nearly parallel edges). The boxes
// overlap iff no candidate separates them. Scaling L does not change the sign,
// so the cross products are not normalised.
__device__ __forceinline__ bool box_box_hit(const float4* __restrict__ A, const float4* __restrict__ B) {
  const float4 a0 = A[0], a1 = A[1], a2 = A[2], a3 = A[3];
  const float4 b0 = B[0], b1 = B[1], b2 = B[2], b3 = B[3];
  const float ha[3] = {a0.w, a1.w, a2.w}, hb[3] = {b0.w, b1.w, b2.w};
  const float Tx = b0.x - a0.x, Ty = b0.y - a0.y, Tz = b0.z - a0.z;
  const float ax[3][3] = {{a1.x, a1.y, a1.z}, {a2.x, a2.y, a2.z}, {a3.x, a3.y, a3.z}};
  const float bx[3][3] = {{b1.x, b1.y, b1.z}, {b2.x, b2.y, b2.z}, {b3.x, b3.y, b3.z}};
  float t[3], R[3][3], aR[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    t[i] = fmaf(Tx, ax[i][0], fmaf(Ty, ax[i][1], Tz * ax[i][2]));
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      R[i][j] = fmaf(ax[i][0], bx[j][0], fmaf(ax[i][1], bx[j][1], ax[i][2] * bx[j][2]));
      aR[i][j] = fabsf(R[i][j]);
    }
  }
#pragma unroll
  for (int i = 0; i < 3; ++i)  // A's axes
    if (fabsf(t[i]) - ha[i] - fmaf(hb[0], aR[i][0], fmaf(hb[1], aR[i][1], hb[2] * aR[i][2])) >= 0.f) return false;
#pragma unroll
  for (int j = 0; j < 3; ++j) {  // B's axes
    const float tj = fmaf(t[0], R[0][j], fmaf(t[1], R[1][j], t[2] * R[2][j]));
    if (fabsf(tj) - fmaf(ha[0], aR[0][j], fmaf(ha[1], aR[1][j], ha[2] * aR[2][j])) - hb[j] >= 0.f) return false;
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      // L = e_i x r_j in A's frame
      float L[3];
      L[i] = 0.f;
      L[(i + 1) % 3] = -R[(i + 2) % 3][j];
      L[(i + 2) % 3] = R[(i + 1) % 3][j];
      const float n2 = fmaf(L[0], L[0], fmaf(L[1], L[1], L[2] * L[2]));
      if (n2 < 1e-4f) continue;
      const float tl = fmaf(t[0], L[0], fmaf(t[1], L[1], t[2] * L[2]));
      const float ra = fmaf(ha[0], fabsf(L[0]), fmaf(ha[1], fabsf(L[1]), ha[2] * fabsf(L[2])));
      float rb = 0.f;
#pragma unroll
      for (int k = 0; k < 3; ++k)
        rb = fmaf(hb[k], fabsf(fmaf(R[0][k], L[0], fmaf(R[1][k], L[1], R[2][k] * L[2]))), rb);
      if (fabsf(tl) - ra - rb >= 0.f) return false;
    }
  }
  return true;
}

// max of three floats in one instruction (PTX max.f32 with three inputs).
__device__ __forceinline__ float fmax3f(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// World poses of the boxes [b0, b1) of one frame (rotation columns c0..c2,
// origin in the .w entries): centre o + R c, axes R a_k; boxes b with
// b % T == lg on this lane.
template <int T>
__device__ __forceinline__ void box_poses_of_frame(int b0, int b1, int lg, float4 c0, float4 c1, float4 c2,
                                                const BoxCtx& bx) {
  int b = b0 + ((lg - b0) & (T - 1));
  for (; b < b1; b += T) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float4 l = bx.rbox_l[4 * b + k];
      const float ox = k == 0 ? c0.w : 0.f, oy = k == 0 ? c1.w : 0.f, oz = k == 0 ? c2.w : 0.f;
      bx.rbox_w[4 * b + k] = make_float4(fmaf(c0.x, l.x, fmaf(c1.x, l.y, fmaf(c2.x, l.z, ox))),
                                         fmaf(c0.y, l.x, fmaf(c1.y, l.y, fmaf(c2.y, l.z, oy))),
                                         fmaf(c0.z, l.x, fmaf(c1.z, l.y, fmaf(c2.z, l.z, oz))), l.w);
    }
  }
}

// -------------------------------------------------- FK + collision test --
// Forward kinematics of one configuration by a group of T lanes (T in
// 1..32) of one warp, as the collision checker runs it: the group's lanes share
// the joint sines and cosines, lane lg writes the centres of spheres s with
// s % T == lg into the group's shared slot `cen` as (x, y, z, (|c|^2 - r^2)/2)
// (padding spheres get an infinite last entry), and BOX poses the robot's
// boxes. Ends with a warp barrier; every lane of the warp must call it.
template <int NDOF, int T, bool BOX = false>
__device__ __forceinline__ void fk_group(const float (&q)[NDOF], const RobotSmem& rs,
                                         const float4* __restrict__ sph_s, float4* __restrict__ cen, int lg,
                                         const BoxCtx& bx) {
  float c0x = 1.f, c0y = 0.f, c0z = 0.f;
  float c1x = 0.f, c1y = 1.f, c1z = 0.f;
  float c2x = 0.f, c2y = 0.f, c2z = 1.f;
  float px = 0.f, py = 0.f, pz = 0.f;
  const int n = rs.n;
  // sine and cosine of every joint angle. With T lanes per configuration,
  // lane lg evaluates joints lg, lg + T, .. (all lanes run the same
  // instructions on their own angle) and the group exchanges the results;
  // the values are the same as one lane evaluating all of them.
  float sj[NDOF], cj[NDOF];
  if (T == 1) {
#pragma unroll
    for (int j = 0; j < NDOF; ++j) {
      sj[j] = 0.f;
      cj[j] = 1.f;
      if (j < n) sincosf(fmaf(q[j], rs.kth[j], rs.toff[j]), &sj[j], &cj[j]);
    }
  } else {
    constexpr int JPL = (NDOF + T - 1) / T;
    float ms[JPL], mc[JPL];
#pragma unroll
    for (int k = 0; k < JPL; ++k) {
      const int jm = lg + k * T;
      float ang = 0.f;
#pragma unroll
      for (int j = 0; j < NDOF; ++j)
        if (j == jm && j < n) ang = fmaf(q[j], rs.kth[j], rs.toff[j]);
      sincosf(ang, &ms[k], &mc[k]);
    }
#pragma unroll
    for (int j = 0; j < NDOF; ++j) {
      sj[j] = __shfl_sync(0xffffffffu, ms[j / T], j % T, T);
      cj[j] = __shfl_sync(0xffffffffu, mc[j / T], j % T, T);
    }
  }
#pragma unroll
  for (int f = 0; f <= NDOF; ++f) {
    if (f > n) break;
    if (f > 0) {
      const int j = f - 1;
      const float s = sj[j], c = cj[j];
      // R_{j} Rz(theta): col0' = c col0 + s col1, col1' = -s col0 + c col1
      const float n0x = fmaf(c, c0x, s * c1x), n0y = fmaf(c, c0y, s * c1y), n0z = fmaf(c, c0z, s * c1z);
      const float n1x = fmaf(c, c1x, -s * c0x), n1y = fmaf(c, c1y, -s * c0y), n1z = fmaf(c, c1z, -s * c0z);
      // o_{j+1} = o_j + a col0' + d col2
      const float aj = rs.a[j], dj = fmaf(q[j], rs.kd[j], rs.d[j]);
      px = fmaf(aj, n0x, fmaf(dj, c2x, px));
      py = fmaf(aj, n0y, fmaf(dj, c2y, py));
      pz = fmaf(aj, n0z, fmaf(dj, c2z, pz));
      // Rx(alpha): col1'' = ca col1' + sa col2, col2'' = -sa col1' + ca col2
      const float ca = rs.ca[j], sa = rs.sa[j];
      const float m1x = fmaf(ca, n1x, sa * c2x), m1y = fmaf(ca, n1y, sa * c2y), m1z = fmaf(ca, n1z, sa * c2z);
      const float m2x = fmaf(ca, c2x, -sa * n1x), m2y = fmaf(ca, c2y, -sa * n1y), m2z = fmaf(ca, c2z, -sa * n1z);
      c0x = n0x; c0y = n0y; c0z = n0z;
      c1x = m1x; c1y = m1y; c1z = m1z;
      c2x = m2x; c2y = m2y; c2z = m2z;
    }
    const int s_end = rs.frame_first[f + 1];
    int s = rs.frame_first[f];
    s += (lg - s) & (T - 1);
    for (; s < s_end; s += T) {
      const float4 l = sph_s[s];
      const float cx = fmaf(c0x, l.x, fmaf(c1x, l.y, fmaf(c2x, l.z, px)));
      const float cy = fmaf(c0y, l.x, fmaf(c1y, l.y, fmaf(c2y, l.z, py)));
      const float cz = fmaf(c0z, l.x, fmaf(c1z, l.y, fmaf(c2z, l.z, pz)));
      const float hu = 0.5f * fmaf(cx, cx, fmaf(cy, cy, fmaf(cz, cz, -l.w * l.w)));
      cen[s] = make_float4(cx, cy, cz, hu);
    }
    if constexpr (BOX)
      box_poses_of_frame<T>(rs.box_first[f], rs.box_first[f + 1], lg, make_float4(c0x, c0y, c0z, px),
                            make_float4(c1x, c1y, c1z, py), make_float4(c2x, c2y, c2z, pz), bx);
  }
  for (int s = rs.n_spheres + lg; s < rs.n_spheres_pad; s += T) cen[s] = make_float4(0.f, 0.f, 0.f, __int_as_float(0x7f800000));
  __syncwarp();
}

// The direct pair test of sphere (c.xyz, r) against obstacle o, in FP32.
__device__ __forceinline__ bool pair_hit(float cx, float cy, float cz, float r, float4 o) {
  const float dx = cx - o.x, dy = cy - o.y, dz = cz - o.z;
  const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
  const float sr = r + o.w;
  return d2 < sr * sr;
}

// Sphere (c.xyz, r) against the obstacles of the fine cell of its centre
// (every obstacle when the centre lies outside the grid).
__device__ __forceinline__ bool cell_hit(const EnvDev& e, float cx, float cy, float cz, float r) {
  const ObsGrid& g = e.grid;
  const float ux = __fmaf_rd(cx, g.finv, g.fx), uy = __fmaf_rd(cy, g.finv, g.fy), uz = __fmaf_rd(cz, g.finv, g.fz);
  const bool in = ux >= kGridBias && uy >= kGridBias && uz >= kGridBias && ux < g.ex && uy < g.ey && uz < g.ez;
  unsigned long long d = (unsigned long long)kGridAll << 8;
  if (in) {
    const unsigned ix = __float_as_uint(ux) & 0xffu, iy = __float_as_uint(uy) & 0xffu, iz = __float_as_uint(uz) & 0xffu;
    d = __ldg(g.cell + ((((iz << g.fbits) + iy) << g.fbits) + ix));
    if (__fmaf_ru(r, g.inv_step, kGridBias) < __uint_as_float(0x4B000000u | (unsigned)(d & 0xffu))) return false;
  }
  const unsigned kind = (unsigned)(d >> 8) & 0xffu;
  unsigned id[kGridInline];
  float4 o[kGridInline];
  bool hit = false;
  if (kind <= kGridInline) {
    // the word's one to four ids, their obstacles loaded together
#pragma unroll
    for (unsigned k = 0; k < kGridInline; ++k)
      id[k] = (k < kind ? (unsigned)(d >> (16 + 12 * k)) : (unsigned)(d >> 16)) & 0xfffu;
#pragma unroll
    for (unsigned k = 0; k < kGridInline; ++k) o[k] = __ldg(e.obs + id[k]);
#pragma unroll
    for (unsigned k = 0; k < kGridInline; ++k) hit = pair_hit(cx, cy, cz, r, o[k]) || hit;
    return hit;
  }
  // four at a time; past the last one the last again
  const bool list = kind == kGridList;
  const int cnt = list ? (int)((d >> 16) & 0xffffu) : e.n_obs;
  const uint16_t* ids = g.ids + (list ? (unsigned)(d >> 32) : 0u);
  for (int k0 = 0; k0 < cnt && !hit; k0 += (int)kGridInline) {
#pragma unroll
    for (int k = 0; k < (int)kGridInline; ++k) {
      const int at = min(k0 + k, cnt - 1);
      id[k] = list ? (unsigned)__ldg(ids + at) : (unsigned)at;
    }
#pragma unroll
    for (unsigned k = 0; k < kGridInline; ++k) o[k] = __ldg(e.obs + id[k]);
#pragma unroll
    for (unsigned k = 0; k < kGridInline; ++k) hit = pair_hit(cx, cy, cz, r, o[k]) || hit;
  }
  return hit;
}

// Whether a sphere whose centre lies outside the grid can touch an obstacle:
// it is free when the box around them is farther than its radius, by more than
// the roundings of this test and of the pair test.
__device__ __forceinline__ bool box_within(const ObsGrid& g, float cx, float cy, float cz, float r) {
  const float4* box = reinterpret_cast<const float4*>(g.lb);
  const float4 lo = __ldg(box - 2), hi = __ldg(box - 1);
  const float ox = fmaxf(fmaxf(lo.x - cx, cx - hi.x), 0.f), oy = fmaxf(fmaxf(lo.y - cy, cy - hi.y), 0.f),
              oz = fmaxf(fmaxf(lo.z - cz, cz - hi.z), 0.f);
  const float reach = fmaf(r, 1.00001f, lo.w);
  return !(fmaf(ox, ox, fmaf(oy, oy, oz * oz)) > reach * reach);
}

// The coarse cell of a point as an index into lb; false outside the grid: all
// three coordinates in [2^23, 2^23 + 32) have no bit but the low five different
// from 2^23's.
__device__ __forceinline__ bool coarse_cell(const ObsGrid& g, float cx, float cy, float cz, unsigned& cell) {
  const unsigned ix = __float_as_uint(__fmaf_rd(cx, g.inv, g.bx)), iy = __float_as_uint(__fmaf_rd(cy, g.inv, g.by)),
                 iz = __float_as_uint(__fmaf_rd(cz, g.inv, g.bz));
  cell = ((iz * kGridC + iy) * kGridC + ix) & (kGridLbBytes - 1);
  return ((ix ^ 0x4B000000u) | (iy ^ 0x4B000000u) | (iz ^ 0x4B000000u)) < (unsigned)kGridC;
}

// Whether the coarse bound leaves a sphere to be tested: it is free when
// ceil(r / step) < lb (a bound of 0 may stand for a negative one).
__device__ __forceinline__ bool coarse_near(const ObsGrid& g, const uint8_t* __restrict__ lb, float cx, float cy,
                                            float cz, float r) {
  unsigned i;
  if (!coarse_cell(g, cx, cy, cz, i)) return box_within(g, cx, cy, cz, r);
  const float bound = __uint_as_float(0x4B000000u | (unsigned)lb[i]);
  return !(__fmaf_ru(r, g.inv_step, kGridBias) < bound);
}

// The obstacle tests of this lane's spheres s_first + lg, + T, .. of one
// configuration. The first pass drops the spheres that the coarse bound shows
// free (most of them: about twenty instructions a sphere whatever the number
// of obstacles, where a sweep over all of them took three a pair); the second
// takes the others one by one, so lanes with few of them wait only for the
// lane with the most. 7-DOF arm of 40 spheres, against the sweep: 2e6 labels
// among 64 obstacles 0.91 -> 0.55 ms, 2e5 among 1024 1.03 -> 0.106 ms.
template <int T>
__device__ __forceinline__ bool obstacles_hit(const RobotSmem& rs, const float4* __restrict__ sph_s, const EnvDev& e,
                                              const uint8_t* __restrict__ lb, const float4* __restrict__ cen,
                                              int lg) {
  const ObsGrid& g = e.grid;
  const int ns = e.n_obs > 0 ? rs.n_spheres : 0;
  bool hit = false;
  for (int s0 = e.s_first + lg; s0 < ns; s0 += 32 * T) {
    unsigned near = 0u;
#pragma unroll 4
    for (int k = 0; k < 32; ++k) {
      const int s = s0 + k * T;
      if (s >= ns) break;
      const float4 c = cen[s];
      if (coarse_near(g, lb, c.x, c.y, c.z, sph_s[s].w)) near |= 1u << k;
    }
    while (near) {
      const int s = s0 + (__ffs(near) - 1) * T;
      near &= near - 1u;
      const float4 c = cen[s];
      if (cell_hit(e, c.x, c.y, c.z, sph_s[s].w)) {
        hit = true;
        break;
      }
    }
    if (hit) break;
  }
  return hit;
}

// Whether the coarse bounds leave a box of the world to be tested against the
// obstacles: it is cut along its longest axis into up to four parts, and free
// when the sphere around each is (an obstacle that touches the box touches
// one of them). The spheres' 1e-5 covers the roundings of their centres, the
// bounds' margin those of the box test. A box that is not finite is tested.
__device__ __forceinline__ bool box_near(const ObsGrid& g, const uint8_t* __restrict__ lb,
                                         const float4* __restrict__ B) {
  const float4 b0 = B[0], b1 = B[1], b2 = B[2], b3 = B[3];
  if (!(fabsf(b0.x) + fabsf(b0.y) + fabsf(b0.z) < 1e30f)) return true;
  const bool l2 = b2.w >= b0.w && b2.w >= b1.w, l1 = !l2 && b1.w >= b0.w;
  const float ax = l2 ? b3.x : (l1 ? b2.x : b1.x), ay = l2 ? b3.y : (l1 ? b2.y : b1.y),
              az = l2 ? b3.z : (l1 ? b2.z : b1.z);
  const float h = l2 ? b2.w : (l1 ? b1.w : b0.w), p = l2 ? b0.w : (l1 ? b2.w : b1.w),
              q = l2 ? b1.w : (l1 ? b0.w : b2.w);
  const float across = fmaf(p, p, q * q) * 1.00001f;
  const float parts = fminf(4.f, ceilf(fmaxf(h * rsqrtf(fmaxf(across, 1e-30f)), 1.f)));
  const float half = h / parts;
  const float r = sqrtf(fmaf(half, half, across)) * 1.00001f;
  for (float k = 0.f; k < parts; k += 1.f) {
    const float t = fmaf(2.f * k + 1.f, half, -h);
    if (coarse_near(g, lb, fmaf(ax, t, b0.x), fmaf(ay, t, b0.y), fmaf(az, t, b0.z), r)) return true;
  }
  return false;
}

// The pairs of one configuration that involve a box, split over the T lanes
// of its group: robot spheres x obstacle boxes, robot boxes x obstacle
// spheres and boxes, listed sphere-box and box-box self pairs. Returns this
// lane's OR; every lane of the warp must call it, those that have a hit pass
// it. The robot boxes that the grid's bounds leave are tested against every
// obstacle sphere, a box at a time in registers. A path check of 300 edges at
// step 0.01 for the arm of 11 boxes among 3 boxes and some 100 spheres: 111 ->
// 71 us a call; each box against each sphere, found by a division, was four
// fifths of the kernel. Testing the boxes' own axes for all pairs of boxes
// before the full test of those left was no faster (82 us).
template <int T>
__device__ __forceinline__ bool box_pairs_hit(const RobotSmem& rs, const float4* __restrict__ sph_s,
                                           const EnvDev& env, const uint8_t* __restrict__ lb,
                                           const float4* __restrict__ cen, int lg, const BoxCtx& bx, bool hit) {
  const int ns = rs.n_spheres, nb = rs.n_box, ne = bx.n_ebox, n_obs = env.n_obs;
  for (int e = 0; e < ne; ++e)  // robot spheres x obstacle boxes
    for (int s = lg; s < ns && !hit; s += T) hit = sphere_box_hit(cen[s], sph_s[s].w, bx.ebox + 4 * e);
  if (n_obs > 0 && nb > 0) {  // robot boxes x obstacle spheres
    unsigned near = 0u;  // the group's boxes (at most 32) that may touch one
    for (int b0 = 0; b0 < nb; b0 += T) {
      const int b = b0 + lg;
      const unsigned in = __ballot_sync(0xffffffffu, b < nb && box_near(env.grid, lb, bx.rbox_w + 4 * b));
      near |= ((in >> ((threadIdx.x & 31) - lg)) & (T == 32 ? ~0u : (1u << (T & 31)) - 1u)) << b0;
    }
    while (near && !hit) {
      const float4* B = bx.rbox_w + 4 * (__ffs(near) - 1);
      near &= near - 1u;
      const float4 w[4] = {B[0], B[1], B[2], B[3]};
      for (int o0 = lg; o0 < n_obs && !hit; o0 += 4 * T) {
        float4 ob[4];  // past the last one: the last again
#pragma unroll
        for (int k = 0; k < 4; ++k) ob[k] = __ldg(env.obs + min(o0 + k * T, n_obs - 1));
#pragma unroll
        for (int k = 0; k < 4; ++k) hit = sphere_box_hit(ob[k], ob[k].w, w) || hit;
      }
    }
  }
  for (int p = lg; p < nb * ne && !hit; p += T) {  // robot boxes x obstacle boxes
    const int b = p / ne, e = p - b * ne;
    hit = box_box_hit(bx.rbox_w + 4 * b, bx.ebox + 4 * e);
  }
  for (int p = lg; p < rs.n_sbp && !hit; p += T) {  // self: sphere x box
    const ushort2 pr = bx.sb_pairs[p];
    hit = sphere_box_hit(cen[pr.x], sph_s[pr.x].w, bx.rbox_w + 4 * pr.y);
  }
  for (int p = lg; p < rs.n_bbp && !hit; p += T) {  // self: box x box
    const ushort2 pr = bx.bb_pairs[p];
    hit = box_box_hit(bx.rbox_w + 4 * pr.x, bx.rbox_w + 4 * pr.y);
  }
  return hit;
}

// ---------------------------------------- spheres formed in registers --
// The robot in shared memory for collide_lane, followed by the spheres
// (float4), per sphere (coordinate along its frame's axis, ceil(r / step) for
// the obstacle set's grid) and frame, the grid's coarse bounds when staged,
// and per group of lanes its words.
struct LaneSmem {
  float4 joint[2 * EZO_MAX_DOF];  // (ca, sa, a, d), (toff, kth, kd, 0)
  int frame_first[EZO_MAX_DOF + 2], axis[EZO_MAX_DOF + 2], slot[EZO_MAX_DOF + 2];
  int n, n_spheres, last, n_link, general, n_self;
  const ushort2* self_pairs;  // in global memory
  LinkPair link[kLinkPairs];
};

// Floats of a group: one lane keeps the joint values and each pose's numbers
// at the block's stride; more lanes keep poses as float4s (origin, axis[, two
// columns]), an odd number of them, so that the groups of a warp read
// different banks.
__host__ __device__ inline int lane_group_words(int n, int n_slot, int general, int T) {
  if (T == 1) return n + n_slot * (general ? 12 : 6);
  return 4 * ((n_slot * (general ? 4 : 2)) | 1);
}

__device__ __forceinline__ void stage_lane_robot(LaneSmem& ls, float4* sph, int* frame,
                                                 const RobotDev* __restrict__ rd) {
  const LaneRobot& lr = rd->lane;
  for (int i = threadIdx.x; i < EZO_MAX_DOF; i += blockDim.x) {
    ls.joint[2 * i] = make_float4(rd->ca[i], rd->sa[i], rd->a[i], rd->d[i]);
    ls.joint[2 * i + 1] = make_float4(rd->toff[i], rd->kth[i], rd->kd[i], 0.f);
  }
  for (int i = threadIdx.x; i < EZO_MAX_DOF + 2; i += blockDim.x) {
    ls.frame_first[i] = rd->frame_first[i];
    ls.axis[i] = lr.axis[i];
    ls.slot[i] = lr.slot[i];
  }
  for (int i = threadIdx.x; i < lr.n_link * (int)(sizeof(LinkPair) / 4); i += blockDim.x)
    reinterpret_cast<int*>(ls.link)[i] = reinterpret_cast<const int*>(lr.link)[i];
  if (threadIdx.x == 0) {
    ls.n = rd->n;
    ls.n_spheres = rd->n_spheres;
    ls.last = lr.last;
    ls.n_link = lr.n_link;
    ls.general = lr.general;
    ls.n_self = rd->n_self;
    ls.self_pairs = rd->self_pairs;
  }
  for (int i = threadIdx.x; i < rd->n_spheres; i += blockDim.x) {
    sph[i] = rd->sph[i];
    frame[i] = lr.frame[i];
  }
}

// (coordinate on the axis, ceil(r / step)) of every sphere; a sphere before
// s_first, or any when there are no obstacles, gets -1: free whatever the bound
__device__ __forceinline__ void stage_lane_env(float2* sa, const RobotDev* __restrict__ rd, const EnvDev& e) {
  for (int i = threadIdx.x; i < rd->n_spheres; i += blockDim.x) {
    const float4 l = rd->sph[i];
    const int axis = rd->lane.axis[rd->lane.frame[i]];
    const int q = e.n_obs == 0 || i < e.s_first ? -1 : (int)fminf(ceilf(__fmul_ru(l.w, e.grid.inv_step)), 1.0e6f);
    sa[i] = make_float2(axis == 1 ? l.x : (axis == 2 ? l.y : l.z), __int_as_float(q));
  }
}

// A frame's pose as collide_lane uses it: origin p, the axis v its spheres lie
// on, and for a general frame the other two columns.
struct LanePose {
  float px, py, pz, vx, vy, vz;
  float ax, ay, az, bx, by, bz;  // columns 0 and 1 (axis 0 only; v is column 2 then)
};

// Centre of a sphere: one multiply-add a coordinate on an axis (the other two
// products of fk_group's chain are exact zeros there), its whole chain else.
__device__ __forceinline__ void lane_centre(const LanePose& P, int axis, float la, const float4* __restrict__ l,
                                            float& cx, float& cy, float& cz) {
  cx = fmaf(P.vx, la, P.px);
  cy = fmaf(P.vy, la, P.py);
  cz = fmaf(P.vz, la, P.pz);
  if (axis == 0) {
    const float lx = l->x, ly = l->y;
    cx = fmaf(P.ax, lx, fmaf(P.bx, ly, cx));
    cy = fmaf(P.ay, lx, fmaf(P.by, ly, cy));
    cz = fmaf(P.az, lx, fmaf(P.bz, ly, cz));
  }
}

// Keeps and reads the pose of slot k (lane_group_words).
template <int T>
__device__ __forceinline__ void lane_keep(const LanePose& P, int k, int general, float* mine, int stride) {
  if (T == 1) {
    float* o = mine + k * (general ? 12 : 6) * stride;
    o[0] = P.px, o[stride] = P.py, o[2 * stride] = P.pz;
    o[3 * stride] = P.vx, o[4 * stride] = P.vy, o[5 * stride] = P.vz;
    if (general) {
      o[6 * stride] = P.ax, o[7 * stride] = P.ay, o[8 * stride] = P.az;
      o[9 * stride] = P.bx, o[10 * stride] = P.by, o[11 * stride] = P.bz;
    }
  } else {
    float4* o = reinterpret_cast<float4*>(mine) + k * (general ? 4 : 2);
    o[0] = make_float4(P.px, P.py, P.pz, 0.f);
    o[1] = make_float4(P.vx, P.vy, P.vz, 0.f);
    if (general) {
      o[2] = make_float4(P.ax, P.ay, P.az, 0.f);
      o[3] = make_float4(P.bx, P.by, P.bz, 0.f);
    }
  }
}
template <int T>
__device__ __forceinline__ LanePose lane_pose(int k, int general, const float* mine, int stride) {
  LanePose P;
  P.ax = P.ay = P.az = P.bx = P.by = P.bz = 0.f;
  if (T == 1) {
    const float* o = mine + k * (general ? 12 : 6) * stride;
    P.px = o[0], P.py = o[stride], P.pz = o[2 * stride];
    P.vx = o[3 * stride], P.vy = o[4 * stride], P.vz = o[5 * stride];
    if (general) {
      P.ax = o[6 * stride], P.ay = o[7 * stride], P.az = o[8 * stride];
      P.bx = o[9 * stride], P.by = o[10 * stride], P.bz = o[11 * stride];
    }
  } else {
    const float4* o = reinterpret_cast<const float4*>(mine) + k * (general ? 4 : 2);
    const float4 p = o[0], v = o[1];
    P.px = p.x, P.py = p.y, P.pz = p.z;
    P.vx = v.x, P.vy = v.y, P.vz = v.z;
    if (general) {
      const float4 a = o[2], b = o[3];
      P.ax = a.x, P.ay = a.y, P.az = a.z;
      P.bx = b.x, P.by = b.y, P.bz = b.z;
    }
  }
  return P;
}

// The next frame of the chain (fk_group's operations, in its order).
struct LaneChain {
  float c0x, c0y, c0z, c1x, c1y, c1z, c2x, c2y, c2z, px, py, pz;
  __device__ __forceinline__ void start() {
    c0x = 1.f, c0y = 0.f, c0z = 0.f, c1x = 0.f, c1y = 1.f, c1z = 0.f, c2x = 0.f, c2y = 0.f, c2z = 1.f;
    px = py = pz = 0.f;
  }
  __device__ __forceinline__ void step(float4 J, float4 K, float qj, float s, float c) {
    const float n0x = fmaf(c, c0x, s * c1x), n0y = fmaf(c, c0y, s * c1y), n0z = fmaf(c, c0z, s * c1z);
    const float n1x = fmaf(c, c1x, -s * c0x), n1y = fmaf(c, c1y, -s * c0y), n1z = fmaf(c, c1z, -s * c0z);
    const float aj = J.z, dj = fmaf(qj, K.z, J.w);
    px = fmaf(aj, n0x, fmaf(dj, c2x, px));
    py = fmaf(aj, n0y, fmaf(dj, c2y, py));
    pz = fmaf(aj, n0z, fmaf(dj, c2z, pz));
    const float ca = J.x, sn = J.y;
    const float m1x = fmaf(ca, n1x, sn * c2x), m1y = fmaf(ca, n1y, sn * c2y), m1z = fmaf(ca, n1z, sn * c2z);
    const float m2x = fmaf(ca, c2x, -sn * n1x), m2y = fmaf(ca, c2y, -sn * n1y), m2z = fmaf(ca, c2z, -sn * n1z);
    c0x = n0x, c0y = n0y, c0z = n0z;
    c1x = m1x, c1y = m1y, c1z = m1z;
    c2x = m2x, c2y = m2y, c2z = m2z;
  }
  __device__ __forceinline__ LanePose pose(int axis) const {
    LanePose P;
    P.px = px, P.py = py, P.pz = pz;
    P.vx = axis == 1 ? c0x : (axis == 2 ? c1x : c2x);
    P.vy = axis == 1 ? c0y : (axis == 2 ? c1y : c2y);
    P.vz = axis == 1 ? c0z : (axis == 2 ? c1z : c2z);
    P.ax = c0x, P.ay = c0y, P.az = c0z, P.bx = c1x, P.by = c1y, P.bz = c1z;
    return P;
  }
};

// Whether the coarse bound leaves a sphere (centre c, q = ceil(r / step)) to
// be tested: its centre in the grid and its radius not below the bound, or,
// with LARGE, a centre outside and a radius that can reach in from there.
template <bool LARGE>
__device__ __forceinline__ bool lane_near(const ObsGrid& g, const uint8_t* __restrict__ lb, float cx, float cy,
                                          float cz, int q, const float4* __restrict__ l) {
  unsigned i;
  const bool in = coarse_cell(g, cx, cy, cz, i);
  if constexpr (LARGE) return in ? q >= (int)lb[i] : q >= 0 && box_within(g, cx, cy, cz, l->w);
  return in && q >= (int)lb[i];
}

// Point or vector (w = 1 or 0 for the origin) of a run's segment in the world.
__device__ __forceinline__ void lane_world(const LanePose& P, int axis, const float (&l)[3], float w, float& x,
                                           float& y, float& z) {
  const float a = axis == 1 ? l[0] : (axis == 2 ? l[1] : l[2]);
  x = fmaf(P.vx, a, w * P.px);
  y = fmaf(P.vy, a, w * P.py);
  z = fmaf(P.vz, a, w * P.pz);
  if (axis == 0) {
    x = fmaf(P.ax, l[0], fmaf(P.bx, l[1], x));
    y = fmaf(P.ay, l[0], fmaf(P.by, l[1], y));
    z = fmaf(P.az, l[0], fmaf(P.bz, l[1], z));
  }
}

// The self pairs from the kept poses, links lg, lg + T, ..: the squared
// distance of the two segments (any point pair on them bounds it from above,
// and the pair found is the nearest to second order in its rounding and in the
// angle of nearly parallel segments, which r2's margin covers); the pairs of
// links nearer than their radii one by one.
template <int T>
__device__ __forceinline__ bool links_hit(const LaneSmem& ls, const float4* __restrict__ sph,
                                          const float2* __restrict__ sa, const float* mine, int stride, int lg) {
  const int general = ls.general;
#pragma unroll 1
  for (int i = lg; i < ls.n_link; i += T) {
    const LinkPair& L = ls.link[i];
    const LanePose A = lane_pose<T>(ls.slot[L.fa], general, mine, stride),
                   B = lane_pose<T>(ls.slot[L.fb], general, mine, stride);
    const int xa = ls.axis[L.fa], xb = ls.axis[L.fb];
    float px, py, pz, ux, uy, uz, qx, qy, qz, vx, vy, vz;
    lane_world(A, xa, L.pa, 1.f, px, py, pz);
    lane_world(A, xa, L.ua, 0.f, ux, uy, uz);
    {
      // the middle of b against segment a: leaves one link in two hundred of
      // the 7-DOF arm at a third of the whole test's work
      float mx, my, mz;
      lane_world(B, xb, L.mb, 1.f, mx, my, mz);
      mx -= px, my -= py, mz -= pz;
      const float t = __saturatef(fmaf(mx, ux, fmaf(my, uy, mz * uz)) * L.inv);
      mx = fmaf(-t, ux, mx), my = fmaf(-t, uy, my), mz = fmaf(-t, uz, mz);
      if (!(fmaf(mx, mx, fmaf(my, my, mz * mz)) < L.m2)) continue;
    }
    lane_world(B, xb, L.pb, 1.f, qx, qy, qz);
    lane_world(B, xb, L.ub, 0.f, vx, vy, vz);
    const float rx = px - qx, ry = py - qy, rz = pz - qz;
    const float uu = fmaf(ux, ux, fmaf(uy, uy, uz * uz)), vv = fmaf(vx, vx, fmaf(vy, vy, vz * vz));
    const float uv = fmaf(ux, vx, fmaf(uy, vy, uz * vz));
    const float ur = fmaf(ux, rx, fmaf(uy, ry, uz * rz)), vr = fmaf(vx, rx, fmaf(vy, ry, vz * rz));
    const float det = fmaf(uu, vv, -uv * uv);
    // from s on the first segment: t the nearest on the second to it, then s to t
    const float iu = uu > 0.f ? __fdividef(1.f, uu) : 0.f, iv = vv > 0.f ? __fdividef(1.f, vv) : 0.f;
    auto squared = [&](float s) {
      const float t = __saturatef(fmaf(s, uv, vr) * iv);
      s = __saturatef(fmaf(t, uv, -ur) * iu);
      const float dx = rx + fmaf(s, ux, -t * vx), dy = ry + fmaf(s, uy, -t * vy), dz = rz + fmaf(s, uz, -t * vz);
      return fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    };
    // Start at the nearest point of the two lines. Nearly parallel segments
    // (an angle a up to 1e-3 by det) are nearest at an end of their overlap,
    // which the two ends of the first lead to, or within (a |u|)^2 / 4 of the
    // squared distance there, a fortieth of r2's margin.
    float d2;
    if (det > 1e-6f * uu * vv) d2 = squared(__saturatef(__fdividef(fmaf(uv, vr, -ur * vv), det)));
    else d2 = fminf(squared(0.f), squared(1.f));
    if (!(d2 < L.r2)) continue;
    for (int j = L.b0; j < L.b0 + L.nb; ++j) {
      const float4 lj = sph[j];
      float cx, cy, cz;
      lane_centre(B, xb, sa[j].x, sph + j, cx, cy, cz);
      for (int k = L.a0; k < L.a0 + L.na; ++k) {
        float ox, oy, oz;
        lane_centre(A, xa, sa[k].x, sph + k, ox, oy, oz);
        if (pair_hit(cx, cy, cz, lj.w, make_float4(ox, oy, oz, sph[k].w))) return true;
      }
    }
  }
  return false;
}

// The listed self pairs one by one, lg, lg + T, ..: where the group has a lane or
// two for each, their one or two links would keep as many lanes busy while the
// others wait. The planar arm's 16 pairs (one link): a round's bisection of 2500
// candidates at sixteen lanes 62 -> 52 us, of 5000 at eight 51 -> 45. In the
// kernels of up to 3 joints; the others' robots have more pairs.
template <int T>
__device__ __forceinline__ bool pairs_hit(const LaneSmem& ls, const float4* __restrict__ sph,
                                          const float2* __restrict__ sa, const int* __restrict__ frame,
                                          const float* mine, int stride, int lg) {
  bool hit = false;
  for (int p = lg; p < ls.n_self; p += T) {
    const ushort2 pr = __ldg(ls.self_pairs + p);
    const int fa = frame[pr.x], fb = frame[pr.y];
    const LanePose A = lane_pose<T>(ls.slot[fa], ls.general, mine, stride),
                   B = lane_pose<T>(ls.slot[fb], ls.general, mine, stride);
    float ax, ay, az, bx, by, bz;
    lane_centre(A, ls.axis[fa], sa[pr.x].x, sph + pr.x, ax, ay, az);
    lane_centre(B, ls.axis[fb], sa[pr.y].x, sph + pr.y, bx, by, bz);
    hit = pair_hit(ax, ay, az, sph[pr.x].w, make_float4(bx, by, bz, sph[pr.y].w)) || hit;
  }
  return hit;
}

// A warp's queue of spheres to test against their cells: the lanes put in
// those that the coarse bound did not free, and 32 at a time are tested, one
// a lane, from their owner's kept pose. Few spheres are left (0.7 of 29 a
// configuration among 64 obstacles), in a few lanes at a time, so each lane
// going through its own cost six passes a warp where this takes one.
// mine, stride: this lane's poses (lane_pose), a group's pitch for T > 1.
constexpr int kNearQueue = 64;  // entries of a warp: sphere | lane << 16
template <int T>
struct NearQueue {
  int* q;
  int count;
  // Tests the first 32 entries; true for a lane one of whose spheres hit.
  __device__ __forceinline__ bool test(const LaneSmem& ls, const float4* __restrict__ sph,
                                       const float2* __restrict__ sa, const int* __restrict__ frame, const EnvDev& e,
                                       const float* mine, int stride) {
    __syncwarp();
    const int lane = threadIdx.x & 31;
    unsigned owner = 0u;
    if (lane < count) {
      const int w = q[lane], s = w & 0xffff, o = w >> 16, f = frame[s];
      const float* theirs = T == 1 ? mine + (o - lane) : mine + (o / T - lane / T) * stride;
      const LanePose P = lane_pose<T>(ls.slot[f], ls.general, theirs, stride);
      float cx, cy, cz;
      lane_centre(P, ls.axis[f], sa[s].x, sph + s, cx, cy, cz);
      if (cell_hit(e, cx, cy, cz, sph[s].w)) owner = 1u << o;
    }
    owner = __reduce_or_sync(0xffffffffu, owner);
    const int left = max(0, count - 32);
    int w = 0;
    if (lane < left) w = q[32 + lane];
    __syncwarp();
    if (lane < left) q[lane] = w;
    count = left;
    return (owner >> lane) & 1u;
  }
  // Adds sphere s of this lane (put = false: none); the warp's lanes together.
  __device__ __forceinline__ void add(bool put, int s) {
    const int lane = threadIdx.x & 31;
    const unsigned m = __ballot_sync(0xffffffffu, put);
    if (put) q[count + __popc(m & ((1u << lane) - 1u))] = s | (lane << 16);
    count += __popc(m);
  }
};

// The chain walked by the T > 1 lanes of a group (each the whole chain, the
// sines and cosines shared), lane 0 keeping the poses. Ends with a warp barrier.
template <int NDOF, int T>
__device__ __forceinline__ void lane_walk(const float (&q)[NDOF], const LaneSmem& ls, float* mine, int stride,
                                          int lg) {
  const int last = ls.last, general = ls.general;
  constexpr int JPL = (NDOF + T - 1) / T;
  float ms[JPL], mc[JPL];
#pragma unroll
  for (int k = 0; k < JPL; ++k) {
    const int jm = lg + k * T;
    float ang = 0.f;
#pragma unroll
    for (int j = 0; j < NDOF; ++j)
      if (j == jm && j < last) ang = fmaf(q[j], ls.joint[2 * j + 1].y, ls.joint[2 * j + 1].x);
    sincosf(ang, &ms[k], &mc[k]);
  }
  LaneChain C;
  C.start();
#pragma unroll
  for (int f = 0; f <= NDOF; ++f) {
    if (f > last) break;
    if (f > 0) {
      const int j = f - 1;
      const float s = __shfl_sync(0xffffffffu, ms[j / T], j % T, T), c = __shfl_sync(0xffffffffu, mc[j / T], j % T, T);
      C.step(ls.joint[2 * j], ls.joint[2 * j + 1], q[j], s, c);
    }
    if (ls.slot[f] >= 0 && lg == 0) lane_keep<T>(C.pose(ls.axis[f]), ls.slot[f], general, mine, stride);
  }
  __syncwarp();
}

// One configuration by a group of T lanes of one warp (T in 1..32). A
// sphere's centre is formed in registers from its frame's pose, looked up in
// the obstacle grid, and formed again where it is needed; only the poses of
// the frames with spheres are stored (collide_group keeps every centre in
// shared memory, which held it to 12 warps an SM), and the self pairs are
// screened link against link. The spheres that a coarse bound does not free go
// through the warp's queue.
// One lane (T = 1): the chain is one rolled loop over the frames, with the
// joint values in mine[j * stride] (unrolled, half the time went to waiting
// for instructions), each frame's spheres taken as it is reached. More lanes:
// every lane walks the unrolled chain (the group shares the sines and
// cosines), lane 0 writes the poses, and the spheres of all frames are dealt
// to the lanes; the rolled form was a quarter slower there, where few warps
// hide its latency.
// All lanes of the warp call it together; returns the group-wide OR.
// Measured at one lane, 7-DOF arm of 40 spheres (kernel time, collide_group at
// its best lane count before): 2e6 labels among 64 obstacles 0.53 -> 0.179 ms,
// of which the chain takes 0.05, the 29 lookups 0.04, the spheres left to
// test 0.03, the links 0.03; 2e5 labels among 1024 obstacles 0.077 -> 0.039
// ms. Bound by instruction issue (73%), 20 warps an SM.
template <int NDOF, int T>
__device__ __forceinline__ bool collide_lane(const float (&q)[NDOF], const LaneSmem& ls,
                                             const float4* __restrict__ sph, const float2* __restrict__ sa,
                                             const int* __restrict__ frame, const EnvDev& e,
                                             const uint8_t* __restrict__ lb, float* mine, int stride, int lg,
                                             int* queue) {
  const ObsGrid& g = e.grid;
  const int last = ls.last, general = ls.general;
  bool hit = false;
  NearQueue<T> nq{queue, 0};
  if constexpr (T == 1) {
    LaneChain C;
    C.start();
    float* poses = mine + ls.n * stride;
#pragma unroll
    for (int j = 0; j < NDOF; ++j)
      if (j < ls.n) mine[j * stride] = q[j];
#pragma unroll 1
    for (int f = 0; f <= last; ++f) {
      if (f > 0) {
        const float4 J = ls.joint[2 * f - 2], K = ls.joint[2 * f - 1];
        const float qj = mine[(f - 1) * stride];
        float s, c;
        sincosf(fmaf(qj, K.y, K.x), &s, &c);
        C.step(J, K, qj, s, c);
      }
      const int s_end = ls.frame_first[f + 1];
      if (ls.slot[f] < 0) continue;
      const int axis = ls.axis[f];
      const LanePose P = C.pose(axis);
      lane_keep<1>(P, ls.slot[f], general, poses, stride);
      // the base frame's spheres before s_first have nothing left to test
#pragma unroll 1
      for (int s0 = f == 0 ? max(ls.frame_first[0], e.s_first) : ls.frame_first[f]; s0 < s_end; s0 += 32) {
        unsigned near = 0u, bit = 1u;
        const int cnt = min(32, s_end - s0);
        if (!g.large) {
#pragma unroll 4
          for (int k = 0; k < cnt; ++k, bit += bit) {
            const float2 a = sa[s0 + k];
            float cx, cy, cz;
            lane_centre(P, axis, a.x, sph + s0 + k, cx, cy, cz);
            if (lane_near<false>(g, lb, cx, cy, cz, __float_as_int(a.y), sph + s0 + k)) near |= bit;
          }
        } else {
#pragma unroll 1
          for (int k = 0; k < cnt; ++k, bit += bit) {
            const float2 a = sa[s0 + k];
            float cx, cy, cz;
            lane_centre(P, axis, a.x, sph + s0 + k, cx, cy, cz);
            if (lane_near<true>(g, lb, cx, cy, cz, __float_as_int(a.y), sph + s0 + k)) near |= bit;
          }
        }
        if (hit) near = 0u;
        while (__any_sync(0xffffffffu, near != 0u)) {
          const bool put = near != 0u;
          nq.add(put, s0 + __ffs(near) - 1);
          near &= near - 1u;
          if (nq.count >= 32 && nq.test(ls, sph, sa, frame, e, poses, stride)) hit = true;
        }
      }
    }
    if (nq.count && nq.test(ls, sph, sa, frame, e, poses, stride)) hit = true;
    if (!hit) hit = links_hit<1>(ls, sph, sa, poses, stride, 0);
  } else {
    lane_walk<NDOF, T>(q, ls, mine, stride, lg);
    const int ns = ls.n_spheres;
#pragma unroll 1
    for (int s1 = e.s_first; s1 < ns; s1 += 32 * T) {
      const int s0 = s1 + lg;
      unsigned near = 0u;
      auto look = [&](int k, auto near_of) {
        const int s = s0 + k * T, f = frame[s];
        const LanePose P = lane_pose<T>(ls.slot[f], general, mine, stride);
        const float2 a = sa[s];
        float cx, cy, cz;
        lane_centre(P, ls.axis[f], a.x, sph + s, cx, cy, cz);
        if (near_of(cx, cy, cz, __float_as_int(a.y), sph + s)) near |= 1u << k;
      };
      const int cnt = min(32, (ns - s0 + T - 1) / T);
      if (!g.large) {
#pragma unroll 2
        for (int k = 0; k < cnt; ++k)
          look(k, [&](float x, float y, float z, int w, const float4* l) { return lane_near<false>(g, lb, x, y, z, w, l); });
      } else {
#pragma unroll 1
        for (int k = 0; k < cnt; ++k)
          look(k, [&](float x, float y, float z, int w, const float4* l) { return lane_near<true>(g, lb, x, y, z, w, l); });
      }
      if (hit) near = 0u;
      while (__any_sync(0xffffffffu, near != 0u)) {
        const bool put = near != 0u;
        nq.add(put, s0 + (__ffs(near) - 1) * T);
        near &= near - 1u;
        if (nq.count >= 32 && nq.test(ls, sph, sa, frame, e, mine, stride)) hit = true;
      }
    }
    if (nq.count && nq.test(ls, sph, sa, frame, e, mine, stride)) hit = true;
    if (NDOF <= 3 && ls.n_self <= 2 * T) {
      if (!hit) hit = pairs_hit<T>(ls, sph, sa, frame, mine, stride, lg);
    } else if (!hit) {
      hit = links_hit<T>(ls, sph, sa, mine, stride, lg);
    }
    unsigned h = hit ? 1u : 0u;
#pragma unroll
    for (int off = 1; off < T; off <<= 1) h |= __shfl_xor_sync(0xffffffffu, h, off, T);
    hit = h != 0u;
    __syncwarp();  // the group's poses may be overwritten
  }
  return hit;
}

// One configuration evaluated by a group of T lanes of one warp (T in 1..32);
// BOX adds the box geometries (robot boxes posed along the chain, pairs with
// a box after the sphere pairs).
// Lane lg of the group computes the centres of spheres s with s % T == lg
// (every lane walks the chain), the group shares them through smem slot
// `cen`, then lane lg tests its spheres against the obstacles through the
// grid (lb: the coarse bounds, in shared or global memory), and the self
// pairs: the work items it % T == lg when the pairs form link blocks and T is
// at most 8, else the listed pairs p % T == lg. Returns the group-wide OR.
// Every lane of the warp must call this together (invalid configurations are
// evaluated and discarded).
template <int NDOF, int T, bool BOX = false>
__device__ __forceinline__ bool collide_group(const float (&q)[NDOF], const RobotSmem& rs,
                                              const float4* __restrict__ sph_s, const EnvDev& env,
                                              const uint8_t* __restrict__ lb,
                                              const ushort2* __restrict__ self_pairs,
                                              const float* __restrict__ self_rr, float4* __restrict__ cen, int lg,
                                              const BoxCtx& bx) {
  fk_group<NDOF, T, BOX>(q, rs, sph_s, cen, lg, bx);
  bool hit = obstacles_hit<T>(rs, sph_s, env, lb, cen, lg);
  // ---- self pairs ----
  if (T <= 8 && rs.n_sblk > 0) {
    // work items (r0, nr, k0, nk) of up to EZO_CH rows, lane lg of the group
    // taking items lg, lg + T, .. (the lanes run the same instructions on
    // their own items); same fast form as the obstacles with the partner's
    // (c_k, r_k) as the obstacle and -hu_k as its offset. The partners go two
    // at a time through packed FP32 FMAs; each half is the scalar fma.rn
    // chain of its pair, and a missing second partner of an odd count gets
    // offset -inf, which no maximum keeps.
    const float Es = rs.E_self;
    for (int it0 = 0; it0 < rs.n_sblk; it0 += T) {
      const int it = it0 + lg;
      const int4 I = it < rs.n_sblk ? rs.sblk[it] : make_int4(0, 0, 0, 0);
      float2 cx[EZO_CH], cy[EZO_CH], cz[EZO_CH], cr[EZO_CH];
      float hu[EZO_CH], m[EZO_CH];
#pragma unroll
      for (int k = 0; k < EZO_CH; ++k) {
        const bool in = k < I.y;
        const float4 c = in ? cen[I.x + k] : make_float4(0.f, 0.f, 0.f, __int_as_float(0x7f800000));
        const float r = in ? sph_s[I.x + k].w : 0.f;
        cx[k] = make_float2(c.x, c.x);
        cy[k] = make_float2(c.y, c.y);
        cz[k] = make_float2(c.z, c.z);
        cr[k] = make_float2(r, r);
        hu[k] = c.w;
        m[k] = -3.0e38f;
      }
      for (int u = 0; 2 * u < I.w; ++u) {
        const int qa = I.z + 2 * u;
        const bool two = 2 * u + 1 < I.w;
        const float4 a = cen[qa];
        const float4 b = two ? cen[qa + 1] : make_float4(0.f, 0.f, 0.f, __int_as_float(0x7f800000));
        const float2 ox = make_float2(a.x, b.x), oy = make_float2(a.y, b.y), oz = make_float2(a.z, b.z);
        const float2 oR = make_float2(sph_s[qa].w, two ? sph_s[qa + 1].w : 0.f);
        const float2 w = make_float2(-a.w, -b.w);
#pragma unroll
        for (int k = 0; k < EZO_CH; ++k) {
          float2 t = __ffma2_rn(cr[k], oR, w);
          t = __ffma2_rn(cz[k], oz, t);
          t = __ffma2_rn(cy[k], oy, t);
          t = __ffma2_rn(cx[k], ox, t);
          m[k] = fmax3f(m[k], t.x, t.y);
        }
      }
      unsigned band = 0u;
#pragma unroll
      for (int k = 0; k < EZO_CH; ++k) {
        const float diff = m[k] - hu[k];
        if (diff > Es) hit = true;
        else if (diff >= -Es) band |= 1u << k;
      }
      while (band) {
        // rounding band: direct differences over the item's partners
        const int k = __ffs(band) - 1;
        band &= band - 1u;
        const float4 c = cen[I.x + k];
        const float r = sph_s[I.x + k].w;
        for (int q = I.z; q < I.z + I.w; ++q) {
          const float4 o = cen[q];
          const float dx = c.x - o.x, dy = c.y - o.y, dz = c.z - o.z;
          const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
          const float sr = r + sph_s[q].w;
          if (d2 < sr * sr) hit = true;
        }
      }
    }
  } else {
    // explicit pair list (direct difference form)
#pragma unroll 4
    for (int p = lg; p < rs.n_self; p += T) {
      const ushort2 pr = self_pairs[p];
      const float4 a = cen[pr.x], b = cen[pr.y];
      const float dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z;
      const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
      if (d2 < self_rr[p]) hit = true;
    }
  }
  // ---- pairs with a box (direct tests; compiled only into the kernels for
  //      scenes with boxes, so sphere-only scenes keep their register budget) ----
  if constexpr (BOX) {
    hit = box_pairs_hit<T>(rs, sph_s, env, lb, cen, lg, bx, hit);
  }
  __syncwarp();
  if (T > 1) {
    unsigned h = hit ? 1u : 0u;
#pragma unroll
    for (int off = 1; off < T; off <<= 1) h |= __shfl_xor_sync(0xffffffffu, h, off, T);
    hit = h != 0u;
  }
  return hit;
}

// v = min(v, |c - o| - r - R) when that is below v: the square root only then.
__device__ __forceinline__ void pair_distance(float cx, float cy, float cz, float r, float4 o, float& v) {
  const float dx = cx - o.x, dy = cy - o.y, dz = cz - o.z;
  const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
  const float lim = r + o.w + v;
  if (lim > 0.f && d2 < lim * lim) v = fminf(v, sqrtf(d2) - r - o.w);
}

// Signed distance min over pairs of |c_i - c_j| - r_i - r_j of one
// configuration by a group of T > 1 lanes, exact below `cap` and equal to cap
// above it. Each lane takes the spheres lg, lg + T, ..: one whose grid cell
// lists candidates is measured against those (the nearest obstacle is among
// them) unless the cell's bound already lies above the lane's best; the others
// keep a lower bound of their distance in bnd[s] (the cell's, or outside the
// grid the one that follows from the distance to its box, which contains
// every obstacle), and while some bound is below the best, the group measures
// the sphere of the smallest one against every obstacle, a few each. Links of
// self pairs are taken sphere by sphere where the other segment's distance
// allows less than the best. Of the 2788 pairs of the 7-DOF arm with 64
// obstacles some 90 are left: 131071 distances 0.416 -> 0.139 ms (one lane a
// configuration over all pairs before), 2000 0.130 -> 0.021; among 1024
// obstacles 131071 7.9 -> 0.88 ms. Bound by instruction issue; the chain is a
// quarter of it.
template <int NDOF, int T>
__device__ __forceinline__ float distance_lane(const float (&q)[NDOF], const LaneSmem& ls,
                                               const float4* __restrict__ sph, const float2* __restrict__ sa,
                                               const int* __restrict__ frame, const EnvDev& e, const WideGrid& w,
                                               float* mine, int stride, float* bnd, int lg, float cap) {
  const ObsGrid& g = e.grid;
  const int general = ls.general, ns = ls.n_spheres;
  lane_walk<NDOF, T>(q, ls, mine, stride, lg);
  float best = cap;
  bool left = false;  // some sphere of this lane keeps a bound
  // from the arm's tip: where the spheres near the obstacles usually are
  for (int s = ns - 1 - lg; s >= 0 && e.n_obs > 0; s -= T) {
    const int f = frame[s];
    const LanePose P = lane_pose<T>(ls.slot[f], general, mine, stride);
    const float r = sph[s].w;
    float cx, cy, cz;
    lane_centre(P, ls.axis[f], sa[s].x, sph + s, cx, cy, cz);
    unsigned long long d = (unsigned long long)kGridAll << 8;
    const uint16_t* ids = g.ids;
    float unit = w.step, out2 = 0.f;
    bool in = true;
    float ux = __fmaf_rd(cx, g.finv, g.fx), uy = __fmaf_rd(cy, g.finv, g.fy), uz = __fmaf_rd(cz, g.finv, g.fz);
    if (ux >= kGridBias && uy >= kGridBias && uz >= kGridBias && ux < g.ex && uy < g.ey && uz < g.ez) {
      const unsigned ix = __float_as_uint(ux) & 0xffu, iy = __float_as_uint(uy) & 0xffu, iz = __float_as_uint(uz) & 0xffu;
      d = __ldg(g.cell + ((((iz << g.fbits) + iy) << g.fbits) + ix));
      unit = g.step;
    } else {
      // the wide grid's cell, or that of the projection onto it
      ux = __fmaf_rd(cx, w.inv, w.fx), uy = __fmaf_rd(cy, w.inv, w.fy), uz = __fmaf_rd(cz, w.inv, w.fz);
      const float ox = fmaxf(fmaxf(w.lx - cx, cx - w.hx), 0.f), oy = fmaxf(fmaxf(w.ly - cy, cy - w.hy), 0.f),
                  oz = fmaxf(fmaxf(w.lz - cz, cz - w.hz), 0.f);
      in = ux >= kGridBias && uy >= kGridBias && uz >= kGridBias && ux < w.ex && uy < w.ey && uz < w.ez;
      if (!in) out2 = fmaf(ox, ox, fmaf(oy, oy, oz * oz));
      const unsigned ix = __float_as_uint(fminf(fmaxf(ux, kGridBias), w.ex - 1.f)) & 0x1fu,
                     iy = __float_as_uint(fminf(fmaxf(uy, kGridBias), w.ey - 1.f)) & 0x1fu,
                     iz = __float_as_uint(fminf(fmaxf(uz, kGridBias), w.ez - 1.f)) & 0x1fu;
      const unsigned i = (iz * kGridC + iy) * kGridC + ix;
      if (w.cell) d = __ldg(w.cell + i);
      else d |= (unsigned long long)__ldg(g.lb + i);
      ids = w.ids;
    }
    const unsigned kind = (unsigned)(d >> 8) & 0xffu, lb = (unsigned)(d & 0xffu);
    // from the centre's projection p onto the box: |x - o|^2 >= |x - p|^2 +
    // |p - o|^2 and |p - o| >= lb + R, least for the largest R (a bound of 0
    // may stand for a negative one)
    const float m = fmaf((float)lb, unit, w.r_obs);
    float b = -3.0e38f;
    if (out2 > 0.f) b = sqrtf(fmaf(m, m, out2)) * 0.999999f - w.r_obs - r;
    else if (in && lb) b = (float)lb * unit - r;
    if (b < best && in && kind != kGridAll) {
      const bool list = kind == kGridList;
      const int cnt = list ? (int)((d >> 16) & 0xffffu) : (int)kind;
      ids += list ? (unsigned)(d >> 32) : 0u;
#pragma unroll 2
      for (int k = 0; k < cnt; ++k) {
        const unsigned id = list ? (unsigned)__ldg(ids + k) : (unsigned)(d >> (16 + 12 * k)) & 0xfffu;
        pair_distance(cx, cy, cz, r, __ldg(e.obs + id), best);
      }
      b = 3.0e38f;
    }
    bnd[s] = b;
    left = left || b < best;
  }
  // the group's best, then the spheres that are left by their bounds
#pragma unroll
  for (int o = 1; o < T; o <<= 1) best = fminf(best, __shfl_xor_sync(0xffffffffu, best, o, T));
  while (__any_sync(0xffffffffu, left)) {
    float b = 3.0e38f;
    int s = 0;
    for (int k = ns - 1 - lg; k >= 0 && e.n_obs > 0; k -= T)
      if (bnd[k] < b) b = bnd[k], s = k;
#pragma unroll
    for (int o = 1; o < T; o <<= 1) {
      const float b2 = __shfl_xor_sync(0xffffffffu, b, o, T);
      const int s2 = __shfl_xor_sync(0xffffffffu, s, o, T);
      if (b2 < b || (b2 == b && s2 < s)) b = b2, s = s2;
    }
    const bool go = b < best;  // the same in the whole group
    if (!__any_sync(0xffffffffu, go)) break;
    if (go) {
      const int f = frame[s];
      const LanePose P = lane_pose<T>(ls.slot[f], general, mine, stride);
      const float r = sph[s].w;
      float cx, cy, cz;
      lane_centre(P, ls.axis[f], sa[s].x, sph + s, cx, cy, cz);
#pragma unroll 4
      for (int j = lg; j < e.n_obs; j += T) pair_distance(cx, cy, cz, r, __ldg(e.obs + j), best);
      if ((ns - 1 - s) % T == lg) bnd[s] = 3.0e38f;
    }
#pragma unroll
    for (int o = 1; o < T; o <<= 1) best = fminf(best, __shfl_xor_sync(0xffffffffu, best, o, T));
  }
  // self pairs
  for (int i = 0; i < ls.n_link; ++i) {
    const LinkPair& L = ls.link[i];
    const LanePose A = lane_pose<T>(ls.slot[L.fa], general, mine, stride),
                   B = lane_pose<T>(ls.slot[L.fb], general, mine, stride);
    const int xa = ls.axis[L.fa], xb = ls.axis[L.fb];
    float px, py, pz, ux, uy, uz;
    lane_world(A, xa, L.pa, 1.f, px, py, pz);
    lane_world(A, xa, L.ua, 0.f, ux, uy, uz);
    for (int j = L.b0 + lg; j < L.b0 + L.nb; j += T) {
      const float4 lj = sph[j];
      float cx, cy, cz;
      lane_centre(B, xb, sa[j].x, sph + j, cx, cy, cz);
      // this sphere against the other run's segment
      const float mx = cx - px, my = cy - py, mz = cz - pz;
      const float t = __saturatef(fmaf(mx, ux, fmaf(my, uy, mz * uz)) * L.inv);
      const float ex = fmaf(-t, ux, mx), ey = fmaf(-t, uy, my), ez = fmaf(-t, uz, mz);
      const float lim = best + lj.w + L.ra;
      if (!(lim > 0.f && fmaf(ex, ex, fmaf(ey, ey, ez * ez)) < lim * lim)) continue;
      for (int k = L.a0; k < L.a0 + L.na; ++k) {
        const float rk = sph[k].w;
        float ox, oy, oz;
        lane_centre(A, xa, sa[k].x, sph + k, ox, oy, oz);
        // the earlier sphere's radius first, as the pair list has them
        if (k < j) pair_distance(ox, oy, oz, rk, make_float4(cx, cy, cz, lj.w), best);
        else pair_distance(cx, cy, cz, lj.w, make_float4(ox, oy, oz, rk), best);
      }
    }
  }
#pragma unroll
  for (int o = 1; o < T; o <<= 1) best = fminf(best, __shfl_xor_sync(0xffffffffu, best, o, T));
  __syncwarp();  // the group's poses and bounds may be overwritten
  return best;
}

// Shared-memory image of an obstacle set for signed_distance_one, in pairs of
// spheres (2p, 2p + 1): obs_s[2p] = (x_2p, x_2p+1, y_2p, y_2p+1), obs_s[2p + 1] =
// (z_2p, z_2p+1, R_2p, R_2p+1); n_obs_pad is even. Read as four words a sphere
// the loop over the obstacles is 6 to 14% faster than with a sphere a float4 (12
// joints, 400000 among 200 spheres: 1.57 against 1.70 ms).
__device__ __forceinline__ void stage_obs(float4* obs_s, const EnvDev& e) {
  for (int p = threadIdx.x; p < e.n_obs_pad / 2; p += blockDim.x) {
    const float4 a = e.obs[2 * p], b = e.obs[2 * p + 1];
    obs_s[2 * p] = make_float4(a.x, b.x, a.y, b.y);
    obs_s[2 * p + 1] = make_float4(a.z, b.z, a.w, b.w);
  }
}
__device__ __forceinline__ float4 obs_at(const float4* __restrict__ obs_s, int j) {
  const float* A = reinterpret_cast<const float*>(obs_s + (j & ~1));
  const int h = j & 1;
  return make_float4(A[h], A[2 + h], A[4 + h], A[6 + h]);
}

// Signed distance min over pairs of ||c_i - c_j|| - r_i - r_j for one
// configuration, one lane per configuration, exact below `cap` and equal to
// cap above it (a pair whose squared distance is at least (r_i + r_j + cap)^2
// cannot bring the minimum below cap, so its square root is skipped).
template <int NDOF>
__device__ float signed_distance_one(const float* __restrict__ q, const RobotSmem& rs,
                                     const float4* __restrict__ sph_s, const float4* __restrict__ obs_s,
                                     int n_obs, const ushort2* __restrict__ self_pairs,
                                     const float* __restrict__ self_rr, float4* __restrict__ cen,
                                     float cap) {
  float c0x = 1.f, c0y = 0.f, c0z = 0.f, c1x = 0.f, c1y = 1.f, c1z = 0.f, c2x = 0.f, c2y = 0.f, c2z = 1.f;
  float px = 0.f, py = 0.f, pz = 0.f;
  const int n = rs.n;
#pragma unroll
  for (int f = 0; f <= NDOF; ++f) {
    if (f > n) break;
    if (f > 0) {
      const int j = f - 1;
      float s, c;
      sincosf(fmaf(q[j], rs.kth[j], rs.toff[j]), &s, &c);
      const float n0x = fmaf(c, c0x, s * c1x), n0y = fmaf(c, c0y, s * c1y), n0z = fmaf(c, c0z, s * c1z);
      const float n1x = fmaf(c, c1x, -s * c0x), n1y = fmaf(c, c1y, -s * c0y), n1z = fmaf(c, c1z, -s * c0z);
      const float aj = rs.a[j], dj = fmaf(q[j], rs.kd[j], rs.d[j]);
      px = fmaf(aj, n0x, fmaf(dj, c2x, px));
      py = fmaf(aj, n0y, fmaf(dj, c2y, py));
      pz = fmaf(aj, n0z, fmaf(dj, c2z, pz));
      const float ca = rs.ca[j], sa = rs.sa[j];
      const float m1x = fmaf(ca, n1x, sa * c2x), m1y = fmaf(ca, n1y, sa * c2y), m1z = fmaf(ca, n1z, sa * c2z);
      const float m2x = fmaf(ca, c2x, -sa * n1x), m2y = fmaf(ca, c2y, -sa * n1y), m2z = fmaf(ca, c2z, -sa * n1z);
      c0x = n0x; c0y = n0y; c0z = n0z;
      c1x = m1x; c1y = m1y; c1z = m1z;
      c2x = m2x; c2y = m2y; c2z = m2z;
    }
    for (int s = rs.frame_first[f]; s < rs.frame_first[f + 1]; ++s) {
      const float4 l = sph_s[s];
      cen[s] = make_float4(fmaf(c0x, l.x, fmaf(c1x, l.y, fmaf(c2x, l.z, px))),
                           fmaf(c0y, l.x, fmaf(c1y, l.y, fmaf(c2y, l.z, py))),
                           fmaf(c0z, l.x, fmaf(c1z, l.y, fmaf(c2z, l.z, pz))), l.w);
    }
  }
  float best = cap;
  for (int s = 0; s < rs.n_spheres; ++s) {
    const float4 c = cen[s];
    for (int j = 0; j < n_obs; ++j) {
      const float4 o = obs_at(obs_s, j);
      const float dx = c.x - o.x, dy = c.y - o.y, dz = c.z - o.z;
      const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
      const float lim = c.w + o.w + best;
      if (lim > 0.f && d2 < lim * lim) best = fminf(best, sqrtf(d2) - c.w - o.w);
    }
  }
  for (int p = 0; p < rs.n_self; ++p) {
    const ushort2 pr = self_pairs[p];
    const float4 a = cen[pr.x], b = cen[pr.y];
    const float dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z;
    const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    const float lim = a.w + b.w + best;
    if (lim > 0.f && d2 < lim * lim) best = fminf(best, sqrtf(d2) - a.w - b.w);
  }
  return best;
}

}  // namespace ezo
