// Rotational transport of small lattices: MacCormack and several FTCS sub-steps
// of a 3-D tile in one launch.
#pragma once

#include "rpk_kernels.cuh"

namespace rpk {

// The passes of a small lattice are launch after launch of kernels that wait for
// each other and for L2 (3.5 us each, whatever they compute), so a block takes a
// tile of one sublattice with a halo deep enough for all passes of the launch and
// recomputes the halo: the predictor costs the tile one layer at its high side,
// the corrector one at its low side, every sub-step one at both. What neighbours
// need lies in shared memory; what only a point itself needs (e, theta_R = a e + c,
// the six face coefficients) stays in registers. A thread takes the same (x, y) of
// kP planes, so that its indices, its x and y neighbours' offsets and its boundary
// are found once.
//   halo axis       the region is the tile and the halo; the layers that a pass
//                   cannot compute hold values that the tile never uses
//   whole periodic  the region is the axis, neighbours wrap
//   walls, ends     the region holds the layer beyond them: constant values at
//                   every stage (a wall's distance goes into the face coefficient)
// 32^3, one sub-step: a step of 13.8 us became 10.0. 128 x 64 x 8 between walls, five
// sub-steps: 33.5 us became 23.2, two kernels before three of this. Bound: launches
// and the latency of its phases; issue takes 2 us of the 5.5 us at 32^3. Indices found
// per point, with spare layers instead of wrapped neighbours: 12.1 and 28.2 us.
constexpr int kBrickThreads = 512;
constexpr int kBrickMaxP = 6;   // most planes of a thread
constexpr int kBrickArrays = 6;
constexpr int kBrickSub = 8;    // most sub-steps of a launch
constexpr size_t kBrickSmem = sizeof(float) * kBrickArrays * kBrickThreads * kBrickMaxP;

struct BrickArgs {
  FastDiv by_tx, by_ty;   // tiles along x and y
  FastDiv by_X, by_area;  // region: x extent, points of a plane
  int tx, ty;
  int own[3];   // points of a tile
  int ext[3];   // points of its region
  int halo[3];  // 0 on a whole periodic axis
  int groups;   // planes taken at once: a thread's planes are this far apart
  int open;     // 1 reservoirs, kWallX, kWallY
  int nsub;
};

template <bool kFirst, int kP>
__global__ void __launch_bounds__(kBrickThreads)
    k_brick_transport(StepConst<float> K, BrickArgs B, const float* e, const float* ucur,
                      const float* uprev, const float* drho, const float* kap,
                      float* __restrict__ e_next, const float* __restrict__ ghost) {
  // places in shared memory and cells in bytes, arrays a constant stride apart: one
  // address for all of them
  extern __shared__ __align__(16) unsigned char brick_smem[];
  constexpr int kStride = sizeof(float) * kBrickThreads * kP;
  enum { kS0 = 0, kS1 = 1, kV = 2, kKap = 5 };  // e, then theta_R; predicted e, then theta_R; velocity; kappa_R
  auto sm = [&](int array, int at) -> float& { return *reinterpret_cast<float*>(brick_smem + array * kStride + at); };
  const int X = B.ext[0], Z = B.ext[2], area = X * B.ext[1];
  // first point of the tile and of the region along each axis
  const unsigned b = blockIdx.x, tyz = B.by_tx.div(b), tz = B.by_ty.div(tyz);
  const int t0[3] = {(int)(b - tyz * B.tx) * B.own[0], (int)(tyz - tz * B.ty) * B.own[1], (int)tz * B.own[2]};
  const int nn[2] = {K.nx, K.ny};
  const bool open[2] = {(B.open & (1 | kWallX)) != 0, (B.open & kWallY) != 0};
  const int zg = (int)B.by_area.div(threadIdx.x), xy = threadIdx.x - zg * area, ry = (int)B.by_X.div(xy);
  const int r[2] = {xy - ry * X, ry};
  bool own = true, live = true;
  const float* gh = nullptr;
  int g[2], lo[2], hi[2];  // position, offsets of the low and high neighbour
  unsigned wall = 0;       // faces on a wall: bit 2 axis + (1: high side)
  const int step[2] = {(int)sizeof(float), X * (int)sizeof(float)};
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const int r0 = open[a] ? min(max(t0[a] - B.halo[a], -1), nn[a] + 1 - B.ext[a]) : t0[a] - B.halo[a];
    g[a] = r0 + r[a];
    own = own && g[a] >= t0[a] && g[a] < min(t0[a] + B.own[a], nn[a]);
    const int wrap = B.halo[a] == 0 ? (B.ext[a] - 1) * step[a] : 0;
    lo[a] = r[a] > 0 ? -step[a] : wrap;
    hi[a] = r[a] < B.ext[a] - 1 ? step[a] : -wrap;
    if (open[a]) {
      if (g[a] < 0 || g[a] >= nn[a]) {
        live = false;
        gh = ghost + ((g[a] < 0 ? 0 : 1) + (a == 0 && !(B.open & 1) ? 2 : 0)) * kGhostStride;
      }
      if (!(B.open & 1)) wall |= (g[a] == 0 ? 1u << (2 * a) : 0u) | (g[a] == nn[a] - 1 ? 2u << (2 * a) : 0u);
    } else {
      g[a] = g[a] < 0 ? g[a] + nn[a] : g[a] >= nn[a] ? g[a] - nn[a] : g[a];
    }
  }
  if (zg >= B.groups) return;  // less than a warp of threads
  // planes beyond the region (Z is padded to groups x kP) are computed and not used
  const int zstep = (int)sizeof(float) * area, istep = B.groups * zstep;
  const int i0 = zg * zstep + (int)sizeof(float) * xy;  // place of plane k: i0 + k istep
  const int zwrap = B.halo[2] == 0 ? (Z - 1) * zstep : 0;
  unsigned cell[kP];
  int zlo[kP], zhi[kP];
#pragma unroll
  for (int k = 0; k < kP; ++k) {
    const int rz = zg + k * B.groups;
    int z = t0[2] - B.halo[2] + rz;
    z = z < 0 ? z + K.nz : z >= K.nz ? z - K.nz : z;
    cell[k] = rz < Z && live ? sizeof(float) * ((z * K.ny + g[1]) * K.nx + g[0]) : 0u;
    zlo[k] = rz > 0 ? -zstep : zwrap;
    zhi[k] = rz < Z - 1 ? zstep : -zwrap;
  }
  pdl_wait();
  auto ld = [](const float* base, unsigned at) { return *reinterpret_cast<const float*>(reinterpret_cast<const char*>(base) + at); };
  const int64_t plane = blockIdx.y * K.n3;
  float ev[kP], kp[kP], dr[kP], v[kP][3], ep[kP];
#pragma unroll
  for (int k = 0; k < kP; ++k) {
    ev[k] = ld(e + plane, cell[k]);
    kp[k] = ld(kap + plane, cell[k]);
    dr[k] = ld(drho + plane, cell[k]);
    if (kFirst) {
#pragma unroll
      for (int a = 0; a < 3; ++a)
        v[k][a] = 1.5f * ld(ucur + plane + 2 * a * K.n3, cell[k]) - 0.5f * ld(uprev + plane + 2 * a * K.n3, cell[k]);
    }
  }
  if (gh) {
#pragma unroll
    for (int k = 0; k < kP; ++k) {
      ev[k] = gh[kGhE];
      kp[k] = gh[kGhKap];
      dr[k] = gh[kGhDrho];
#pragma unroll
      for (int a = 0; a < 3; ++a) v[k][a] = gh[kGhU + a];
    }
  }
#pragma unroll
  for (int k = 0; k < kP; ++k) {
    const int i = i0 + k * istep;
    sm(kKap, i) = kp[k];
    if (kFirst) {
      sm(kS0, i) = ev[k];
#pragma unroll
      for (int a = 0; a < 3; ++a) sm(kV + a, i) = v[k][a];
    }
  }
  __syncthreads();
  if (kFirst) {
#pragma unroll
    for (int k = 0; k < kP; ++k) {
        const int i = i0 + k * istep, q[3] = {i + hi[0], i + hi[1], i + zhi[k]};
      float div = 0.f;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const float vp = v[k][a], vq = sm(kV + a, q[a]), eq = sm(kS0, q[a]);
        div += K.E0 * (vq - vp) + (eq * vq - ev[k] * vp);
      }
      ep[k] = live ? ev[k] - K.dt * div : ev[k];
      sm(kS1, i) = ep[k];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kP; ++k) {
        const int i = i0 + k * istep, q[3] = {i + lo[0], i + lo[1], i + zlo[k]};
      float div = 0.f;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const float vp = v[k][a], vq = sm(kV + a, q[a]), eq = sm(kS1, q[a]);
        div += K.E0 * (vp - vq) + (ep[k] * vp - eq * vq);
      }
      if (live) ev[k] = 0.5f * (ev[k] + ep[k] - K.dt * div);
    }
  }
  const float t0d = K.delta * K.theta0;
  float ca[kP], cc[kP], th[kP], face[kP][6];
#pragma unroll
  for (int k = 0; k < kP; ++k) {
    const int i = i0 + k * istep, q[6] = {i + lo[0], i + hi[0], i + lo[1], i + hi[1], i + zlo[k], i + zhi[k]};
    const float inv = 1.f / (K.delta * (1.f + dr[k]));
    ca[k] = 2.f * inv;
    cc[k] = -t0d * dr[k] * inv;
    th[k] = fmaf(ca[k], ev[k], cc[k]);
    sm(kS0, i) = th[k];
#pragma unroll
    for (int f = 0; f < 6; ++f) face[k][f] = live ? (K.hsub * 0.5f) * (kp[k] + sm(kKap, q[f])) : 0.f;
  }
  if (wall && live) {
    // a wall lies 1/4 or 3/4 from the point: kappa_R (theta_w - theta_R) / d, kappa_R
    // of the point
#pragma unroll
    for (int k = 0; k < kP; ++k)
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        const bool near = ((f & 1) == 0) == (blockIdx.y == 0);
        if ((wall >> f) & 1u) face[k][f] = K.hsub * kp[k] * (near ? 4.f : 4.f / 3.f);
      }
  }
  __syncthreads();
  int from = 0, to = kStride;  // kS0, kS1
  for (int j = B.nsub; j > 0; --j) {
#pragma unroll
    for (int k = 0; k < kP; ++k) {
        const int i = i0 + k * istep, j0 = i + from, q[6] = {j0 + lo[0], j0 + hi[0], j0 + lo[1], j0 + hi[1], j0 + zlo[k], j0 + zhi[k]};
#pragma unroll
      for (int f = 0; f < 6; ++f) ev[k] = fmaf(face[k][f], sm(0, q[f]) - th[k], ev[k]);
      th[k] = fmaf(ca[k], ev[k], cc[k]);
      if (j > 1) sm(0, i + to) = th[k];
    }
    if (j > 1) __syncthreads();
    from = to;
    to = kStride - to;
  }
  if (own) {
    char* const out = reinterpret_cast<char*>(e_next + plane);
#pragma unroll
    for (int k = 0; k < kP; ++k) {
      const int rz = zg + k * B.groups, z = rz - B.halo[2];
      if (rz < Z && z >= 0 && z < B.own[2] && t0[2] + z < K.nz) *reinterpret_cast<float*>(out + cell[k]) = ev[k];
    }
  }
}

}  // namespace rpk
