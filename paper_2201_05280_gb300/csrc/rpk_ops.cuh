// Kernel launch sequences of one precision (included by rpk_ops_<prec>.cu,
// which instantiate Ops<Store, Real> for their storage type).
#pragma once

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "rpk_internal.h"
#include "rpk_brick.cuh"

namespace rpk {

// Per-launch constants of the step (Sec. 5) for relaxation parameters r on an
// nx x ny x nz grid with nsub FTCS sub-steps; computed in double, then cast.
template <typename Real>
static StepConst<Real> make_step_const(const rpk_relax& r, int nsub, int nx, int ny, int nz,
                                       int paper = 0) {
  const double tau_s = 1.0 / (1.0 / r.tau + 1.0 / r.tau1);
  const double beta = r.dt / (2.0 * tau_s + r.dt);
  const double B = 1.0 + r.tau / r.tau1;
  StepConst<Real> K;
  K.nx = nx;
  K.ny = ny;
  K.nz = nz;
  K.n3 = (int64_t)nx * ny * nz;
  K.by_nx = FastDiv((unsigned)nx);
  K.by_ny = FastDiv((unsigned)ny);
  K.by_nxp = FastDiv((unsigned)std::max(1, nx / 2));
  K.theta0 = Real(kTheta0);
  K.c_keep = Real(1.0 - 2.0 * beta);
  K.c_relax = Real(2.0 * beta);
  K.beta = Real(beta);
  K.w_es = Real(tau_s / r.tau);
  K.w_eq = Real(tau_s / r.tau1);
  K.b = Real(r.b);
  K.inv_sig = Real(1.0 / (1.0 + r.dt / (2.0 * tau_s) - r.b * r.dt / (2.0 * r.tau)));
  K.inv_d = Real(1.0 / (1.0 + r.dt / (2.0 * r.tau1)));
  K.delta = Real(r.delta);
  K.inv_3pd = Real(1.0 / (3.0 + r.delta));
  K.exc = Real(r.dt * r.delta / (2.0 * r.tau1));
  K.kapc = Real(r.k_r * 5.0 * r.tau / (2.0 * B));
  K.E0 = Real(0.5 * r.delta * kTheta0);
  const double i1 = 1.0 / kTheta0, cr = 2.0 * beta;
  K.spare = Real(0);
  K.two_id = Real(2.0 / r.delta);
  K.c_d = Real(r.delta / (3.0 + r.delta));
  K.c_3 = Real(3.0 / (3.0 + r.delta));
  K.bsig = Real(tau_s / r.tau * r.b / (1.0 + r.dt / (2.0 * tau_s) - r.b * r.dt / (2.0 * r.tau)));
  K.q1h = Real(0.5 * cr * i1);
  K.q1 = Real(cr * i1);
  K.q2h = Real(0.5 * cr * i1 * i1);
  K.q2 = Real(cr * i1 * i1);
  K.q36 = Real(cr * i1 * i1 * i1 / 6.0);
  K.q32 = Real(0.5 * cr * i1 * i1 * i1);
  K.q3 = Real(cr * i1 * i1 * i1);
  K.dt = Real(r.dt);
  K.hsub = Real(r.dt / std::max(1, nsub));
  const double X = 3.0 * r.dt / (2.0 * r.tau1 * (3.0 + r.delta));
  K.paper = paper;
  K.ra_keep = Real(1.0 / (1.0 + X));
  K.ra_t = Real(X / (1.0 + X));
  K.pa = Real(r.delta * X / 3.0);
  K.inv_1pa = Real(1.0 / (1.0 + r.delta * X / 3.0));
  return K;
}

template <typename Real>
static StepConst<Real> make_const(const rpk_lattice* L) {
  return make_step_const<Real>(L->relax, L->nsub, L->grid.nx, L->grid.ny, L->grid.nz, L->rot_mode);
}

// Threads per block for n points or pairs per sublattice: 128, or fewer (down
// to one warp) while the two sublattices' blocks would leave SMs without one.
static inline int block_for(const rpk_lattice* L, int64_t n) {
  int b = 128;
  while (b > 32 && 2 * ((n + b - 1) / b) < L->sms) b /= 2;
  return b;
}

// Launch shape of a kernel with one point (n = n3) or pair (n = n3 / 2) per thread.
struct PointLaunch {
  dim3 grid;
  int block;
  PointLaunch(const rpk_lattice* L, int64_t n)
      : grid((unsigned)((n + block_for(L, n) - 1) / block_for(L, n)), 2), block(block_for(L, n)) {}
};

static inline rpk_status check_launch(const char* what) {
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) return cuda_fail(err, what);
  return RPK_OK;
}

// FP64 lattices of at most two warps of points per SM: four warps share each
// (k_collide_split; steps, us, a thread per point / split: 2000 cells 23.7 / 18.6, 4864
// cells 26.7 / 24.7, 5500 cells, three warps on some SMs, 28.8 / 31.1; 12^3 35.0 / 28.7,
// 20^3 37.0 / 47.2).
static inline bool split_groups(const rpk_lattice* L) {
  return L->store_elem == 8 && 2 * ((L->n3 + 31) / 32) <= 2 * (int64_t)L->sms;
}

// Launch a kernel of the step so that its blocks may become resident while the
// previous kernel of the stream still runs (it waits in pdl_wait): 32^3 FP32 21.4
// -> 17.4 us a step of four kernels. Larger FP64 lattices keep ordinary launches: their
// pipe is the bound, and blocks placed beside a running kernel's share SMs that would
// otherwise have had fewer (ordinary / overlapping, us a step: 1000 cells 16.5 / 13.1,
// 12^3 28.8 / 25.1, 20^3 with 8 sub-steps 80 / 60, 26^3 59.5 / 52.6; but 36^3 125 / 136
// and, one thread a point of a line, 5500 cells 28.8 / 38.1).
static inline bool overlap_launches(const rpk_lattice* L) {
  return L->real_elem == 4 || split_groups(L) || (L->grid.ny * L->grid.nz > 1 && L->n3 <= 128 * (int64_t)L->sms);
}

template <typename... KArgs, typename... Args>
static void launch_step(rpk_lattice* L, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, Args... args) {
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = L->stream;
  cudaLaunchAttribute a{};
  a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &a;
  c.numAttrs = overlap_launches(L) && !L->apart ? 1 : 0;
  cudaLaunchKernelEx(&c, kernel, static_cast<KArgs>(args)...);
}

// Walls in use: kWallY and / or kWallX.
static inline int wall_mask(const rpk_lattice* L) {
  return (L->walls ? kWallY : 0) | (L->xwalls ? kWallX : 0);
}

// rho_w - 1 of every wall column from the current (post-collision)
// populations; precedes every pull when walls are on.
template <typename Store, typename Real, int kBC>
static rpk_status wall_launch_t(rpk_lattice* L, const StepConst<Real>& K) {
  const int64_t n = ((kBC & kWallY) ? 2 * (int64_t)L->grid.nx * L->grid.nz : 0) +
                    ((kBC & kWallX) ? 2 * (int64_t)L->grid.ny * L->grid.nz : 0);
  launch_step(L, k_wall_rho<Store, Real, kBC>, (unsigned)((n + 31) / 32), 32, 0, K, static_cast<const Store*>(L->pop[L->cur]), static_cast<const Real*>(L->ghost),
      static_cast<Real*>(L->wrho));
  return check_launch("k_wall_rho");
}

template <typename Store, typename Real>
static rpk_status wall_launch(rpk_lattice* L, const StepConst<Real>& K) {
  switch (wall_mask(L)) {
    case kWallY: return wall_launch_t<Store, Real, kWallY>(L, K);
    case kWallX: return wall_launch_t<Store, Real, kWallX>(L, K);
    default: return wall_launch_t<Store, Real, kWallY | kWallX>(L, K);
  }
}

template <typename Store, typename Real, bool kPull, int kBC>
static rpk_status collide_launch(rpk_lattice* L, const StepConst<Real>& K) {
  const Store* pin = static_cast<const Store*>(L->pop[L->cur]);
  Store* pout = static_cast<Store*>(L->pop[L->cur ^ 1]);
  Real* ucur = static_cast<Real*>(L->u[L->steps & 1]);
  const Real* wcol = static_cast<const Real*>(L->wrho);
  const PointLaunch pt(L, L->n3);
  if constexpr (std::is_same<Store, double>::value) {
    if (split_groups(L)) {
      const dim3 grid((unsigned)((L->n3 + 31) / 32), 2);
      launch_step(L, L->rot_mode ? k_collide_split<kPull, kBC, true> : k_collide_split<kPull, kBC, false>, grid, 128, 0, K,
                  pin, pout, static_cast<const Real*>(L->e), static_cast<Real*>(L->e_star), static_cast<Real*>(L->drho),
                  ucur, static_cast<Real*>(L->kap), static_cast<const Real*>(L->ghost), L->status,
                  L->rot_mode ? static_cast<Real*>(L->thbuf) : nullptr, wcol);
      return check_launch("k_collide_split");
    }
  }
  if (L->rot_mode) {
    if constexpr (kPull && kBC == 0 && sizeof(Real) == 4) {
      if (L->grid.nx % 2 == 0) {
        // two x-adjacent points per thread, packed FP32x2 arithmetic
        const PointLaunch at(L, L->n3 / 2);
        launch_step(L, k_collide_pair<Store, true>, at.grid, at.block, 0, K, pin, pout, static_cast<const Real*>(L->e), static_cast<Real*>(L->e_star),
            static_cast<Real*>(L->drho), ucur, static_cast<Real*>(L->kap), L->status,
            static_cast<Real*>(L->thbuf));
        return check_launch("k_collide_pair");
      }
    }
    launch_step(L, k_collide<Store, Real, kPull, kBC, true>, pt.grid, pt.block, 0, K, pin, pout, static_cast<const Real*>(L->e), static_cast<Real*>(L->e_star),
        static_cast<Real*>(L->drho), ucur, static_cast<Real*>(L->kap),
        static_cast<const Real*>(L->ghost), L->status, static_cast<Real*>(L->thbuf), wcol);
    return check_launch("k_collide");
  }
  if constexpr (kPull && kBC == 0 && sizeof(Real) == 4) {
    if (L->grid.nx % 2 == 0) {
      // two x-adjacent points per thread, packed FP32x2 arithmetic
      const PointLaunch at(L, L->n3 / 2);
      launch_step(L, k_collide_pair<Store, false>, at.grid, at.block, 0, K, pin, pout, static_cast<const Real*>(L->e), static_cast<Real*>(L->e_star),
          static_cast<Real*>(L->drho), ucur, static_cast<Real*>(L->kap), L->status, nullptr);
      return check_launch("k_collide_pair");
    }
  }
  launch_step(L, k_collide<Store, Real, kPull, kBC, false>, pt.grid, pt.block, 0, K, pin, pout, static_cast<const Real*>(L->e), static_cast<Real*>(L->e_star),
      static_cast<Real*>(L->drho), ucur, static_cast<Real*>(L->kap),
      static_cast<const Real*>(L->ghost), L->status, nullptr, wcol);
  return check_launch("k_collide");
}

// Transport of a quasi-1-D lattice: nsub sub-steps in equal parts of at most
// kLineSub, the first part with the MacCormack passes; returns the launches.
// Tiles of 64 points while that leaves no more tiles than SMs (FP64 issues two
// lanes per cycle and SM, so narrow tiles on every SM beat wide ones on a
// few), else 128.
template <typename Real, int kBC>
static int line_launches(rpk_lattice* L, const StepConst<Real>& K, const Real* es, const Real* ucur,
                         const Real* uprev, const Real* drho, const Real* kap, Real* e, Real* ea, Real* eb,
                         const Real* gh) {
  const int parts = (L->nsub + kLineSub - 1) / kLineSub;
  const Real* src = es;
  for (int i = 0, done = 0; i < parts; ++i) {
    const int m = (L->nsub - done + parts - i - 1) / (parts - i);
    const int halo = 2 * (m + (i == 0 ? 1 : 0));
    const int tile = 2 * ((L->grid.nx + 63 - halo) / (64 - halo)) <= L->sms ? 64 : 128;
    const dim3 grid((unsigned)((L->grid.nx + tile - halo - 1) / (tile - halo)), 2);
    const size_t smem = 2 * tile * sizeof(Real);
    Real* dst = i == parts - 1 ? e : (src == ea ? eb : ea);
    if (i == 0)
      launch_step(L, k_line_transport<Real, kBC, true>, grid, tile, smem, K, src, ucur, uprev, drho, kap, dst, gh, m);
    else
      launch_step(L, k_line_transport<Real, kBC, false>, grid, tile, smem, K, src, ucur, uprev, drho, kap, dst, gh, m);
    src = dst;
    done += m;
  }
  return parts;
}

// Block of k_brick_transport: its region and how the threads share it.
struct BrickBlock {
  int ext[3], halo[3];
  int planes, groups;  // planes a thread, threads a column
  int threads;
  size_t smem;
};

// Fill in the block of tiles of own points with halo h; false if it does not fit.
static inline bool brick_block(const rpk_lattice* L, int open, const int (&own)[3], int h, BrickBlock& b) {
  const int n[3] = {L->grid.nx, L->grid.ny, L->grid.nz};
  for (int a = 0; a < 3; ++a) {
    const bool op = (a == 0 && (open & (1 | kWallX))) || (a == 1 && (open & kWallY));
    b.halo[a] = !op && (int64_t)own[a] + 2 * h > n[a] ? 0 : h;
    b.ext[a] = op ? std::min(own[a] + 2 * h, n[a] + 2) : b.halo[a] ? own[a] + 2 * h : n[a];
  }
  if ((int64_t)b.ext[0] * b.ext[1] > kBrickThreads) return false;
  const int area = b.ext[0] * b.ext[1], Z = b.ext[2], columns = kBrickThreads / area;
  if (Z > kBrickMaxP * columns) return false;
  b.planes = (Z + columns - 1) / columns;
  b.groups = (Z + b.planes - 1) / b.planes;
  b.threads = (area * b.groups + 31) / 32 * 32;
  b.smem = sizeof(float) * kBrickArrays * kBrickThreads * b.planes;
  return true;
}

static inline auto brick_kernel(bool first, int planes) {
  static constexpr decltype(&k_brick_transport<true, 1>) kernels[2][kBrickMaxP] = {
      {k_brick_transport<false, 1>, k_brick_transport<false, 2>, k_brick_transport<false, 3>,
       k_brick_transport<false, 4>, k_brick_transport<false, 5>, k_brick_transport<false, 6>},
      {k_brick_transport<true, 1>, k_brick_transport<true, 2>, k_brick_transport<true, 3>,
       k_brick_transport<true, 4>, k_brick_transport<true, 5>, k_brick_transport<true, 6>}};
  return kernels[first][planes - 1];
}

// The cheapest split of a small lattice's transport into launches and tiles, or
// none if a launch per pass costs less. Times in cycles, fitted to measurements: a
// launch costs 3000 plus the greater of latency (1500, 600 a sub-step and 2500 for
// each round of resident blocks) and work (for each warp and plane on the busiest SM
// 50 and 22 a sub-step; 60 more for the MacCormack passes); a launch per pass costs 4900 plus one for 60 points of a sublattice, four
// points a thread, or 5000 plus one for 36. Steps of both, us, passes / tiles: 16^3
// 10.4 / 7.2, 40^3 16.3 / 14.4, 48^3 20.1 / 22.0 (passes taken), 64^3 45.5 / 53.7
// (passes); between walls with five sub-steps 64 x 32 x 4 24.2 / 13.2, 150 x 90 x 8
// 43.9 / 37.7, 160 x 96 x 16 80.6 / 81.3 (passes).
static inline rpk_status make_brick_plan(rpk_lattice* L, int open) {
  BrickPlan& B = L->brick;
  if (B.nsub == L->nsub && B.open == open) return RPK_OK;
  B = BrickPlan();
  auto made = [&] {
    B.nsub = L->nsub;
    B.open = open;
    return RPK_OK;
  };
  if (L->n3 > (int64_t)kBrickMaxP * kBrickThreads * L->sms) return made();
  const int n[3] = {L->grid.nx, L->grid.ny, L->grid.nz};
  static constexpr int kCuts[] = {1, 2, 3, 4, 5, 6, 8, 10, 12, 16, 20, 24, 32, 48, 64, 96, 128};
  // the cuts of an axis that give tiles of different length, fewest first
  struct Cut {
    int count, own;
  } cuts[3][sizeof(kCuts) / sizeof(int)];
  int ncuts[3] = {0, 0, 0};
  for (int a = 0; a < 3; ++a)
    for (int c : kCuts) {
      const int own = (n[a] + c - 1) / c;
      if (c <= n[a] && (ncuts[a] == 0 || cuts[a][ncuts[a] - 1].own != own)) cuts[a][ncuts[a]++] = {c, own};
    }
  // best tile of a launch of m sub-steps
  auto best = [&](int m, bool first, BrickPlan::Part& part) {
    double cost = 1e30;
    for (int kz = 0; kz < ncuts[2]; ++kz)
      for (int ky = 0; ky < ncuts[1]; ++ky)
        for (int kx = 0; kx < ncuts[0]; ++kx) {
          const int cx = cuts[0][kx].count, cy = cuts[1][ky].count, cz = cuts[2][kz].count;
          if (cx * cy * cz > 2 * L->sms) break;
          const int own[3] = {cuts[0][kx].own, cuts[1][ky].own, cuts[2][kz].own};
          BrickBlock b;
          if (cost <= 7000.0 + 600.0 * m) return cost;  // the least of any tile
          if (!brick_block(L, open, own, m + (first ? 1 : 0), b)) continue;
          const int blocks = (2 * cx * cy * cz + L->sms - 1) / L->sms;  // of the busiest SM
          const int rounds = (blocks * b.threads + kBrickThreads - 1) / kBrickThreads;
          const double latency = 1500 + 600 * m + 2500 * rounds;
          const double work = (double)blocks * (b.threads / 32) * b.planes * (50 + (first ? 60 : 0) + 22 * m);
          const double c = 3000 + std::max(latency, work);
          if (c < cost) {
            cost = c;
            part = {m, {own[0], own[1], own[2]}};
          }
        }
    return cost;
  };
  double cost = (2 + L->nsub) * (open == 0 && L->grid.nx % 4 == 0 ? 4900 + L->n3 / 60.0 : 5000 + L->n3 / 36.0);
  for (int m = std::min(L->nsub, kBrickSub); m >= 1; --m) {
    const int parts = (L->nsub + m - 1) / m;
    if (m > 1 && (L->nsub + m - 2) / (m - 1) == parts) continue;  // as many launches of fewer sub-steps
    if (7000.0 * parts + 600.0 * L->nsub >= cost) continue;        // their least cost
    BrickPlan::Part first, full, rest;
    // parts of m or m - 1 sub-steps, the first with the deeper halo a short one
    const int shorter = parts * m - L->nsub, m0 = m - (shorter ? 1 : 0);
    double c = best(m0, true, first);
    const int nfull = L->nsub - m0 - (shorter ? shorter - 1 : 0) * (m - 1);
    if (parts > 1 && nfull > 0) c += nfull / m * best(m, false, full);
    if (shorter > 1) c += (shorter - 1) * best(m - 1, false, rest);
    if (c < cost) {
      cost = c;
      B.part[0] = first, B.part[1] = full, B.part[2] = rest;
      B.times[0] = 1, B.times[1] = nfull / m, B.times[2] = std::max(0, shorter - 1);
    }
  }
  if (!B.launches()) return made();
  for (int planes = 1; planes <= kBrickMaxP; ++planes)
    for (bool first : {true, false})
      RPK_CUDA(cudaFuncSetAttribute(brick_kernel(first, planes), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBrickSmem));
  return made();
}

// Transport of a small lattice in FP32 by its plan (conservative form).
static inline rpk_status brick_launch(rpk_lattice* L, const StepConst<float>& K, int open) {
  const float* src = static_cast<const float*>(L->e_star);
  RPK_CUDA(timing_begin(L));
  const int parts = L->brick.launches();
  for (int i = 0; i < parts; ++i) {
    const BrickPlan::Part& part = L->brick.at(i);
    BrickArgs B{};
    B.nsub = part.nsub;
    B.open = open;
    BrickBlock b;
    if (!brick_block(L, open, part.own, part.nsub + (i == 0 ? 1 : 0), b)) return fail(RPK_ERR_STATE, "transport tile does not fit");
    const int n[3] = {L->grid.nx, L->grid.ny, L->grid.nz};
    unsigned cuts[3];
    for (int a = 0; a < 3; ++a) {
      B.own[a] = part.own[a];
      B.ext[a] = b.ext[a];
      B.halo[a] = b.halo[a];
      cuts[a] = (n[a] + part.own[a] - 1) / part.own[a];
    }
    B.tx = cuts[0];
    B.ty = cuts[1];
    B.groups = b.groups;
    B.by_tx = FastDiv(cuts[0]);
    B.by_ty = FastDiv(cuts[1]);
    B.by_X = FastDiv(b.ext[0]);
    B.by_area = FastDiv(b.ext[0] * b.ext[1]);
    float* dst = static_cast<float*>(i + 1 == parts ? L->e : src == L->e_a ? L->e_b : L->e_a);
    launch_step(L, brick_kernel(i == 0, b.planes), dim3(cuts[0] * cuts[1] * cuts[2], 2), dim3(b.threads), b.smem, K, B, src,
                static_cast<const float*>(L->u[L->steps & 1]), static_cast<const float*>(L->u[(L->steps + 1) & 1]),
                static_cast<const float*>(L->drho), static_cast<const float*>(L->kap), dst,
                static_cast<const float*>(L->ghost));
    src = dst;
  }
  RPK_CUDA(timing_end(L, RPK_KC_TRANSPORT, parts));
  return check_launch("rotational transport (brick)");
}

template <typename Real, int kBC>
static rpk_status transport_launch(rpk_lattice* L, const StepConst<Real>& K) {
  const Real* ucur = static_cast<const Real*>(L->u[L->steps & 1]);
  const Real* uprev = static_cast<const Real*>(L->u[(L->steps + 1) & 1]);
  const Real* gh = static_cast<const Real*>(L->ghost);
  const Real* drho = static_cast<const Real*>(L->drho);
  const Real* kap = static_cast<const Real*>(L->kap);
  Real* es = static_cast<Real*>(L->e_star);
  Real* ea = static_cast<Real*>(L->e_a);
  Real* eb = static_cast<Real*>(L->e_b);
  Real* v = static_cast<Real*>(L->vbuf);
  Real* th = static_cast<Real*>(L->thbuf);
  Real* e = static_cast<Real*>(L->e);
  const dim3 tb(kTBX, kTBY);
  const dim3 tgrid((unsigned)((L->grid.nx + kTBX - 1) / kTBX),
                   (unsigned)((L->grid.ny + kTBY - 1) / kTBY), (unsigned)(2 * L->grid.nz));
  RPK_CUDA(timing_begin(L));
  if (L->rot_mode) {
    // paper mode: MacCormack on theta_R, FTCS sub-steps, the last with the
    // second relaxation half step (th holds the time-t theta_T)
    if constexpr (kBC == 0 && sizeof(Real) == 4) {
      if (L->grid.nx % 4 == 0) {
        // periodic FP32 grid, nx a multiple of 4: four x-adjacent points per thread
        const dim3 qgrid((unsigned)((L->grid.nx / 4 + kTBX - 1) / kTBX),
                         (unsigned)((L->grid.ny + kTBY - 1) / kTBY), (unsigned)(2 * L->grid.nz));
        launch_step(L, k_pm_pred4, qgrid, tb, 0, K, es, ucur, ea);
        launch_step(L, k_pm_corr4, qgrid, tb, 0, K, es, ea, ucur, eb);
        const Real* src = eb;
        for (int k = 0; k < L->nsub; ++k) {
          Real* dst = (k == L->nsub - 1) ? e : (src == eb ? ea : eb);
          launch_step(L, k_pm_ftcs4, qgrid, tb, 0, K, src, drho, kap, th, dst, k == L->nsub - 1);
          src = dst;
        }
        RPK_CUDA(timing_end(L, RPK_KC_TRANSPORT, 2 + L->nsub));
        return check_launch("rotational transport (paper mode)");
      }
    }
    launch_step(L, k_pm_pred<Real, kBC>, tgrid, tb, 0, K, es, ucur, ea, gh);
    launch_step(L, k_pm_corr<Real, kBC>, tgrid, tb, 0, K, es, ea, ucur, eb, gh);
    const Real* src = eb;
    for (int k = 0; k < L->nsub; ++k) {
      Real* dst = (k == L->nsub - 1) ? e : (src == eb ? ea : eb);
      launch_step(L, k_pm_ftcs<Real, kBC>, tgrid, tb, 0, K, src, drho, kap, th, dst, gh,
                                                         k == L->nsub - 1);
      src = dst;
    }
    RPK_CUDA(timing_end(L, RPK_KC_TRANSPORT, 2 + L->nsub));
    return check_launch("rotational transport (paper mode)");
  }
  if constexpr (kBC == 0 || kBC == 1) {
    if (L->grid.ny == 1 && L->grid.nz == 1) {
      const int n = line_launches<Real, kBC>(L, K, es, ucur, uprev, drho, kap, e, ea, eb, gh);
      RPK_CUDA(timing_end(L, RPK_KC_TRANSPORT, n));
      return check_launch("rotational transport (line)");
    }
  }
  // predictor and corrector, then the FTCS sub-steps: e in place from the
  // second on, theta_R between the transport's scratch planes
  bool quads = false;
  if constexpr (kBC == 0 && sizeof(Real) == 4) quads = L->grid.nx % 4 == 0;
  // periodic FP32 grid, nx a multiple of 4: four x-adjacent points per thread
  const dim3 qgrid((unsigned)((L->grid.nx / 4 + kTBX - 1) / kTBX),
                   (unsigned)((L->grid.ny + kTBY - 1) / kTBY), (unsigned)(2 * L->grid.nz));
  if (quads) {
    if constexpr (kBC == 0 && sizeof(Real) == 4) {
      launch_step(L, k_mac_pred4, qgrid, tb, 0, K, es, ucur, uprev, ea, v);
      launch_step(L, k_mac_corr4, qgrid, tb, 0, K, es, ea, v, drho, eb, th);
    }
  } else {
    launch_step(L, k_mac_pred<Real, kBC>, tgrid, tb, 0, K, es, ucur, uprev, ea, v, gh);
    launch_step(L, k_mac_corr<Real, kBC>, tgrid, tb, 0, K, es, ea, v, drho, eb, th, gh);
  }
  const Real* src = eb;
  for (int k = 0; k < L->nsub; ++k) {
    Real* th_next = k == L->nsub - 1 ? nullptr : (th == ea ? static_cast<Real*>(L->thbuf) : ea);
    if (quads) {
      if constexpr (kBC == 0 && sizeof(Real) == 4)
        launch_step(L, k_ftcs4, qgrid, tb, 0, K, src, th, kap, e, drho, th_next);
    } else {
      launch_step(L, k_ftcs<Real, kBC>, tgrid, tb, 0, K, src, th, kap, e, drho, th_next, gh);
    }
    src = e;
    th = th_next;
  }
  RPK_CUDA(timing_end(L, RPK_KC_TRANSPORT, 2 + L->nsub));
  return check_launch("rotational transport");
}

template <typename Store, typename Real>
rpk_status Ops<Store, Real>::step(rpk_lattice* L, int64_t n) {
  const StepConst<Real> K = make_const<Real>(L);
  const bool res = L->grid.bc_x == RPK_BC_RESERVOIR;
  const int wm = wall_mask(L);
  // FP32 storage only: 16-bit states depend on the rounding of every step, and FP64's
  // pipe has no room for a recomputed halo
  bool brick = false;
  if constexpr (std::is_same<Store, float>::value) {
    if (!L->rot_mode && (wm || L->grid.ny > 1 || L->grid.nz > 1)) {
      const rpk_status st = make_brick_plan(L, res ? 1 : wm);
      if (st != RPK_OK) return st;
      brick = L->brick.launches() > 0;
    }
  }
  for (int64_t t = 0; t < n; ++t) {
    rpk_status st;
    RPK_CUDA(timing_begin(L));
    const bool wall_pull = wm && !L->streamed;
    if (wall_pull) {
      st = wall_launch<Store, Real>(L, K);
      if (st != RPK_OK) return st;
    }
    if (L->streamed)
      st = res ? collide_launch<Store, Real, false, 1>(L, K) : collide_launch<Store, Real, false, 0>(L, K);
    else if (wm == kWallY)
      st = collide_launch<Store, Real, true, kWallY>(L, K);
    else if (wm == kWallX)
      st = collide_launch<Store, Real, true, kWallX>(L, K);
    else if (wm)
      st = collide_launch<Store, Real, true, kWallY | kWallX>(L, K);
    else
      st = res ? collide_launch<Store, Real, true, 1>(L, K) : collide_launch<Store, Real, true, 0>(L, K);
    if (st != RPK_OK) return st;
    RPK_CUDA(timing_end(L, RPK_KC_COLLIDE, wall_pull ? 2 : 1));
    if (brick) {
      if constexpr (std::is_same<Store, float>::value) st = brick_launch(L, K, res ? 1 : wm);
    } else if (wm == kWallY)
      st = transport_launch<Real, kWallY>(L, K);
    else if (wm == kWallX)
      st = transport_launch<Real, kWallX>(L, K);
    else if (wm)
      st = transport_launch<Real, kWallY | kWallX>(L, K);
    else
      st = res ? transport_launch<Real, 1>(L, K) : transport_launch<Real, 0>(L, K);
    if (st != RPK_OK) return st;
    L->cur ^= 1;
    L->streamed = false;
    L->steps += 1;
  }
  return RPK_OK;
}

template <typename Store, typename Real>
rpk_status Ops<Store, Real>::init(rpk_lattice* L, const double* rho, const double* u,
                                  const double* T, const double* R) {
  const StepConst<Real> K = make_const<Real>(L);
  const Real hdt = Real(0.5 * L->relax.dt / L->relax.tau1);
  L->cur = 0;
  unsigned long long* check = reinterpret_cast<unsigned long long*>(L->diag_out);
  RPK_CUDA(cudaMemsetAsync(check, 0, 2 * sizeof(unsigned long long), L->stream));
  const PointLaunch pt(L, L->n3);
  k_init<Store, Real><<<pt.grid, pt.block, 0, L->stream>>>(
      K, hdt, rho, u, T, R, static_cast<Store*>(L->pop[0]), static_cast<Real*>(L->e),
      static_cast<Real*>(L->u[0]), static_cast<Real*>(L->u[1]), check);
  return check_launch("k_init");
}

template <typename Store, typename Real>
rpk_status Ops<Store, Real>::ghosts(rpk_lattice* L) {
  const StepConst<Real> K = make_const<Real>(L);
  const Real hdt = Real(0.5 * L->relax.dt / L->relax.tau1);
  double* dst = L->diag_partial;  // 24 doubles of staging
  // blocks 0, 1: the reservoirs' states or the y walls; blocks 2, 3: the x
  // walls. A wall's state: rho = 1 at its velocity, theta_T = theta_R = theta_w.
  double st24[24] = {0};
  auto wall_state = [&](const double* wl, double* out6) {
    const double s6[6] = {1.0, wl[0], wl[1], wl[2], wl[3], wl[3]};
    for (int k = 0; k < 6; ++k) out6[k] = s6[k];
  };
  const double rest[4] = {0.0, 0.0, 0.0, kTheta0};  // fills blocks nothing reads
  if (L->walls) {
    wall_state(L->wall, st24);
    wall_state(L->wall + 4, st24 + 6);
  } else if (L->grid.bc_x == RPK_BC_RESERVOIR) {
    for (int k = 0; k < 12; ++k) st24[k] = L->res[k];
  } else {
    wall_state(rest, st24);
    wall_state(rest, st24 + 6);
  }
  wall_state(L->xwalls ? L->xwall : rest, st24 + 12);
  wall_state(L->xwalls ? L->xwall + 4 : rest, st24 + 18);
  RPK_CUDA(cudaMemcpyAsync(dst, st24, 24 * sizeof(double), cudaMemcpyHostToDevice, L->stream));
  k_ghost<Real><<<1, 32, 0, L->stream>>>(K, hdt, dst, static_cast<Real*>(L->ghost));
  rpk_status st = check_launch("k_ghost");
  if (st != RPK_OK) return st;
  k_ghost<Real><<<1, 32, 0, L->stream>>>(K, hdt, dst + 12, static_cast<Real*>(L->ghost) + 2 * kGhostStride);
  st = check_launch("k_ghost");
  if (st != RPK_OK) return st;
  RPK_CUDA(cudaStreamSynchronize(L->stream));
  return RPK_OK;
}

template <typename Store, typename Real>
rpk_status Ops<Store, Real>::moments(rpk_lattice* L, double* rho, double* u, double* T,
                                     double* R, double* E) {
  const StepConst<Real> K = make_const<Real>(L);
  const Store* pin = static_cast<const Store*>(L->pop[L->cur]);
  const Real* e = static_cast<const Real*>(L->e);
  const Real* gh = static_cast<const Real*>(L->ghost);
  const Real* wcol = static_cast<const Real*>(L->wrho);
  const PointLaunch pt(L, L->n3);
  const bool res = L->grid.bc_x == RPK_BC_RESERVOIR;
  const int wm = wall_mask(L);
  if (L->streamed) {
    k_moments<Store, Real, false, 0><<<pt.grid, pt.block, 0, L->stream>>>(K, pin, e, gh, rho, u, T, R, E, wcol);
  } else if (wm) {
    rpk_status st = wall_launch<Store, Real>(L, K);
    if (st != RPK_OK) return st;
    if (wm == kWallY)
      k_moments<Store, Real, true, kWallY><<<pt.grid, pt.block, 0, L->stream>>>(K, pin, e, gh, rho, u, T, R, E, wcol);
    else if (wm == kWallX)
      k_moments<Store, Real, true, kWallX><<<pt.grid, pt.block, 0, L->stream>>>(K, pin, e, gh, rho, u, T, R, E, wcol);
    else
      k_moments<Store, Real, true, kWallY | kWallX><<<pt.grid, pt.block, 0, L->stream>>>(K, pin, e, gh, rho, u, T, R,
                                                                                E, wcol);
  } else if (res) {
    k_moments<Store, Real, true, 1><<<pt.grid, pt.block, 0, L->stream>>>(K, pin, e, gh, rho, u, T, R, E, wcol);
  } else {
    k_moments<Store, Real, true, 0><<<pt.grid, pt.block, 0, L->stream>>>(K, pin, e, gh, rho, u, T, R, E, wcol);
  }
  return check_launch("k_moments");
}

template <typename Store, typename Real>
rpk_status Ops<Store, Real>::diag(rpk_lattice* L, double out[8]) {
  const StepConst<Real> K = make_const<Real>(L);
  const Store* pin = static_cast<const Store*>(L->pop[L->cur]);
  const Real* e = static_cast<const Real*>(L->e);
  const Real* gh = static_cast<const Real*>(L->ghost);
  // one wave of resident blocks (4 per SM in FP32 arithmetic), grid-stride
  const int64_t need = (L->npts + kDiagThreads - 1) / kDiagThreads;
  const int64_t wave = (int64_t)L->sms * (sizeof(Real) == 4 ? 4 : 1);
  const int nblk = (int)std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(kDiagBlocks, wave), need));
  const Real* wcol = static_cast<const Real*>(L->wrho);
  const bool res = L->grid.bc_x == RPK_BC_RESERVOIR;
  const int wm = wall_mask(L);
  bool pair = false;
  if constexpr (sizeof(Real) == 4) pair = !L->streamed && !wm && !res && L->grid.nx % 2 == 0;
  if (pair) {
    if constexpr (sizeof(Real) == 4) {
      // two points per thread (3 blocks per SM)
      const int64_t pneed = (L->npts / 2 + kDiagThreads - 1) / kDiagThreads;
      const int pblk = (int)std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(kDiagBlocks, (int64_t)L->sms * 3), pneed));
      if (L->rot_mode)
        k_diag_pair<Store, true><<<pblk, kDiagThreads, 0, L->stream>>>(K, pin, e, L->diag_partial);
      else
        k_diag_pair<Store, false><<<pblk, kDiagThreads, 0, L->stream>>>(K, pin, e, L->diag_partial);
      rpk_status st0 = check_launch("k_diag_pair");
      if (st0 != RPK_OK) return st0;
      k_diag_final<<<1, 1024, 0, L->stream>>>(L->diag_partial, pblk, L->diag_out);
      st0 = check_launch("k_diag_final");
      if (st0 != RPK_OK) return st0;
      RPK_CUDA(cudaMemcpyAsync(out, L->diag_out, kDiagVals * sizeof(double), cudaMemcpyDeviceToHost,
                               L->stream));
      RPK_CUDA(cudaStreamSynchronize(L->stream));
      return RPK_OK;
    }
  }
  if (L->streamed) {
    k_diag<Store, Real, false, 0><<<nblk, kDiagThreads, 0, L->stream>>>(K, pin, e, gh, L->diag_partial, wcol);
  } else if (wm) {
    rpk_status sw = wall_launch<Store, Real>(L, K);
    if (sw != RPK_OK) return sw;
    if (wm == kWallY)
      k_diag<Store, Real, true, kWallY><<<nblk, kDiagThreads, 0, L->stream>>>(K, pin, e, gh, L->diag_partial,
                                                                               wcol);
    else if (wm == kWallX)
      k_diag<Store, Real, true, kWallX><<<nblk, kDiagThreads, 0, L->stream>>>(K, pin, e, gh, L->diag_partial,
                                                                               wcol);
    else
      k_diag<Store, Real, true, kWallY | kWallX><<<nblk, kDiagThreads, 0, L->stream>>>(
          K, pin, e, gh, L->diag_partial, wcol);
  } else if (res) {
    k_diag<Store, Real, true, 1><<<nblk, kDiagThreads, 0, L->stream>>>(K, pin, e, gh, L->diag_partial, wcol);
  } else {
    k_diag<Store, Real, true, 0><<<nblk, kDiagThreads, 0, L->stream>>>(K, pin, e, gh, L->diag_partial, wcol);
  }
  rpk_status st = check_launch("k_diag");
  if (st != RPK_OK) return st;
  k_diag_final<<<1, 1024, 0, L->stream>>>(L->diag_partial, nblk, L->diag_out);
  st = check_launch("k_diag_final");
  if (st != RPK_OK) return st;
  RPK_CUDA(cudaMemcpyAsync(out, L->diag_out, kDiagVals * sizeof(double), cudaMemcpyDeviceToHost,
                           L->stream));
  RPK_CUDA(cudaStreamSynchronize(L->stream));
  return RPK_OK;
}

}  // namespace rpk
