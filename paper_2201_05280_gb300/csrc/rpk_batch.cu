// Batched quasi-1-D tubes: many independent nx x 1 x 1 lattices (shock tubes
// with x reservoirs) advanced by one persistent kernel launch.
//
// Each CTA takes whole tubes from a work queue (an atomic counter over a
// longest-work-first order) and runs every step of a tube itself: the pull +
// collide pass over the tube's 2 nx points reads and writes the tube's
// populations in device memory, while the auxiliary rotational energy, the
// two velocity slots, rho - 1, kappa_R, the predictor and theta_R of the tube
// live in shared memory for the whole time loop, so the transport (MacCormack
// and the FTCS sub-steps) costs no device-memory traffic. Tubes need no
// synchronisation with each other, so the launch has no grid-wide barrier. The
// method is that of the lattice kernels on an nx x 1 x 1 grid, where every y and z
// neighbour is the point itself and contributes exact zeros; the collision is the
// factored form of FP64 lattices in FP32 too, so FP32 tubes and FP32 lattices agree to
// rounding, not bit for bit.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "rpk_internal.h"
#include "rpk_ops.cuh"

namespace rpk {

// Shared arrays per tube point: e (e*, corrected e), u slot 0, u slot 1, rho - 1,
// kappa, predictor, and for FTCS theta_R of the corrector; the backward-Euler solve
// needs four values per block of kBE points instead. Shared memory that is not
// asked for stays L1 cache, which bounds the loads in flight: with seven arrays
// tubes of 4000 cells (224 KB) ran at 13.3 G point steps a second, with six at 15.8
// (backward Euler); FTCS is bound by its sub-steps.
// Tube lengths and CTAs per SM are accepted as for seven arrays either way.
constexpr int kBatchArrays = 6;
constexpr int kBatchRuleArrays = 7;
constexpr size_t kBatchSmemLimit = 227 * 1024;

template <typename Real>
struct TubeDev {
  StepConst<Real> K;  // nx, ny = nz = 1, n3 = nx and the relaxation constants
  Real hdt;           // dt / (2 tau1), for the initial state
  int nx, nsteps, nsub, cur;
  int streamed, pad0, pad1, pad2;
  int64_t pop_off;   // element offset of the tube in each population buffer
  int64_t pt_off;    // point offset in the concatenated point arrays
  int64_t snap_off;  // float offset of the tube's snapshots
  Real ghost[2 * kGhostStride];
};

// Gathered point index of point p (0 <= p < 2 nx) of a tube.
__device__ __forceinline__ PointIdx tube_point(int nx, int p) {
  PointIdx P;
  P.s = p >= nx;
  P.x = p - P.s * nx;
  P.y = 0;
  P.z = 0;
  P.cell = P.x;
  return P;
}

// The pull of `gather` on an nx x 1 x 1 lattice between reservoirs: only x
// shifts, 32-bit offsets, and no end checks where every source is inside.
template <typename Store, typename Real>
__device__ __forceinline__ void gather_line(const Store* __restrict__ pin, const Real* __restrict__ ghost, int nx,
                                            int s, int x, Real (&h)[kQ]) {
  const Store* same = pin + s * kQ * nx + x;
  const Store* other = pin + (1 - s) * kQ * nx + x;
  const int hp = s ? 0 : -1, hm = s ? 1 : 0;  // source offsets of the half velocities, c_x > 0 and < 0
  if (x >= 2 && x < nx - 2) {
    h[0] = to_real<Store, Real>(same[0]);
    static_for<kQ - 1>([&](auto qc) {
      constexpr int q = decltype(qc)::value + 1;
      constexpr Vel2 v = vel2(q);
      if constexpr ((v.x & 1) != 0)
        h[q] = to_real<Store, Real>(other[q * nx + (v.x > 0 ? hp : hm)]);
      else
        h[q] = to_real<Store, Real>(same[q * nx - v.x / 2]);
    });
  } else {
    h[0] = to_real<Store, Real>(same[0]);
    static_for<kQ - 1>([&](auto qc) {
      constexpr int q = decltype(qc)::value + 1;
      constexpr Vel2 v = vel2(q);
      constexpr bool half = (v.x & 1) != 0;
      const int d = half ? (v.x > 0 ? hp : hm) : -v.x / 2;
      if (x + d < 0 || x + d >= nx)
        h[q] = ghost[(v.x > 0 ? 0 : kGhostStride) + q];
      else
        h[q] = to_real<Store, Real>((half ? other : same)[q * nx + d]);
    });
  }
}

// One backward-Euler step of the rotational diffusion on a tube's two lines,
//     (delta rho / 2) phi - dt [K+ (phi_+ - phi) - K- (phi - phi_-)] = e - delta theta0 D / 2
// for phi = theta_R - theta0, by substructuring: every thread eliminates inside
// blocks of kBE points, leaving each point as x = r + l x_prev + u x_sep in terms of
// the last points (separators) of the previous and its own block; one warp per
// line reduces the separators' equations the same way to one per lane, solves
// those 32 by parallel cyclic reduction in shuffles and substitutes back; then
// all points follow independently. Three block barriers (cyclic reduction over
// the points needed 2 log2(nx) + 3) and one division per point. kBE is odd, so
// threads striding by it hit distinct banks.
// Each row carries its excess g = 1 - l - u along: l, u, g and r are then sums and
// products of non-negative numbers, with no cancellation however large K is
// (FP32, K = 400: error 9e-9 rms of phi where the reduction of the assembled
// matrix has 1.9e-7).
// In: e (sE), D (sD), kappa (sK). l -> sL, r -> sR, u -> sE (e is read by its own
// thread only), g of each block's first and last point -> sG. Out: e in sE.
constexpr int kBE = 9;

// A row of the elimination: x = r + l x_prev + u x_next, l + u + g = 1.
template <typename Real>
struct BeRow {
  Real l, u, g, r;
};

// Row x = (rr + kf x_before + kq x_next) / (s + kf + kq) after x_before = row p.
template <typename Real>
__device__ __forceinline__ BeRow<Real> be_eliminate(const BeRow<Real>& p, Real kf, Real kq, Real s, Real rr) {
  const Real inv = Real(1) / fmad(kf, p.l + p.g, s + kq);
  return {kf * p.l * inv, kq * inv, fmad(kf, p.g, s) * inv, fmad(kf, p.r, rr) * inv};
}

// Row a with its x_next replaced by row n (in the same x_prev).
template <typename Real>
__device__ __forceinline__ void be_fold(BeRow<Real>& a, const BeRow<Real>& n) {
  a.l = fmad(a.u, n.l, a.l);
  a.g = fmad(a.u, n.g, a.g);
  a.r = fmad(a.u, n.r, a.r);
  a.u = a.u * n.u;
}

template <typename Real>
__device__ __forceinline__ void be_blocks(const StepConst<Real>& K, int nx, int nthreads, Real* sE, const Real* sD,
                                          const Real* sK, Real* sL, Real* sR, Real* sG, Real kGl, Real kGh, Real thGl,
                                          Real thGh) {
  const int nb = (nx + kBE - 1) / kBE;
  const Real half = Real(0.5), t0d = K.delta * K.theta0;
  for (int b = threadIdx.x; b < 2 * nb; b += nthreads) {
    const int line = b >= nb, x0 = (b - line * nb) * kBE, n = min(kBE, nx - x0), o = line * nx + x0;
    BeRow<Real> w[kBE];
    Real g_last = Real(0);
    Real kp = sK[o];
    Real kf = K.dt * (half * (kp + (x0 == 0 ? kGl : sK[o - 1])));  // face below
#pragma unroll
    for (int i = 0; i < kBE; ++i) {
      if (i < n) {
        const bool top = x0 + i == nx - 1;
        const Real kn = top ? kGh : sK[o + i + 1];
        const Real kq = K.dt * (half * (kp + kn));  // face above
        const Real dr = sD[o + i];
        Real s = half * K.delta * (Real(1) + dr), r = sE[o + i] - half * t0d * dr;
        Real l = kf, u = kq;
        if (x0 + i == 0) {  // the reservoirs' values are known
          r = fmad(kf, thGl, r);
          s += kf;
          l = Real(0);
        }
        if (top) {
          r = fmad(kq, thGh, r);
          s += kq;
          u = Real(0);
        }
        // before a block's first point lies x_prev itself
        const BeRow<Real> before = i == 0 ? BeRow<Real>{Real(1), Real(0), Real(0), Real(0)} : w[i > 0 ? i - 1 : 0];
        w[i] = be_eliminate(before, l, u, s, r);
        g_last = w[i].g;
        kp = kn;
        kf = kq;
      }
    }
#pragma unroll
    for (int i = kBE - 3; i >= 0; --i)
      if (i < n - 2) be_fold(w[i], w[i + 1]);
#pragma unroll
    for (int i = 0; i < kBE; ++i)
      if (i < n) {
        sL[o + i] = w[i].l;
        sE[o + i] = w[i].u;
        sR[o + i] = w[i].r;
      }
    sG[2 * b] = w[0].g;
    sG[2 * b + 1] = g_last;
  }
}

// Separators of a line by one warp; their solution replaces sR at the separators.
template <typename Real>
__device__ __forceinline__ void be_separators(int nx, int line, Real* sL, Real* sU, Real* sR, Real* sG) {
  const unsigned all = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int nb = (nx + kBE - 1) / kBE, per = (nb + 31) / 32;
  const int j0 = lane * per, cnt = max(0, min(per, nb - j0));
  auto sep = [&](int j) { return line * nx + min((j + 1) * kBE, nx) - 1; };
  Real* gl = sG + 2 * line * nb;  // g of block j's first (2 j) and last (2 j + 1) point
  auto get = [&](int j) {
    const int p = sep(j);
    return BeRow<Real>{sL[p], sU[p], gl[2 * j + 1], sR[p]};
  };
  auto put = [&](int j, const BeRow<Real>& w) {
    const int p = sep(j);
    sL[p] = w.l, sU[p] = w.u, gl[2 * j + 1] = w.g, sR[p] = w.r;
  };
  const BeRow<Real> none{Real(0), Real(1), Real(0), Real(0)};  // x_next is the separator itself
  // forward sweep over the lane's separators, rows kept at the separators' slots
  BeRow<Real> w{Real(0), Real(0), Real(1), Real(0)};
  for (int k = 0; k < cnt; ++k) {
    const int j = j0 + k;
    BeRow<Real> a = get(j);
    // the next block's first point by the separators (its own last point when
    // the block has one point; nothing beyond the last block, where u = 0)
    const int q = line * nx + (j + 1) * kBE;
    const BeRow<Real> n = j + 1 < nb && (j + 1) * kBE < nx - 1 ? BeRow<Real>{sL[q], sU[q], gl[2 * j + 2], sR[q]} : none;
    // a = r + l x_prev + u (n.r + n.l x + n.u x_next): 1 - u n.l = l + g + u (n.u + n.g)
    const Real inv = Real(1) / (a.l + fmad(a.u, n.u + n.g, a.g));
    a.g = fmad(a.u, n.g, a.g) * inv;
    a.r = fmad(a.u, n.r, a.r) * inv;
    a.u = a.u * n.u * inv;
    a.l = a.l * inv;
    w = k == 0 ? a : be_eliminate(w, a.l, a.u, a.g, a.r);
    put(j, w);
  }
  // the lane's first separator by the previous lane's last one and its own
  // last one; w stays the last row
  BeRow<Real> f = none;
  if (cnt > 1) {
    f = get(j0 + cnt - 2);
    for (int k = cnt - 3; k >= 0; --k) {
      BeRow<Real> a = get(j0 + k);
      be_fold(a, f);
      put(j0 + k, a);
      f = a;
    }
  }
  // last rows by the lanes' last separators
  const BeRow<Real> n{__shfl_down_sync(all, f.l, 1), __shfl_down_sync(all, f.u, 1), __shfl_down_sync(all, f.g, 1),
                      __shfl_down_sync(all, f.r, 1)};
  BeRow<Real> y = w;
  if (lane < 31 && cnt > 0 && j0 + cnt < nb) {
    const Real inv = Real(1) / (w.l + fmad(w.u, n.u + n.g, w.g));
    y = {w.l * inv, w.u * n.u * inv, fmad(w.u, n.g, w.g) * inv, fmad(w.u, n.r, w.r) * inv};
  }
#pragma unroll
  for (int h = 1; h < 32; h *= 2) {
    const Real lm = __shfl_up_sync(all, y.l, h), gm = __shfl_up_sync(all, y.g, h), rm = __shfl_up_sync(all, y.r, h);
    const Real up = __shfl_down_sync(all, y.u, h), gp = __shfl_down_sync(all, y.g, h), rp = __shfl_down_sync(all, y.r, h);
    const Real l = lane >= h ? y.l : Real(0), u = lane + h < 32 ? y.u : Real(0);
    const Real inv = Real(1) / fmad(l, lm + gm, fmad(u, up + gp, y.g));
    y = {l * lm * inv, u * up * inv, fmad(l, gm, fmad(u, gp, y.g)) * inv, fmad(l, rm, fmad(u, rp, y.r)) * inv};
  }
  const Real v = y.r;
  Real vp = __shfl_up_sync(all, v, 1);
  if (lane == 0) vp = Real(0);
  for (int k = 0; k < cnt; ++k) {
    const int p = sep(j0 + k);
    sR[p] = k == cnt - 1 ? v : fmad(sL[p], vp, fmad(sU[p], v, sR[p]));
  }
}

// e of every point from its block's and the previous block's separators.
template <typename Real>
__device__ __forceinline__ void be_points(const StepConst<Real>& K, int nx, int nthreads, Real* sE, const Real* sD,
                                          const Real* sL, const Real* sR) {
  for (int p = threadIdx.x; p < 2 * nx; p += nthreads) {
    const int s = p >= nx, x = p - s * nx, j = x / kBE;
    const int q = s * nx + min((j + 1) * kBE, nx) - 1;
    Real phi = sR[q];
    if (p != q) {
      phi = fmad(sE[p], phi, sR[p]);  // u
      if (j > 0) phi = fmad(sL[p], sR[s * nx + j * kBE - 1], phi);
    }
    const Real dr = sD[p];
    sE[p] = Real(0.5) * K.delta * ((Real(1) + dr) * phi + K.theta0 * dr);
  }
}

__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// FTCS sub-steps of a tube's two sublattice lines, several per block barrier.
// A warp takes a piece of a line, kP consecutive points per lane, in
// registers: neighbours inside a lane are registers, those of the next lane
// one shuffle each side, so m <= kP sub-steps need no barrier; lanes 0 and 31
// are halo (recomputed by the neighbouring pieces) and the 30 lanes between
// are written. kP is odd: 32 lanes reading with stride kP hit 32 banks.
// Bound: the FP32 pipes (theta, the face difference, two products and the update
// of every point and sub-step) and the chain of one sub-step. Arithmetic in the
// order of the lattice's FTCS kernels, so results are those of one barrier per
// sub-step bit for bit.
// With a block barrier and 10 shared loads per point and sub-step it took 0.8
// us a sub-step for tubes of 1500 cells; now 0.11 (0.16 with every piece loaded
// anew for each 5 to 13 sub-steps). 304 tubes of 500 to 1500 cells: 405 -> 70 ms.
template <typename Real>
struct FtcsLine {
  const Real* a;     // theta_R - theta0 = a e + c
  const Real* c;
  const Real* th0;   // theta_R - theta0 of the corrector, for the first sub-step
  const Real* face;  // K of the face below each point
  const Real* last;  // and of the face above the last point, per line
  int nx;
  Real h;             // dt / nsub
  Real th_lo, th_hi;  // reservoir values
};

// A piece in registers.
template <int kP, typename Real>
struct FtcsPiece {
  Real e[kP], a[kP], c[kP], f[kP + 1], th[kP];
  int at, nv;  // the lane's first point in a field; how many of its points lie on the line

  // Piece w of the tube's 2 x pieces, from the field ein.
  __device__ __forceinline__ void load(const FtcsLine<Real>& L, const Real* ein, int w, int pieces, bool first) {
    const int lane = threadIdx.x & 31, s = w >= pieces;
    const int x0 = (w - s * pieces) * 30 * kP + (lane - 1) * kP;  // -kP below the line's low end
    at = s * L.nx + x0;
    nv = x0 < 0 ? 0 : min(kP, max(0, L.nx - x0));
    const Real out = x0 < 0 ? L.th_lo : L.th_hi;
#pragma unroll
    for (int i = 0; i < kP; ++i) {
      const bool in = i < nv;
      // beyond an end: theta stays the reservoir's (a = 0)
      e[i] = in ? ein[at + i] : Real(0);
      a[i] = in ? L.a[at + i] : Real(0);
      c[i] = in ? L.c[at + i] : out;
      f[i] = in ? L.face[at + i] : Real(0);
      if (x0 + i == L.nx) f[i] = L.last[s];
      th[i] = fmad(a[i], e[i], c[i]);
    }
    f[kP] = __shfl_down_sync(0xffffffffu, f[0], 1);
    if (first) {
#pragma unroll
      for (int i = 0; i < kP; ++i)
        if (i < nv) th[i] = L.th0[at + i];
    }
  }

  // m <= kP sub-steps.
  __device__ __forceinline__ void advance(Real h, int m) {
#pragma unroll 1
    for (int k = 0; k < m; ++k) {
      const Real lo = __shfl_up_sync(0xffffffffu, th[kP - 1], 1);
      const Real hi = __shfl_down_sync(0xffffffffu, th[0], 1);
      Real d = th[0] - lo;
#pragma unroll
      for (int i = 0; i < kP; ++i) {
        const Real dn = (i + 1 < kP ? th[i + 1] : hi) - th[i];
        e[i] = fmad(h, fmad(f[i + 1], dn, -(f[i] * d)), e[i]);
        d = dn;
      }
#pragma unroll
      for (int i = 0; i < kP; ++i) th[i] = fmad(a[i], e[i], c[i]);
    }
  }

  __device__ __forceinline__ void store(Real* out) const {
#pragma unroll
    for (int i = 0; i < kP; ++i)
      if (i < nv) out[at + i] = e[i];
  }
  // e of the whole lane from a neighbour's store
  __device__ __forceinline__ void fetch(const Real* in) {
#pragma unroll
    for (int i = 0; i < kP; ++i)
      if (i < nv) {
        e[i] = in[at + i];
        th[i] = fmad(a[i], e[i], c[i]);
      }
  }
};

// More pieces than warps: every kP sub-steps all pieces go through registers.
template <int kP, typename Real>
__device__ __forceinline__ void ftcs_pass(const FtcsLine<Real>& L, const Real* ein, Real* eout, int m,
                                          int nwarps, bool first) {
  const int lane = threadIdx.x & 31, pieces = (L.nx + 30 * kP - 1) / (30 * kP);
  for (int w = threadIdx.x >> 5; w < 2 * pieces; w += nwarps) {
    FtcsPiece<kP, Real> P;
    P.load(L, ein, w, pieces, first);
    P.advance(L.h, m);
    if (lane > 0 && lane < 31) P.store(eout);
  }
}

// At most one piece per warp: it stays in registers for all sub-steps of the
// time step, and every kP of them the neighbours exchange their end lanes' points
// through two buffers used in turn. Warps without a piece only keep the barriers
// (one common path for both made the compiler spill the pieces around them).
template <int kP, typename Real>
__device__ __forceinline__ void ftcs_resident(const FtcsLine<Real>& L, Real* sE, Real* buf0, Real* buf1, int nsub) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int pieces = (L.nx + 30 * kP - 1) / (30 * kP);
  if (w >= 2 * pieces) {  // keeps the barriers' count
    for (int k = 0; k < nsub; k += kP) __syncthreads();
    __syncthreads();
    return;
  }
  FtcsPiece<kP, Real> P;
  P.load(L, sE, w, pieces, true);
  __syncthreads();  // every halo is read before sE is written
  Real* buf = buf0;
  Real* next = buf1;
  P.advance(L.h, min(nsub, kP));
#pragma unroll 1
  for (int k = kP; k < nsub; k += kP) {
    if (lane == 1 || lane == 30) P.store(buf);
    __syncthreads();
    if (lane == 0 || lane == 31) P.fetch(buf);
    P.advance(L.h, min(nsub - k, kP));
    Real* t = buf;
    buf = next;
    next = t;
  }
  if (lane > 0 && lane < 31) P.store(sE);
  __syncthreads();
}

// Points per lane: the fewest with which every warp has at most one piece; else
// (negative: passes) the fewest point slots per warp over the rounds that the
// pieces take, among equals the most (fewest barriers).
template <typename Real>
__device__ __forceinline__ int ftcs_width(int nx, int nwarps) {
  int best = 5, cost = 1 << 30;
  for (int w = 5; w <= (sizeof(Real) == 8 ? 5 : 13); w += (w < 9 ? 2 : 4)) {
    const int pieces = 2 * ((nx + 30 * w - 1) / (30 * w));
    if (pieces <= nwarps) return w;
    const int c = (pieces + nwarps - 1) / nwarps * w;
    if (c <= cost) {
      cost = c;
      best = w;
    }
  }
  return -best;
}

// kCtas: CTAs per SM that must fit its registers (see BatchOps); 0 leaves it open.
template <typename Store, typename Real, int kThreads, bool kImplicit, int kCtas>
__global__ void __launch_bounds__(kThreads, kCtas)
    k_batch(TubeDev<Real>* __restrict__ tubes, const int* __restrict__ order, int ntubes,
            int* __restrict__ counter, Store* __restrict__ pop0, Store* __restrict__ pop1,
            Real* __restrict__ e_state, Real* __restrict__ ux_state, float* __restrict__ snaps,
            int save_every, int max_np, int prefetch, unsigned* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Real* sE = reinterpret_cast<Real*>(smem_raw);  // auxiliary E_R (state), e* after the exchange, then corrector
  Real* sU0 = sE + max_np;                       // u_x ring slot 0
  Real* sU1 = sU0 + max_np;                      // u_x ring slot 1
  Real* sD = sU1 + max_np;                       // rho - 1
  Real* sK = sD + max_np;                        // kappa_R
  Real* sP = sK + max_np;                        // predictor
  [[maybe_unused]] Real* sG = sP + max_np;       // backward Euler: row excesses at block ends
  [[maybe_unused]] Real* sT = sG;                // FTCS: theta_R - theta0 of the corrector
  __shared__ int s_slot;
  __shared__ Real s_last[2];  // K of each line's last face
  const int tid = threadIdx.x;
  for (;;) {
    __syncthreads();
    if (tid == 0) s_slot = atomicAdd(counter, 1);
    __syncthreads();
    const int slot = s_slot;
    if (slot >= ntubes) break;
    TubeDev<Real>* T = tubes + order[slot];
    const StepConst<Real> K = T->K;
    const int nx = T->nx, np = 2 * nx, nsteps = T->nsteps, nsub = T->nsub;
    const Real* ghost = T->ghost;
    const Real* gl = ghost;
    const Real* gh = ghost + kGhostStride;
    Real* gE = e_state + T->pt_off;
    Real* gU = ux_state + T->pt_off;
    for (int p = tid; p < np; p += kThreads) {
      sE[p] = gE[p];
      sU1[p] = gU[p];  // u(t-1) for the first step
    }
    int cur = T->cur;
    bool streamed = T->streamed != 0;
    Store* bufs[2] = {pop0 + T->pop_off, pop1 + T->pop_off};
    const Real t0d = K.delta * K.theta0;
    // theta_R of the two reservoirs (constant)
    const Real thGl = (Real(2) * gl[kGhE] - t0d * gl[kGhDrho]) / (K.delta * (Real(1) + gl[kGhDrho]));
    const Real thGh = (Real(2) * gh[kGhE] - t0d * gh[kGhDrho]) / (K.delta * (Real(1) + gh[kGhDrho]));
    __syncthreads();
    for (int t = 0; t < nsteps; ++t) {
      Real* uc = (t & 1) ? sU1 : sU0;
      const Real* up = (t & 1) ? sU0 : sU1;
      const Store* pin = bufs[cur];
      Store* pout = bufs[cur ^ 1];
      const bool snap = (t % save_every) == 0;
      float* sn = snaps + T->snap_off + (int64_t)(t / save_every) * 4 * np;
      // 1. pull + collide + exchange of every point of the tube
      for (int p = tid; p < np; p += kThreads) {
        const int s = p >= nx, x = p - s * nx;
        // the populations of this warp's next points come from device memory while
        // these are worked on: lane l asks for planes l and l + 32 (L2 only, one
        // request per plane and warp). 3000 cells: 13.9 -> 15.6 G point steps a
        // second; where the running tubes fit L2 it costs (1000 cells: 16.1 -> 15.5)
        const int pn = p - (tid & 31) + kThreads;
        if (prefetch && pn < np) {
          const int sn = pn >= nx, xn = pn - sn * nx;
          prefetch_l2(pin + (sn * kQ + (tid & 31)) * nx + xn);
          if ((tid & 31) < kQ - 32) prefetch_l2(pin + (sn * kQ + 32 + (tid & 31)) * nx + xn);
        }
        Real h[kQ];
        if (streamed) {
#pragma unroll
          for (int q = 0; q < kQ; ++q) h[q] = to_real<Store, Real>(pin[(s * kQ + q) * nx + x]);
        } else {
          gather_line<Store, Real>(pin, ghost, nx, s, x, h);
        }
        Mom<Real> m;
        Store* out = pout + s * kQ * nx + x;
        const Real es = collide_shells<Real, false>(
            K, h, sE[p], [&](int q, Real v) { out[q * nx] = from_real<Store, Real>(v); }, m);
        sE[p] = es;
        sD[p] = m.drho;
        uc[p] = m.j[0] * m.inv_rho;
        sK[p] = K.kapc * m.rho * (K.theta0 + m.dth);
        flag_moments(m, K.theta0, status);
        if (snap) {
          sn[p] = (float)(Real(1) + m.drho);
          sn[np + p] = (float)(m.j[0] * m.inv_rho);
          sn[2 * np + p] = (float)(K.theta0 + m.dT);
          sn[3 * np + p] = (float)(Real(0.5) * K.delta * m.rho * (K.theta0 + m.dR));
        }
      }
      __syncthreads();
      // 2. MacCormack predictor (forward difference along x, same sublattice)
      for (int p = tid; p < np; p += kThreads) {
        const int s = p >= nx, x = p - s * nx;
        const Real vp = Real(1.5) * uc[p] - Real(0.5) * up[p];
        Real eq, vq;
        if (x + 1 >= nx) {
          eq = gh[kGhE];
          vq = gh[kGhU];
        } else {
          eq = sE[p + 1];
          vq = Real(1.5) * uc[p + 1] - Real(0.5) * up[p + 1];
        }
        const Real e0 = sE[p];
        Real div = Real(0);
        div += K.E0 * (vq - vp) + (eq * vq - e0 * vp);
        sP[p] = e0 - K.dt * div;
      }
      __syncthreads();
      // 3. corrector (backward difference), then theta_R of the result for FTCS
      for (int p = tid; p < np; p += kThreads) {
        const int s = p >= nx, x = p - s * nx;
        const Real vp = Real(1.5) * uc[p] - Real(0.5) * up[p];
        Real eq, vq;
        if (x == 0) {
          eq = gl[kGhE];
          vq = gl[kGhU];
        } else {
          eq = sP[p - 1];
          vq = Real(1.5) * uc[p - 1] - Real(0.5) * up[p - 1];
        }
        const Real epp = sP[p];
        Real div = Real(0);
        div += K.E0 * (vp - vq) + (epp * vp - eq * vq);
        const Real val = Real(0.5) * (sE[p] + epp - K.dt * div);
        sE[p] = val;
        if constexpr (!kImplicit) {
          const Real dr = sD[p];
          sT[p] = (Real(2) * val - t0d * dr) / (K.delta * (Real(1) + dr));
        }
      }
      __syncthreads();
      if constexpr (kImplicit) {
        // 4'. backward-Euler variant: l -> sP, u -> sE, r -> the u(t-1) slot (dead
        //     until the next step's u), g at the blocks' ends -> sG
        Real* r = (t & 1) ? sU0 : sU1;
        be_blocks(K, nx, kThreads, sE, sD, sK, sP, r, sG, gl[kGhKap], gh[kGhKap], thGl, thGh);
        __syncthreads();
        if (tid < 64) be_separators(nx, tid >> 5, sP, sE, r, sG);
        __syncthreads();
        be_points(K, nx, kThreads, sE, sD, sP, r);
        __syncthreads();
      } else {
        // 4. FTCS sub-steps, e += h sum_faces K_face (theta_nb - theta) with
        //    theta_R = a e + c, a = 2/(delta(1 + D)), c = -delta theta0 D/(delta(1 + D))
        //    (affine in e at fixed rho; the first sub-step takes the corrector's
        //    theta_R): a -> sP, c -> sD, K of every point's low face -> the u(t-1) slot (dead until the next step's u), e between sE and sK.
        Real* face = (t & 1) ? sU0 : sU1;
        for (int p = tid; p < np; p += kThreads) {
          const int s = p >= nx, x = p - s * nx;
          const Real dr = sD[p], kp = sK[p];
          const Real inv = Real(1) / (K.delta * (Real(1) + dr));
          sP[p] = Real(2) * inv;
          sD[p] = -t0d * dr * inv;
          face[p] = Real(0.5) * (kp + (x == 0 ? gl[kGhKap] : sK[p - 1]));
          if (x == nx - 1) s_last[s] = Real(0.5) * (kp + gh[kGhKap]);
        }
        __syncthreads();
        const FtcsLine<Real> FL{sP, sD, sT, face, s_last, nx, K.hsub, thGl, thGh};
        const int width = ftcs_width<Real>(nx, kThreads / 32);
        auto by_width = [&](auto&& run) {
          const int v = width < 0 ? -width : width;
          if constexpr (sizeof(Real) == 8) {
            run(std::integral_constant<int, 5>{});
          } else {
            if (v == 5) run(std::integral_constant<int, 5>{});
            else if (v == 7) run(std::integral_constant<int, 7>{});
            else if (v == 9) run(std::integral_constant<int, 9>{});
            else run(std::integral_constant<int, 13>{});
          }
        };
        if (width > 0) {
          by_width([&](auto wc) { ftcs_resident<decltype(wc)::value>(FL, sE, sK, sT, nsub); });
        } else {
          Real* ein = sE;
          Real* eout = sK;
          for (int k = 0; k < nsub;) {
            const int m = min(nsub - k, -width);
            by_width([&](auto wc) { ftcs_pass<decltype(wc)::value>(FL, ein, eout, m, kThreads / 32, k == 0); });
            k += m;
            __syncthreads();
            Real* tmp = ein;
            ein = eout;
            eout = tmp;
          }
          if (ein != sE) {
            for (int p = tid; p < np; p += kThreads) sE[p] = ein[p];
            __syncthreads();
          }
        }
      }
      cur ^= 1;
      streamed = false;
    }
    // write the tube's state back
    const Real* ulast = (nsteps == 0) ? sU1 : (((nsteps - 1) & 1) ? sU1 : sU0);
    for (int p = tid; p < np; p += kThreads) {
      gE[p] = sE[p];
      gU[p] = ulast[p];
    }
    if (tid == 0) {
      T->cur = cur;
      T->streamed = streamed ? 1 : 0;
    }
  }
}

// Initial state and reservoir tables: one block per tube.
template <typename Store, typename Real>
__global__ void k_batch_init(TubeDev<Real>* __restrict__ tubes, const double* __restrict__ rho,
                             const double* __restrict__ u, const double* __restrict__ T,
                             const double* __restrict__ R, int64_t total_pts,
                             const double* __restrict__ res, Store* __restrict__ pop0,
                             Real* __restrict__ e_state, Real* __restrict__ ux_state) {
  TubeDev<Real>* tb = tubes + blockIdx.x;
  const StepConst<Real> K = tb->K;
  const Real hdt = tb->hdt;
  const int nx = tb->nx, np = 2 * nx;
  const int64_t off = tb->pt_off;
  Store* base = pop0 + tb->pop_off;
  for (int p = threadIdx.x; p < np; p += blockDim.x) {
    const PointIdx P = tube_point(nx, p);
    const int64_t g = off + p;
    Real h[kQ], e;
    init_point<Real, true>(K, hdt, rho[g], u[g], u[total_pts + g], u[2 * total_pts + g], T[g], R[g], h, e);
    Store* out = base + (int64_t)(P.s * kQ) * K.n3 + P.cell;
#pragma unroll
    for (int q = 0; q < kQ; ++q) out[(int64_t)q * K.n3] = from_real<Store, Real>(h[q]);
    e_state[g] = e;
    ux_state[g] = Real(u[g]);
  }
  if (threadIdx.x < 2) {
    const int side = threadIdx.x;
    const double* st = res + 12 * (int64_t)blockIdx.x + 6 * side;
    Real h[kQ], e;
    init_point<Real, true>(K, hdt, st[0], st[1], st[2], st[3], st[4], st[5], h, e);
    Real* gg = tb->ghost + side * kGhostStride;
    for (int q = 0; q < kQ; ++q) gg[q] = h[q];
    gg[kGhE] = e;
    gg[kGhDrho] = Real(st[0] - 1.0);
    gg[kGhU] = Real(st[1]);
    gg[kGhU + 1] = Real(st[2]);
    gg[kGhU + 2] = Real(st[3]);
    const double theta = (3.0 * st[4] + (double)K.delta * st[5]) / (3.0 + (double)K.delta);
    gg[kGhKap] = Real((double)K.kapc * st[0] * theta);
  }
  if (threadIdx.x == 0) {
    tb->cur = 0;
    tb->streamed = 1;
  }
}

// Moments of the current state, one block per tube (FP64 outputs).
template <typename Store, typename Real>
__global__ void k_batch_moments(const TubeDev<Real>* __restrict__ tubes, const Store* __restrict__ pop0,
                                const Store* __restrict__ pop1, const Real* __restrict__ e_state,
                                int64_t total_pts, double* __restrict__ out) {
  const TubeDev<Real>* tb = tubes + blockIdx.x;
  const StepConst<Real> K = tb->K;
  const int nx = tb->nx, np = 2 * nx;
  const Store* pin = (tb->cur ? pop1 : pop0) + tb->pop_off;
  const int64_t off = tb->pt_off;
  for (int p = threadIdx.x; p < np; p += blockDim.x) {
    const PointIdx P = tube_point(nx, p);
    Real h[kQ];
    if (tb->streamed)
      gather<Store, Real, false, 1>(pin, tb->ghost, K, P, h);
    else
      gather<Store, Real, true, 1>(pin, tb->ghost, K, P, h);
    Mom<Real> m;
    raw_moments_shells(h, m);
    recover(m, e_state[off + p], K);
    const int64_t g = off + p;
    const double rh = 1.0 + to_double(m.drho), thR = to_double(K.theta0) + to_double(m.dR);
    out[g] = rh;
    out[total_pts + g] = to_double(m.j[0] * m.inv_rho);
    out[2 * total_pts + g] = to_double(m.j[1] * m.inv_rho);
    out[3 * total_pts + g] = to_double(m.j[2] * m.inv_rho);
    out[4 * total_pts + g] = to_double(K.theta0) + to_double(m.dT);
    out[5 * total_pts + g] = thR;
    out[6 * total_pts + g] = 0.5 * to_double(K.delta) * rh * thR;
  }
}

// Moment blocks (per tube [4][2 nx] floats: rho, u_x, theta_T, E_R, at float
// offset 4 pt_off) -> the FP64 staging rows read by k_batch_init (rho, u (3
// rows), theta_T, theta_R). theta_R = 2 E_R / (delta rho); theta_T when delta = 0.
// Non-positive or non-finite values set bit 2 of the status word.
template <typename Real>
__global__ void k_state_to_stage(const TubeDev<Real>* __restrict__ tubes, const float* __restrict__ state,
                                 int64_t n, double* __restrict__ stage, unsigned* __restrict__ status) {
  const TubeDev<Real>* tb = tubes + blockIdx.x;
  const int np = 2 * tb->nx;
  const int64_t off = tb->pt_off;
  const float* s = state + 4 * off;
  const double delta = (double)tb->K.delta;
  bool bad = false;
  for (int p = threadIdx.x; p < np; p += blockDim.x) {
    const double rho = s[p], ux = s[np + p], T = s[2 * np + p], er = s[3 * np + p];
    const double R = delta > 0.0 ? 2.0 * er / (delta * rho) : T;
    bad |= !(rho > 0.0) || !(T > 0.0) || !(R > 0.0) || !isfinite(rho) || !isfinite(ux) ||
           !isfinite(T) || !isfinite(R);
    stage[off + p] = rho;
    stage[n + off + p] = ux;
    stage[2 * n + off + p] = 0.0;
    stage[3 * n + off + p] = 0.0;
    stage[4 * n + off + p] = T;
    stage[5 * n + off + p] = R;
  }
  if (bad) atomicOr(status, 4u);
}

// FP64 moment rows of k_batch_moments -> moment blocks (rho, u_x, theta_T, E_R).
template <typename Real>
__global__ void k_stage_to_state(const TubeDev<Real>* __restrict__ tubes, const double* __restrict__ stage,
                                 int64_t n, float* __restrict__ state) {
  const TubeDev<Real>* tb = tubes + blockIdx.x;
  const int np = 2 * tb->nx;
  const int64_t off = tb->pt_off;
  float* s = state + 4 * off;
  for (int p = threadIdx.x; p < np; p += blockDim.x) {
    s[p] = (float)stage[off + p];
    s[np + p] = (float)stage[n + off + p];
    s[2 * np + p] = (float)stage[4 * n + off + p];
    s[3 * np + p] = (float)stage[6 * n + off + p];
  }
}

template <typename Real>
__global__ void k_set_steps(TubeDev<Real>* __restrict__ tubes, const int* __restrict__ nsteps, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) tubes[i].nsteps = nsteps[i];
}

}  // namespace rpk

using namespace rpk;

struct rpk_batch {
  int precision = RPK_F32, ntubes = 0, save_every = 1, device = 0;
  cudaStream_t stream = nullptr;
  std::vector<rpk_tube> tubes;
  std::vector<int> nsub;
  std::vector<int64_t> pt_off, snap_off;
  int64_t total_pts = 0, pop_elems = 0, snap_floats = 0;
  int max_nx = 0;
  size_t real_elem = 4, store_elem = 4;
  void* pop[2] = {nullptr, nullptr};
  void* e_state = nullptr;
  void* ux_state = nullptr;
  void* tubes_dev = nullptr;
  int* order_dev = nullptr;
  int* counter = nullptr;
  float* snaps = nullptr;
  unsigned* status = nullptr;
  double* stage = nullptr;  // 7 x total_pts doubles, for init and reads
  double* res_dev = nullptr;  // 12 reservoir values per tube
  int* steps_dev = nullptr;   // per-tube step counts for rpk_batch_set_steps
  std::vector<int> max_steps; // step counts given at creation (bound the snapshot storage)
  bool nsub_ok = false;       // every tube's FTCS sub-step count is resolved
  int implicit = 0;           // rotational diffusion: 0 FTCS sub-steps, 1 backward Euler
  bool init_ok = false;
  int threads = 256, ctas_per_sm = 1;
  cudaGraphExec_t graph = nullptr;
  int graph_threads = 0, graph_ctas = 0, graph_implicit = 0;
};

namespace {

template <typename Store, typename Real>
struct BatchOps {
  // one kernel per thread count and diffusion, so that neither form's registers
  // bind the other. 256 threads in FP32 take 254 registers; several CTAs per SM of
  // tubes up to kTwoCtaCells take a kernel held to the 128 that two leave. Two CTAs
  // of 256 per SM, ms, backward Euler / FTCS: 1216 tubes of 60 to 150 cells 2.16 / 1.43
  // -> 1.56 / 1.02, of 500 to 700 6.30 / 6.49 -> 5.74 / 5.44; 456 of 1000 to 1500 5.04 /
  // 5.49 -> 5.17 / 5.55, so longer tubes keep the kernel with all registers.
  static constexpr int kTwoCtaCells = 1000;
  template <bool kImplicit>
  static void* kernel_of(int threads, bool two) {
    constexpr int kTwo = sizeof(Real) == 4 ? 2 : 0;
    switch (threads) {
      case 128: return (void*)k_batch<Store, Real, 128, kImplicit, 0>;
      case 256:
        return two ? (void*)k_batch<Store, Real, 256, kImplicit, kTwo> : (void*)k_batch<Store, Real, 256, kImplicit, 0>;
      case 384: return (void*)k_batch<Store, Real, 384, kImplicit, 0>;
      case 512: return (void*)k_batch<Store, Real, 512, kImplicit, 0>;
      default: return nullptr;
    }
  }
  static void* kernel(const rpk_batch* B, int threads, int ctas) {
    const bool two = ctas >= 2 && B->max_nx <= kTwoCtaCells;
    return B->implicit ? kernel_of<true>(threads, two) : kernel_of<false>(threads, two);
  }
};

bool supported_threads(int t) { return t == 128 || t == 256 || t == 384 || t == 512; }

size_t batch_smem(const rpk_batch* B) {
  const size_t n = B->max_nx, blocks = (n + kBE - 1) / kBE;
  return (kBatchArrays * 2 * n + (B->implicit ? 4 * blocks : 2 * n)) * B->real_elem;
}

size_t batch_smem_rule(const rpk_batch* B) { return (size_t)kBatchRuleArrays * 2 * B->max_nx * B->real_elem; }

template <typename F>
rpk_status with_batch_types(int precision, F&& f) {
  if (precision == RPK_F64) return f(BatchOps<double, double>{}, (double*)nullptr);
  return f(BatchOps<float, float>{}, (float*)nullptr);
}

void free_batch(rpk_batch* B) {
  if (B->graph) cudaGraphExecDestroy(B->graph);
  void* ptrs[] = {B->pop[0], B->pop[1], B->e_state, B->ux_state, B->tubes_dev, B->order_dev,
                  B->counter, B->snaps,  B->status, B->stage,    B->res_dev,   B->steps_dev};
  for (void* p : ptrs)
    if (p) cudaFree(p);
}

rpk_status dev_alloc(void** p, size_t bytes) {
  cudaError_t err = cudaMalloc(p, bytes);
  if (err != cudaSuccess) {
    *p = nullptr;
    cudaGetLastError();
    return fail(err == cudaErrorMemoryAllocation ? RPK_ERR_OOM : RPK_ERR_CUDA,
                std::string("batch allocation failed: ") + cudaGetErrorString(err));
  }
  return RPK_OK;
}

// Work order of the queue: longest work first (collide work ~ points x steps,
// diffusion ~ points x steps x nsub).
rpk_status upload_order(rpk_batch* B) {
  std::vector<int> order(B->ntubes);
  for (int i = 0; i < B->ntubes; ++i) order[i] = i;
  std::vector<double> work(B->ntubes);
  for (int i = 0; i < B->ntubes; ++i)
    work[i] = 2.0 * B->tubes[i].nx * B->tubes[i].nsteps * (8.0 + (B->implicit ? 4.0 : B->nsub[i]));
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return work[a] > work[b]; });
  RPK_CUDA(cudaMemcpyAsync(B->order_dev, order.data(), sizeof(int) * B->ntubes,
                           cudaMemcpyHostToDevice, B->stream));
  RPK_CUDA(cudaStreamSynchronize(B->stream));
  return RPK_OK;
}

// Upload the tube descriptors (constants, offsets, nsub) and the work order.
template <typename Real>
rpk_status upload_tubes(rpk_batch* B) {
  std::vector<TubeDev<Real>> td(B->ntubes);
  int64_t pop_off = 0;
  for (int i = 0; i < B->ntubes; ++i) {
    const rpk_tube& t = B->tubes[i];
    TubeDev<Real>& d = td[i];
    std::memset(&d, 0, sizeof(d));
    d.K = make_step_const<Real>(t.relax, B->nsub[i], t.nx, 1, 1);
    d.hdt = Real(0.5 * t.relax.dt / t.relax.tau1);
    d.nx = t.nx;
    d.nsteps = t.nsteps;
    d.nsub = B->nsub[i];
    d.cur = 0;
    d.streamed = 1;
    d.pop_off = pop_off;
    d.pt_off = B->pt_off[i];
    d.snap_off = B->snap_off[i];
    pop_off += (int64_t)2 * kQ * t.nx;
  }
  RPK_CUDA(cudaMemcpyAsync(B->tubes_dev, td.data(), sizeof(TubeDev<Real>) * B->ntubes,
                           cudaMemcpyHostToDevice, B->stream));
  RPK_CUDA(cudaStreamSynchronize(B->stream));
  return upload_order(B);
}

// Shared-memory limit of the kernel variant (outside any stream capture).
template <typename Store, typename Real>
rpk_status prepare_batch(rpk_batch* B, int threads, int ctas_per_sm) {
  void* kfn = BatchOps<Store, Real>::kernel(B, threads, ctas_per_sm);
  if (!kfn) return fail(RPK_ERR_ARG, "unsupported thread count");
  RPK_CUDA(cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)batch_smem(B)));
  return RPK_OK;
}

template <typename Store, typename Real>
rpk_status launch_batch(rpk_batch* B, cudaStream_t stream, int threads, int ctas_per_sm) {
  int nsm = 0;
  RPK_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, B->device));
  const size_t smem = batch_smem(B);
  const int grid = std::max(1, std::min(B->ntubes, nsm * ctas_per_sm));
  RPK_CUDA(cudaMemsetAsync(B->counter, 0, sizeof(int), stream));
  TubeDev<Real>* tubes = static_cast<TubeDev<Real>*>(B->tubes_dev);
  Store* p0 = static_cast<Store*>(B->pop[0]);
  Store* p1 = static_cast<Store*>(B->pop[1]);
  Real* es = static_cast<Real*>(B->e_state);
  Real* us = static_cast<Real*>(B->ux_state);
  const int max_np = 2 * B->max_nx;
  void* kfn = BatchOps<Store, Real>::kernel(B, threads, ctas_per_sm);
  int ntubes = B->ntubes, save_every = B->save_every;
  // both population buffers of the tubes that run at a time, against L2
  int l2 = 0;
  RPK_CUDA(cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, B->device));
  int prefetch = (double)B->total_pts / ntubes * grid * 2 * kQ * sizeof(Store) > (double)l2;
  void* args[] = {&tubes, &B->order_dev, &ntubes, &B->counter, &p0,         &p1,
                  &es,    &us,           &B->snaps, &save_every, (void*)&max_np, &prefetch, &B->status};
  RPK_CUDA(cudaLaunchKernel(kfn, dim3(grid), dim3(threads), args, smem, stream));
  RPK_CUDA(cudaGetLastError());
  return RPK_OK;
}

// Tube descriptors, then the initial state from the staging rows (filled from
// host fields before the call, or from device moment blocks here).
rpk_status init_from_stage(rpk_batch* B, const float* state) {
  const int64_t n = B->total_pts;
  double* s = B->stage;
  rpk_status st = with_batch_types(B->precision, [&](auto ops, auto* real_tag) {
    using Real = std::remove_pointer_t<decltype(real_tag)>;
    return upload_tubes<Real>(B);
  });
  if (st != RPK_OK) return st;
  RPK_CUDA(cudaMemsetAsync(B->status, 0, sizeof(unsigned), B->stream));
  if (B->precision == RPK_F64) {
    auto* td = static_cast<TubeDev<double>*>(B->tubes_dev);
    if (state) k_state_to_stage<double><<<B->ntubes, 256, 0, B->stream>>>(td, state, n, s, B->status);
    k_batch_init<double, double><<<B->ntubes, 256, 0, B->stream>>>(
        td, s, s + n, s + 4 * n, s + 5 * n, n, B->res_dev, static_cast<double*>(B->pop[0]),
        static_cast<double*>(B->e_state), static_cast<double*>(B->ux_state));
  } else {
    auto* td = static_cast<TubeDev<float>*>(B->tubes_dev);
    if (state) k_state_to_stage<float><<<B->ntubes, 256, 0, B->stream>>>(td, state, n, s, B->status);
    k_batch_init<float, float><<<B->ntubes, 256, 0, B->stream>>>(
        td, s, s + n, s + 4 * n, s + 5 * n, n, B->res_dev, static_cast<float*>(B->pop[0]),
        static_cast<float*>(B->e_state), static_cast<float*>(B->ux_state));
  }
  RPK_CUDA(cudaGetLastError());
  RPK_CUDA(cudaStreamSynchronize(B->stream));
  B->init_ok = true;
  return RPK_OK;
}

bool config_fits(const rpk_batch* B, int threads, int ctas) {
  return supported_threads(threads) && ctas >= 1 && batch_smem_rule(B) * ctas <= kBatchSmemLimit &&
         threads * ctas <= 2048;
}

}  // namespace

extern "C" {

int rpk_batch_max_nx(int precision) {
  const size_t real = precision == RPK_F64 ? 8 : 4;
  return (int)((kBatchSmemLimit - 1024) / (kBatchRuleArrays * 2 * real));
}

rpk_status rpk_batch_create(int precision, int ntubes, const rpk_tube* tubes, int save_every,
                            void* cuda_stream, rpk_batch** out) {
  if (!out || !tubes) return fail(RPK_ERR_ARG, "NULL argument");
  *out = nullptr;
  if (precision != RPK_F64 && precision != RPK_F32)
    return fail(RPK_ERR_ARG, "batched tubes support RPK_F64 and RPK_F32");
  if (ntubes < 1) return fail(RPK_ERR_ARG, "ntubes must be >= 1");
  if (save_every < 1) return fail(RPK_ERR_ARG, "save_every must be >= 1");
  const int max_nx = rpk_batch_max_nx(precision);
  for (int i = 0; i < ntubes; ++i) {
    const rpk_tube& t = tubes[i];
    if (t.nx < 2 || t.nx > max_nx)
      return fail(RPK_ERR_ARG, "tube " + std::to_string(i) + ": nx must lie in [2, " +
                                   std::to_string(max_nx) + "] for this precision");
    if (t.nsteps < 0) return fail(RPK_ERR_ARG, "tube " + std::to_string(i) + ": nsteps < 0");
    rpk_status st = validate_relax(&t.relax);
    if (st != RPK_OK) return fail(st, "tube " + std::to_string(i) + ": " + rpk_last_error());
    for (int side = 0; side < 2; ++side) {
      const double* r = t.res + 6 * side;
      if (!(r[0] > 0.0) || !(r[4] > 0.0) || !(r[5] > 0.0))
        return fail(RPK_ERR_PARAM, "tube " + std::to_string(i) + ": reservoir rho, theta must be > 0");
    }
  }
  rpk_batch* B = new (std::nothrow) rpk_batch();
  if (!B) return fail(RPK_ERR_OOM, "host allocation failed");
  B->precision = precision;
  B->ntubes = ntubes;
  B->save_every = save_every;
  B->stream = static_cast<cudaStream_t>(cuda_stream);
  B->tubes.assign(tubes, tubes + ntubes);
  B->nsub.assign(ntubes, 1);
  B->real_elem = B->store_elem = precision == RPK_F64 ? 8 : 4;
  cudaError_t err = cudaGetDevice(&B->device);
  if (err != cudaSuccess) {
    delete B;
    return cuda_fail(err, "cudaGetDevice");
  }
  B->pt_off.resize(ntubes);
  B->snap_off.resize(ntubes);
  for (int i = 0; i < ntubes; ++i) {
    B->pt_off[i] = B->total_pts;
    B->snap_off[i] = B->snap_floats;
    const int64_t np = 2 * (int64_t)tubes[i].nx;
    const int64_t nsnap = (tubes[i].nsteps + save_every - 1) / save_every;
    B->total_pts += np;
    B->snap_floats += nsnap * 4 * np;
    B->max_nx = std::max(B->max_nx, tubes[i].nx);
  }
  B->pop_elems = (int64_t)kQ * B->total_pts;
  const size_t tube_bytes = precision == RPK_F64 ? sizeof(TubeDev<double>) : sizeof(TubeDev<float>);
  rpk_status st = RPK_OK;
  if (st == RPK_OK) st = dev_alloc(&B->pop[0], B->pop_elems * B->store_elem);
  if (st == RPK_OK) st = dev_alloc(&B->pop[1], B->pop_elems * B->store_elem);
  if (st == RPK_OK) st = dev_alloc(&B->e_state, B->total_pts * B->real_elem);
  if (st == RPK_OK) st = dev_alloc(&B->ux_state, B->total_pts * B->real_elem);
  if (st == RPK_OK) st = dev_alloc(&B->tubes_dev, tube_bytes * ntubes);
  if (st == RPK_OK) st = dev_alloc((void**)&B->order_dev, sizeof(int) * ntubes);
  if (st == RPK_OK) st = dev_alloc((void**)&B->counter, sizeof(int));
  if (st == RPK_OK) st = dev_alloc((void**)&B->snaps, std::max<int64_t>(1, B->snap_floats) * sizeof(float));
  if (st == RPK_OK) st = dev_alloc((void**)&B->status, sizeof(unsigned));
  if (st == RPK_OK) st = dev_alloc((void**)&B->stage, sizeof(double) * 7 * B->total_pts);
  if (st == RPK_OK) st = dev_alloc((void**)&B->res_dev, sizeof(double) * 12 * ntubes);
  if (st == RPK_OK) st = dev_alloc((void**)&B->steps_dev, sizeof(int) * ntubes);
  if (st == RPK_OK) {
    std::vector<double> res(12 * (size_t)ntubes);
    for (int i = 0; i < ntubes; ++i) std::memcpy(&res[12 * (size_t)i], tubes[i].res, 12 * sizeof(double));
    cudaError_t e = cudaMemcpyAsync(B->res_dev, res.data(), res.size() * sizeof(double),
                                    cudaMemcpyHostToDevice, B->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(B->stream);
    if (e != cudaSuccess) st = cuda_fail(e, "rpk_batch_create");
  }
  if (st != RPK_OK) {
    free_batch(B);
    delete B;
    return st;
  }
  B->max_steps.resize(ntubes);
  B->nsub_ok = true;
  for (int i = 0; i < ntubes; ++i) {
    B->max_steps[i] = tubes[i].nsteps;
    if (tubes[i].relax.nsub > 0)
      B->nsub[i] = tubes[i].relax.nsub;
    else
      B->nsub_ok = false;
  }
  *out = B;
  return RPK_OK;
}

void rpk_batch_destroy(rpk_batch* B) {
  if (!B) return;
  cudaStreamSynchronize(B->stream);
  free_batch(B);
  delete B;
}

rpk_status rpk_batch_init(rpk_batch* B, const double* rho, const double* u, const double* T,
                          const double* R) {
  if (!B || !rho || !u || !T || !R) return fail(RPK_ERR_ARG, "NULL argument");
  RPK_CUDA(cudaSetDevice(B->device));
  const int64_t n = B->total_pts;
  for (int64_t p = 0; p < n; ++p)
    if (!(rho[p] > 0.0) || !(T[p] > 0.0) || !(R[p] > 0.0) || !std::isfinite(rho[p]) ||
        !std::isfinite(T[p]) || !std::isfinite(R[p]))
      return fail(RPK_ERR_PARAM, "fields need finite rho > 0, theta_T > 0, theta_R > 0");
  for (int64_t p = 0; p < 3 * n; ++p)
    if (!std::isfinite(u[p])) return fail(RPK_ERR_PARAM, "u not finite");
  // FTCS sub-steps per tube (rpk_auto_nsub with one active axis when nsub = 0)
  for (int i = 0; i < B->ntubes; ++i) {
    const rpk_tube& t = B->tubes[i];
    if (t.relax.nsub > 0) {
      B->nsub[i] = t.relax.nsub;
      continue;
    }
    double tmax = 0.0;
    for (int64_t p = B->pt_off[i]; p < B->pt_off[i] + 2 * t.nx; ++p)
      tmax = std::max(tmax, (3.0 * T[p] + t.relax.delta * R[p]) / (3.0 + t.relax.delta));
    for (int side = 0; side < 2; ++side)
      tmax = std::max(tmax, (3.0 * t.res[6 * side + 4] + t.relax.delta * t.res[6 * side + 5]) /
                                (3.0 + t.relax.delta));
    B->nsub[i] = rpk_auto_nsub(&t.relax, tmax, 1);
  }
  B->nsub_ok = true;
  double* s = B->stage;
  RPK_CUDA(cudaMemcpyAsync(s, rho, n * sizeof(double), cudaMemcpyHostToDevice, B->stream));
  RPK_CUDA(cudaMemcpyAsync(s + n, u, 3 * n * sizeof(double), cudaMemcpyHostToDevice, B->stream));
  RPK_CUDA(cudaMemcpyAsync(s + 4 * n, T, n * sizeof(double), cudaMemcpyHostToDevice, B->stream));
  RPK_CUDA(cudaMemcpyAsync(s + 5 * n, R, n * sizeof(double), cudaMemcpyHostToDevice, B->stream));
  return init_from_stage(B, nullptr);
}

rpk_status rpk_batch_init_device(rpk_batch* B, const float* state) {
  if (!B || !state) return fail(RPK_ERR_ARG, "NULL argument");
  if (!B->nsub_ok)
    return fail(RPK_ERR_STATE, "FTCS sub-step counts unresolved: give relax.nsub > 0 for every "
                               "tube or initialise once from host fields");
  RPK_CUDA(cudaSetDevice(B->device));
  return init_from_stage(B, state);
}

rpk_status rpk_batch_set_steps(rpk_batch* B, const int* nsteps) {
  if (!B || !nsteps) return fail(RPK_ERR_ARG, "NULL argument");
  for (int i = 0; i < B->ntubes; ++i)
    if (nsteps[i] < 0 || nsteps[i] > B->max_steps[i])
      return fail(RPK_ERR_ARG, "tube " + std::to_string(i) + ": nsteps must lie in [0, " +
                                   std::to_string(B->max_steps[i]) + "] (its count at creation)");
  RPK_CUDA(cudaSetDevice(B->device));
  for (int i = 0; i < B->ntubes; ++i) B->tubes[i].nsteps = nsteps[i];
  if (!B->init_ok) return RPK_OK;  // uploaded with the tube descriptors at initialisation
  RPK_CUDA(cudaMemcpyAsync(B->steps_dev, nsteps, sizeof(int) * B->ntubes, cudaMemcpyHostToDevice,
                           B->stream));
  const int blocks = (B->ntubes + 255) / 256;
  if (B->precision == RPK_F64)
    k_set_steps<double><<<blocks, 256, 0, B->stream>>>(static_cast<TubeDev<double>*>(B->tubes_dev),
                                                        B->steps_dev, B->ntubes);
  else
    k_set_steps<float><<<blocks, 256, 0, B->stream>>>(static_cast<TubeDev<float>*>(B->tubes_dev),
                                                       B->steps_dev, B->ntubes);
  RPK_CUDA(cudaGetLastError());
  return upload_order(B);  // synchronises the stream
}

rpk_status rpk_batch_moments_device(rpk_batch* B, float* state) {
  if (!B || !state) return fail(RPK_ERR_ARG, "NULL argument");
  if (!B->init_ok) return fail(RPK_ERR_STATE, "initialise the batch first");
  RPK_CUDA(cudaSetDevice(B->device));
  const int64_t n = B->total_pts;
  if (B->precision == RPK_F64) {
    const auto* td = static_cast<const TubeDev<double>*>(B->tubes_dev);
    k_batch_moments<double, double><<<B->ntubes, 256, 0, B->stream>>>(
        td, static_cast<const double*>(B->pop[0]), static_cast<const double*>(B->pop[1]),
        static_cast<const double*>(B->e_state), n, B->stage);
    k_stage_to_state<double><<<B->ntubes, 256, 0, B->stream>>>(td, B->stage, n, state);
  } else {
    const auto* td = static_cast<const TubeDev<float>*>(B->tubes_dev);
    k_batch_moments<float, float><<<B->ntubes, 256, 0, B->stream>>>(
        td, static_cast<const float*>(B->pop[0]), static_cast<const float*>(B->pop[1]),
        static_cast<const float*>(B->e_state), n, B->stage);
    k_stage_to_state<float><<<B->ntubes, 256, 0, B->stream>>>(td, B->stage, n, state);
  }
  RPK_CUDA(cudaGetLastError());
  return RPK_OK;
}

rpk_status rpk_batch_set_diffusion(rpk_batch* B, int mode) {
  if (!B) return fail(RPK_ERR_ARG, "NULL batch");
  if (mode != 0 && mode != 1) return fail(RPK_ERR_ARG, "mode must be 0 (FTCS) or 1 (backward Euler)");
  B->implicit = mode;
  return RPK_OK;
}

rpk_status rpk_batch_set_config(rpk_batch* B, int threads, int ctas_per_sm) {
  if (!B) return fail(RPK_ERR_ARG, "NULL batch");
  if (!config_fits(B, threads, ctas_per_sm))
    return fail(RPK_ERR_ARG, "unsupported configuration (threads in {128,256,384,512}; shared "
                             "memory of the CTAs per SM must fit)");
  B->threads = threads;
  B->ctas_per_sm = ctas_per_sm;
  return RPK_OK;
}

rpk_status rpk_batch_run(rpk_batch* B) {
  if (!B) return fail(RPK_ERR_ARG, "NULL batch");
  if (!B->init_ok) return fail(RPK_ERR_STATE, "initialise the batch first");
  RPK_CUDA(cudaSetDevice(B->device));
  if (!B->graph || B->graph_threads != B->threads || B->graph_ctas != B->ctas_per_sm ||
      B->graph_implicit != B->implicit) {
    if (B->graph) {
      cudaGraphExecDestroy(B->graph);
      B->graph = nullptr;
    }
    rpk_status pst = with_batch_types(B->precision, [&](auto ops, auto* real_tag) {
      using Real = std::remove_pointer_t<decltype(real_tag)>;
      return prepare_batch<Real, Real>(B, B->threads, B->ctas_per_sm);
    });
    if (pst != RPK_OK) return pst;
    cudaStream_t cap = nullptr;
    RPK_CUDA(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
    cudaError_t err = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    rpk_status st = RPK_OK;
    if (err == cudaSuccess) {
      st = with_batch_types(B->precision, [&](auto ops, auto* real_tag) {
        using Real = std::remove_pointer_t<decltype(real_tag)>;
        return launch_batch<Real, Real>(B, cap, B->threads, B->ctas_per_sm);
      });
      cudaGraph_t g = nullptr;
      cudaError_t e2 = cudaStreamEndCapture(cap, &g);
      if (st == RPK_OK && e2 == cudaSuccess) e2 = cudaGraphInstantiate(&B->graph, g, 0);
      if (g) cudaGraphDestroy(g);
      err = e2;
    }
    cudaStreamDestroy(cap);
    if (st != RPK_OK) return st;
    if (err != cudaSuccess) return cuda_fail(err, "batch graph capture");
    B->graph_threads = B->threads;
    B->graph_ctas = B->ctas_per_sm;
    B->graph_implicit = B->implicit;
  }
  RPK_CUDA(cudaGraphLaunch(B->graph, B->stream));
  return RPK_OK;
}

rpk_status rpk_batch_read_moments(rpk_batch* B, double* rho, double* u, double* T, double* R,
                                  double* E) {
  if (!B) return fail(RPK_ERR_ARG, "NULL batch");
  if (!B->init_ok) return fail(RPK_ERR_STATE, "initialise the batch first");
  RPK_CUDA(cudaSetDevice(B->device));
  const int64_t n = B->total_pts;
  if (B->precision == RPK_F64)
    k_batch_moments<double, double><<<B->ntubes, 256, 0, B->stream>>>(
        static_cast<const TubeDev<double>*>(B->tubes_dev), static_cast<const double*>(B->pop[0]),
        static_cast<const double*>(B->pop[1]), static_cast<const double*>(B->e_state), n, B->stage);
  else
    k_batch_moments<float, float><<<B->ntubes, 256, 0, B->stream>>>(
        static_cast<const TubeDev<float>*>(B->tubes_dev), static_cast<const float*>(B->pop[0]),
        static_cast<const float*>(B->pop[1]), static_cast<const float*>(B->e_state), n, B->stage);
  RPK_CUDA(cudaGetLastError());
  const size_t b = n * sizeof(double);
  if (rho) RPK_CUDA(cudaMemcpyAsync(rho, B->stage, b, cudaMemcpyDeviceToHost, B->stream));
  if (u) RPK_CUDA(cudaMemcpyAsync(u, B->stage + n, 3 * b, cudaMemcpyDeviceToHost, B->stream));
  if (T) RPK_CUDA(cudaMemcpyAsync(T, B->stage + 4 * n, b, cudaMemcpyDeviceToHost, B->stream));
  if (R) RPK_CUDA(cudaMemcpyAsync(R, B->stage + 5 * n, b, cudaMemcpyDeviceToHost, B->stream));
  if (E) RPK_CUDA(cudaMemcpyAsync(E, B->stage + 6 * n, b, cudaMemcpyDeviceToHost, B->stream));
  unsigned flags = 0;
  RPK_CUDA(cudaMemcpyAsync(&flags, B->status, sizeof(unsigned), cudaMemcpyDeviceToHost, B->stream));
  RPK_CUDA(cudaStreamSynchronize(B->stream));
  if (flags) return fail(RPK_ERR_NUMERIC, "a tube flagged a non-finite or non-positive moment");
  return RPK_OK;
}

rpk_status rpk_batch_snapshots(rpk_batch* B, float* out, int64_t* count) {
  if (!B || !count) return fail(RPK_ERR_ARG, "NULL argument");
  RPK_CUDA(cudaSetDevice(B->device));
  *count = B->snap_floats;
  if (out && B->snap_floats > 0) {
    RPK_CUDA(cudaMemcpyAsync(out, B->snaps, B->snap_floats * sizeof(float), cudaMemcpyDeviceToHost,
                             B->stream));
    RPK_CUDA(cudaStreamSynchronize(B->stream));
  }
  return RPK_OK;
}

rpk_status rpk_batch_autotune(rpk_batch* B, int64_t out[3]) {
  if (!B || !out) return fail(RPK_ERR_ARG, "NULL argument");
  if (!B->init_ok) return fail(RPK_ERR_STATE, "initialise the batch first");
  RPK_CUDA(cudaSetDevice(B->device));
  int nsm = 0;
  RPK_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, B->device));
  // sample: up to 2 tubes per SM spread over the work order, 32 steps each, at rest
  const int nsample = std::min(B->ntubes, 2 * nsm);
  std::vector<rpk_tube> tv;
  for (int i = 0; i < nsample; ++i) {
    rpk_tube t = B->tubes[(int64_t)i * B->ntubes / nsample];
    t.nsteps = std::min(t.nsteps, 32);
    t.relax.nsub = B->nsub[(int64_t)i * B->ntubes / nsample];
    tv.push_back(t);
  }
  rpk_batch* S = nullptr;
  rpk_status st = rpk_batch_create(B->precision, nsample, tv.data(), 1 << 30, B->stream, &S);
  if (st != RPK_OK) return st;
  S->max_nx = B->max_nx;  // same shared-memory footprint as the real launch
  S->implicit = B->implicit;
  std::vector<double> rho(S->total_pts, 1.0), u(3 * S->total_pts, 0.0), T(S->total_pts, kTheta0);
  st = rpk_batch_init(S, rho.data(), u.data(), T.data(), T.data());
  double best_ms = 1e300;
  int best_t = B->threads, best_c = B->ctas_per_sm;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (st == RPK_OK) {
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    const int cand_t[] = {128, 256, 384, 512};
    for (int t : cand_t) {
      for (int c = 1; c <= 4; ++c) {
        if (!config_fits(S, t, c)) continue;
        float ms = 0.f;
        st = with_batch_types(B->precision, [&](auto ops, auto* real_tag) {
          using Real = std::remove_pointer_t<decltype(real_tag)>;
          return prepare_batch<Real, Real>(S, t, c);
        });
        for (int rep = 0; rep < 2 && st == RPK_OK; ++rep) {
          cudaEventRecord(e0, B->stream);
          st = with_batch_types(B->precision, [&](auto ops, auto* real_tag) {
            using Real = std::remove_pointer_t<decltype(real_tag)>;
            return launch_batch<Real, Real>(S, B->stream, t, c);
          });
          cudaEventRecord(e1, B->stream);
          cudaEventSynchronize(e1);
          cudaEventElapsedTime(&ms, e0, e1);
        }
        if (st != RPK_OK) break;
        if (ms < best_ms) {
          best_ms = ms;
          best_t = t;
          best_c = c;
        }
      }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
  }
  rpk_batch_destroy(S);
  if (st != RPK_OK) return st;
  B->threads = best_t;
  B->ctas_per_sm = best_c;
  out[0] = best_t;
  out[1] = best_c;
  out[2] = (int64_t)(best_ms * 1000.0);
  return RPK_OK;
}

}  // extern "C"
