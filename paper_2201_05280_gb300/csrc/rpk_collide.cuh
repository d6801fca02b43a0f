// The fused pull-stream + collide + rotational-exchange kernel (hot path,
// rows a1-a6 of the step; Sec. 5).
#pragma once

#include "rpk_device.cuh"
#include "rpk_pair.cuh"

namespace rpk {

// Collision of one gathered point (or pair of points, V = F2), in place of
// the paper's explicit update (Sec. 5):
//   g' = (1 - 2 beta*) g + 2 beta* f^mix,   in h form: h' = c_keep h + c_relax (f^mix/w - 1)
//   Er' = Er + dt (delta rho/2)(theta - theta_R)/tau1   (rotational exchange)
// hands the 41 relaxed populations to emit(q, value) in the order q = 0, 1, 2, ...
// and, with the moments in m complete, the exchanged auxiliary rotational energy
// (paper mode: theta_R after the first backward-Euler half step with the time-t
// theta_T) to fields(e, m): before the populations (kFieldsFirst) or after them.
template <typename Real, bool kPaper, bool kFieldsFirst, typename V, typename Fields, typename Emit>
__device__ __forceinline__ void collide_emit(const StepConst<Real>& K, const V (&h)[kQ], V e, Fields&& fields,
                                             Emit&& emit, Mom<V>& m) {
  raw_moments(h, m);
  recover<Real, kPaper>(m, e, K);
  auto hand_over = [&] {
    if constexpr (kPaper)
      fields(fmad(K.ra_keep, m.dR, K.ra_t * m.dT), m);
    else
      fields(fmad(K.exc * m.rho, m.dth - m.dR, e), m);
  };
  if constexpr (kFieldsFirst) hand_over();
  Herm<V> H;
  mix_coeffs(m, K, H);
  emit(0, fmad(K.c_keep, h[0], K.c_relax * H.e0));
  static_for<kPairs>([&](auto kc) {
    constexpr int k = decltype(kc)::value;
    constexpr Vel2 v = kPairVel2[k];
    const V ev = herm_even<v.x, v.y, v.z>(H);
    const V od = herm_odd<v.x, v.y, v.z>(H);
    emit(2 * k + 1, fmad(K.c_keep, h[2 * k + 1], K.c_relax * (ev + od)));
    emit(2 * k + 2, fmad(K.c_keep, h[2 * k + 2], K.c_relax * (ev - od)));
  });
  if constexpr (!kFieldsFirst) hand_over();
}

// The same with the shell-wise sums and targets: about 430 operations a point
// instead of 690. FP64 is bound by its pipe (two lanes per cycle and SM): 96^3, 760
// of its instructions a point and 2160 us pair by pair, 422 and 1415 us now (0.9 of
// the pipe's rate).
template <typename Real, bool kPaper, typename V, typename Emit>
__device__ __forceinline__ V collide_shells(const StepConst<Real>& K, const V (&h)[kQ], V e, Emit&& emit,
                                            Mom<V>& m) {
  raw_moments_shells(h, m);
  Herm<V> H;
  relaxed_target<Real, kPaper>(m, e, K, H);
  emit(0, fmad(K.c_keep, h[0], H.e0));
  herm_shells(H, [&](int k, V ev, V od) {
    emit(2 * k + 1, fmad(K.c_keep, h[2 * k + 1], ev + od));
    emit(2 * k + 2, fmad(K.c_keep, h[2 * k + 2], ev - od));
  });
  if constexpr (kPaper)
    return fmad(K.ra_keep, m.dR, K.ra_t * m.dT);
  else
    return fmad(K.exc * m.rho, m.dth - m.dR, e);
}

// One point: population q goes to cell of the plane out + q * n3.
template <typename Store, typename Real, bool kPaper = false>
__device__ __forceinline__ Real collide_point(const StepConst<Real>& K, const Real (&h)[kQ], Real e,
                                              Store* __restrict__ out, unsigned cell, Mom<Real>& m) {
  const int64_t n3 = K.n3;
  auto put = [&](int q, Real v) { (out + (int64_t)q * n3)[cell] = from_real<Store, Real>(v); };
  if constexpr (kShells<Store>) {
    return collide_shells<Real, kPaper>(K, h, e, put, m);
  } else {
    Real es;
    collide_emit<Real, kPaper, false>(K, h, e, [&](Real v, const Mom<Real>&) { es = v; }, put, m);
    return es;
  }
}

// Device status flags: 1 non-finite moment, 2 rho <= 0, 4 theta_T or theta_R <= 0.
template <typename Real>
__device__ __forceinline__ void flag_moments(const Mom<Real>& m, Real theta0,
                                             unsigned* __restrict__ status) {
  const bool ok = (m.rho > Real(0)) && (theta0 + m.dT > Real(0)) && (theta0 + m.dR > Real(0));
  if (!ok) {
    unsigned f = 0;
    if (!(m.rho == m.rho) || !(m.dT == m.dT) || !(m.dR == m.dR)) f |= 1u;
    if (!(m.rho > Real(0))) f |= 2u;
    if (!(theta0 + m.dT > Real(0)) || !(theta0 + m.dR > Real(0))) f |= 4u;
    atomicOr(status, f);
  }
}

// One collision per point after the pull (Sec. 5):
//   g' = (1 - 2 beta*) g + 2 beta* f^mix,   in h form: h' = c_keep h + c_relax (f^mix/w - 1)
//   Er' = Er + dt (delta rho/2)(theta - theta_R)/tau1   (rotational exchange)
// Writes h', e', rho - 1, u (ring slot of this step) and kappa_R.
// FP32/16-bit arithmetic: at most 102 registers, so that five 128-thread blocks
// per SM keep enough loads in flight.
template <typename Store, typename Real, bool kPull, int kBC, bool kPaper>
__global__ void __launch_bounds__(128, sizeof(Real) == 4 ? 5 : 1)
    k_collide(StepConst<Real> K, const Store* pin, Store* __restrict__ pout,
              const Real* e_in, Real* __restrict__ e_out, Real* __restrict__ drho_out,
              Real* __restrict__ u_out, Real* __restrict__ kap_out,
              const Real* __restrict__ ghost, unsigned* __restrict__ status,
              Real* __restrict__ tt_out, const Real* wcol) {
  pdl_wait();
  PointIdx P;
  if (!point_from_block(K, P)) return;
  const int64_t p = (int64_t)P.s * K.n3 + P.cell;
  Real h[kQ];
  gather<Store, Real, kPull, kBC>(pin, ghost, K, P, h, wcol);
  Mom<Real> m;
  const Real es = collide_point<Store, Real, kPaper>(K, h, e_in[p],
                                             pout + (int64_t)(P.s * kQ) * K.n3,
                                             (unsigned)P.cell, m);
  e_out[p] = es;
  drho_out[p] = m.drho;
  const int64_t npts = 2 * K.n3;
  u_out[p] = m.j[0] * m.inv_rho;
  u_out[npts + p] = m.j[1] * m.inv_rho;
  u_out[2 * npts + p] = m.j[2] * m.inv_rho;
  if constexpr (kPaper)
    kap_out[p] = K.kapc * m.rho * fmad(fmad(K.delta, m.dR, Real(3) * m.dT), K.inv_3pd, K.theta0);
  else
    kap_out[p] = K.kapc * m.rho * (K.theta0 + m.dth);
  if constexpr (kPaper) tt_out[p] = m.dT;  // paper mode: theta_T(f) - theta0 of time t
  flag_moments(m, K.theta0, status);
}

// k_collide in FP64 for lattices of one or two warps of points per SM. A quarter of
// an SM issues an FP64 instruction in 64 cycles, however many lanes are active, and
// all four together one in 19: a lone warp's 422 instructions take 27 k cycles with
// three quarters idle. Here four warps share 32 points. Each gathers a group of pairs
// (rest and axes, faces, corners, halves), sums its part of the moments and, after
// an exchange, its part of the target's coefficients; after another it relaxes its
// group: about 185 instructions a warp. 2000-cell tube: a step of 23.7 us became 18.6.
__host__ __device__ constexpr int split_lo(int g) { return g < 3 ? 6 * g : 12 + 4 * (g - 2); }  // first pair of group g

// This group's parts of drho, j and dP (xx yy zz xy xz yz), of raw_moments_shells.
template <int kGroup, typename V>
__device__ __forceinline__ void split_moments(const V (&h)[kQ], V (&p)[10]) {
  constexpr double w1 = pair_weight(0), w2 = pair_weight(3), wf = pair_weight(6), wc = pair_weight(12),
                   wh = pair_weight(16);
  auto ev = [&](int k) { return h[2 * k + 1] + h[2 * k + 2]; };
  auto od = [&](int k) { return h[2 * k + 1] - h[2 * k + 2]; };
  if constexpr (kGroup == 0) {
    const V s0 = ev(0), s1 = ev(1), s2 = ev(2), s3 = ev(3), s4 = ev(4), s5 = ev(5);
    p[0] = fmad(V(w2), s3 + s4 + s5, fmad(V(w1), s0 + s1 + s2, V(kWeightRest) * h[0]));
    p[1] = fmad(V(2 * w2), od(3), V(w1) * od(0));
    p[2] = fmad(V(2 * w2), od(4), V(w1) * od(1));
    p[3] = fmad(V(2 * w2), od(5), V(w1) * od(2));
    p[4] = fmad(V(w1), s0, V(4 * w2) * s3);
    p[5] = fmad(V(w1), s1, V(4 * w2) * s4);
    p[6] = fmad(V(w1), s2, V(4 * w2) * s5);
    p[7] = p[8] = p[9] = V(0);
  } else if constexpr (kGroup == 1) {
    const V ap = ev(6), am = ev(7), bp = ev(8), bm = ev(9), cp = ev(10), cm = ev(11);
    const V A = ap + am, B = bp + bm, C = cp + cm;
    const V oap = od(6), oam = od(7), obp = od(8), obm = od(9), ocp = od(10), ocm = od(11);
    p[0] = V(wf) * (A + B + C);
    p[1] = V(wf) * ((oap + oam) + (obp + obm));
    p[2] = V(wf) * ((oap - oam) + (ocp + ocm));
    p[3] = V(wf) * ((obp - obm) + (ocp - ocm));
    p[4] = V(wf) * (A + B);
    p[5] = V(wf) * (A + C);
    p[6] = V(wf) * (B + C);
    p[7] = V(wf) * (ap - am);
    p[8] = V(wf) * (bp - bm);
    p[9] = V(wf) * (cp - cm);
  } else {
    constexpr int k = split_lo(kGroup);
    constexpr double w = kGroup == 2 ? wc : wh, wj = kGroup == 2 ? wc : 0.5 * wh, wp = kGroup == 2 ? wc : 0.25 * wh;
    auto butterfly = [](V a, V b, V c, V d, V (&o)[4]) {
      const V ab = a + b, cd = c + d, e = a - b, f = c - d;
      o[0] = ab + cd;
      o[1] = ab - cd;
      o[2] = e + f;
      o[3] = e - f;
    };
    V e[4], o[4];
    butterfly(ev(k), ev(k + 1), ev(k + 2), ev(k + 3), e);
    butterfly(od(k), od(k + 1), od(k + 2), od(k + 3), o);
    p[0] = V(w) * e[0];
    p[1] = V(wj) * o[0];
    p[2] = V(wj) * o[1];
    p[3] = V(wj) * o[2];
    p[4] = p[5] = p[6] = V(wp) * e[0];
    p[7] = V(wp) * e[1];
    p[8] = V(wp) * e[2];
    p[9] = V(wp) * e[3];
  }
}

// f(std::integral_constant<int, group>) for the group of this warp.
template <typename F>
__device__ __forceinline__ void split_group(int group, F&& f) {
  if (group == 0)
    f(std::integral_constant<int, 0>{});
  else if (group == 1)
    f(std::integral_constant<int, 1>{});
  else if (group == 2)
    f(std::integral_constant<int, 2>{});
  else
    f(std::integral_constant<int, 3>{});
}

template <bool kPull, int kBC, bool kPaper>
__global__ void __launch_bounds__(128)
    k_collide_split(StepConst<double> K, const double* pin, double* __restrict__ pout, const double* e_in,
                    double* __restrict__ e_out, double* __restrict__ drho_out, double* __restrict__ u_out,
                    double* __restrict__ kap_out, const double* __restrict__ ghost, unsigned* __restrict__ status,
                    double* __restrict__ tt_out, const double* wcol) {
  __shared__ double part[4][10][32];
  __shared__ double coef[20][32];
  pdl_wait();
  const int lane = threadIdx.x & 31, group = threadIdx.x >> 5;
  const unsigned c = blockIdx.x * 32 + lane;
  const bool mine = c < (unsigned)K.n3;
  PointIdx P;
  P.cell = mine ? c : 0u;
  const unsigned row = K.by_nx.div((unsigned)P.cell), z = K.by_ny.div(row);
  P.s = blockIdx.y;
  P.x = (int)((unsigned)P.cell - row * K.nx);
  P.y = (int)(row - z * K.ny);
  P.z = (int)z;
  const int64_t p = (int64_t)P.s * K.n3 + P.cell;
  const double e = e_in[p];
  double own[13];  // the group's populations
  split_group(group, [&](auto gc) {
    constexpr int g = decltype(gc)::value, lo = split_lo(g), hi = split_lo(g + 1), q0 = g ? 2 * lo + 1 : 0;
    double h[kQ], sums[10];
    gather<double, double, kPull, kBC, lo, hi>(pin, ghost, K, P, h, wcol);
    split_moments<g>(h, sums);
#pragma unroll
    for (int k = 0; k < 10; ++k) part[g][k][lane] = sums[k];
#pragma unroll
    for (int q = q0; q < 2 * hi + 1; ++q) own[q - q0] = h[q];
  });
  __syncthreads();
  Mom<double> m;
  {
    double t[10];
#pragma unroll
    for (int k = 0; k < 10; ++k) {
      t[k] = part[1][k][lane] + part[2][k][lane] + part[3][k][lane];
      if (k < 7) t[k] += part[0][k][lane];
    }
    m.drho = t[0];
    m.rho = 1.0 + t[0];
    m.inv_rho = 1.0 / m.rho;
#pragma unroll
    for (int a = 0; a < 3; ++a) m.j[a] = t[1 + a];
#pragma unroll
    for (int a = 0; a < 6; ++a) m.dP[a] = t[4 + a];
  }
  // each group's quarter of the coefficients: the even part and oxyz, or one axis's odd part
  split_group(group, [&](auto gc) {
    constexpr int g = decltype(gc)::value;
    Herm<double> H;
    relaxed_target<double, kPaper>(m, e, K, H);
    auto put = [&](int k, double v) { coef[k][lane] = v; };
    if constexpr (g == 0) {
      put(0, H.e0), put(1, H.exx), put(2, H.eyy), put(3, H.ezz), put(4, H.exy), put(5, H.exz), put(6, H.eyz);
      put(7, H.oxyz);
    } else if constexpr (g == 1) {
      put(8, H.ox), put(9, H.oxxx), put(10, H.oyyx), put(11, H.ozzx);
    } else if constexpr (g == 2) {
      put(12, H.oy), put(13, H.oyyy), put(14, H.oxxy), put(15, H.ozzy);
    } else {
      put(16, H.oz), put(17, H.ozzz), put(18, H.oxxz), put(19, H.oyyz);
    }
  });
  __syncthreads();
  if (!mine) return;
  Herm<double> H;
  {
    auto get = [&](int k) { return coef[k][lane]; };
    H.e0 = get(0), H.exx = get(1), H.eyy = get(2), H.ezz = get(3), H.exy = get(4), H.exz = get(5), H.eyz = get(6);
    H.oxyz = get(7), H.ox = get(8), H.oxxx = get(9), H.oyyx = get(10), H.ozzx = get(11), H.oy = get(12);
    H.oyyy = get(13), H.oxxy = get(14), H.ozzy = get(15), H.oz = get(16), H.ozzz = get(17), H.oxxz = get(18);
    H.oyyz = get(19);
  }
  double* out = pout + (int64_t)(P.s * kQ) * K.n3 + P.cell;
  split_group(group, [&](auto gc) {
    constexpr int g = decltype(gc)::value, lo = split_lo(g), hi = split_lo(g + 1), q0 = g ? 2 * lo + 1 : 0;
    if constexpr (g == 0) out[0] = fmad(K.c_keep, own[0], H.e0);
    herm_shells(H, [&](int k, double ev, double od) {
      if (k < lo || k >= hi) return;
      out[(2 * k + 1) * K.n3] = fmad(K.c_keep, own[2 * k + 1 - q0], ev + od);
      out[(2 * k + 2) * K.n3] = fmad(K.c_keep, own[2 * k + 2 - q0], ev - od);
    });
  });
  const int64_t npts = 2 * K.n3;
  if (group == 1) {
    if constexpr (kPaper)
      e_out[p] = fmad(K.ra_keep, m.dR, K.ra_t * m.dT);
    else
      e_out[p] = fmad(K.exc * m.rho, m.dth - m.dR, e);
    drho_out[p] = m.drho;
  } else if (group == 2) {
    u_out[p] = m.j[0] * m.inv_rho;
    u_out[npts + p] = m.j[1] * m.inv_rho;
    u_out[2 * npts + p] = m.j[2] * m.inv_rho;
  } else if (group == 3) {
    if constexpr (kPaper)
      kap_out[p] = K.kapc * m.rho * fmad(fmad(K.delta, m.dR, 3.0 * m.dT), K.inv_3pd, K.theta0);
    else
      kap_out[p] = K.kapc * m.rho * (K.theta0 + m.dth);
    if constexpr (kPaper) tt_out[p] = m.dT;
    flag_moments(m, K.theta0, status);
  }
}

}  // namespace rpk

namespace rpk {

// Status flags of two points (as flag_moments).
__device__ __forceinline__ void flag_moments2(const Mom<F2>& m, float theta0, unsigned* __restrict__ status) {
  const float rho[2] = {m.rho.v.x, m.rho.v.y}, dT[2] = {m.dT.v.x, m.dT.v.y}, dR[2] = {m.dR.v.x, m.dR.v.y};
#pragma unroll
  for (int l = 0; l < 2; ++l) {
    const bool ok = (rho[l] > 0.0f) && (theta0 + dT[l] > 0.0f) && (theta0 + dR[l] > 0.0f);
    if (!ok) {
      unsigned f = 0;
      if (!(rho[l] == rho[l]) || !(dT[l] == dT[l]) || !(dR[l] == dR[l])) f |= 1u;
      if (!(rho[l] > 0.0f)) f |= 2u;
      if (!(theta0 + dT[l] > 0.0f) || !(theta0 + dR[l] > 0.0f)) f |= 4u;
      atomicOr(status, f);
    }
  }
}

// The pull-stream + collide + exchange step of k_collide for two x-adjacent
// points per thread on a periodic grid with nx even, FP32 arithmetic in
// packed FP32x2 form (the one-point kernel's FP32 arithmetic to rounding, half
// the arithmetic instructions; pair words halve the loads and stores).
// kPaper: the paper's theta_R solver (the state holds theta_R - theta0; the
// time-t theta_T(f) - theta0 goes to tt_out), as in k_collide.
// Bound: the FMA pipes, and registers: four blocks per SM of 16-bit storage leave 128
// for 82 values. The fields are stored before the populations are relaxed, so that
// the moments they come from need not be held until then (spills 172 -> 68 bytes), and
// the paper's solver loads e before the populations (144 -> 52). us at 256^3, FP16 /
// FP16 paper / BF16 / BF16 paper: 1261 / 1261 / 1262 / 1292 with the fields last, now
// 1176 / 1209 / 1245 / 1259. FP16 held as words and converted twice, at five blocks
// per SM (four, paper): 1374 / 1318. FP32 keeps three blocks and does not spill (1703).
template <typename Store, bool kPaper = false>
__global__ void __launch_bounds__(128, sizeof(Store) == 4 ? 3 : 4)
    k_collide_pair(StepConst<float> K, const Store* pin, Store* __restrict__ pout,
                   const float* e_in, float* __restrict__ e_out, float* __restrict__ drho_out,
                   float* __restrict__ u_out, float* __restrict__ kap_out, unsigned* __restrict__ status,
                   float* __restrict__ tt_out) {
  pdl_wait();
  using IO = PairIO<Store>;
  using Word = typename IO::Word;
  int s, i, y, z;
  int64_t cellp;  // pair of the cell
  if (!pair_from_block(K, s, i, y, z, cellp)) return;
  const int64_t n3p = K.n3 >> 1;                // pairs per sublattice
  const int64_t pp = (int64_t)s * n3p + cellp;  // pair in a field plane
  const float2* e2 = reinterpret_cast<const float2*>(e_in) + pp;
  F2 e;
  if constexpr (kPaper) e = F2(*e2);
  F2 h[kQ];
  gather_pair<Store>(reinterpret_cast<const Word*>(pin), K, s, i, y, z, h);
  if constexpr (!kPaper) e = F2(*e2);
  Mom<F2> m;
  Word* out = reinterpret_cast<Word*>(pout) + (int64_t)(s * kQ) * n3p;
  const unsigned cell = (unsigned)cellp;
  collide_emit<float, kPaper, true>(
      K, h, e,
      [&](F2 es, const Mom<F2>& m) {
        reinterpret_cast<float2*>(e_out)[pp] = es.v;
        reinterpret_cast<float2*>(drho_out)[pp] = m.drho.v;
        float2* u2 = reinterpret_cast<float2*>(u_out);
        u2[pp] = (m.j[0] * m.inv_rho).v;
        u2[K.n3 + pp] = (m.j[1] * m.inv_rho).v;
        u2[2 * K.n3 + pp] = (m.j[2] * m.inv_rho).v;
        reinterpret_cast<float2*>(kap_out)[pp] = (K.kapc * m.rho * (K.theta0 + m.dth)).v;
        if constexpr (kPaper) reinterpret_cast<float2*>(tt_out)[pp] = m.dT.v;
        flag_moments2(m, K.theta0, status);
      },
      [&](int q, F2 v) { (out + (int64_t)q * n3p)[cell] = IO::from_f2(v); }, m);
}

}  // namespace rpk
