// Device helpers of the reduced polyatomic ES-BGK lattice-Boltzmann step
// (Kolluru, Atif & Ansumali, arXiv 2201.05280, Sec. 4 and Sec. 5): storage
// conversions, per-launch constants, moments, the f-level recovery, Hermite
// targets and the BCC pull gather.
//
// Data layout (HBM):
//   populations  Store pop[2][41][nz][ny][nx] per buffer, i.e. element
//                (s*41 + q)*n3 + (z*ny + y)*nx + x; two buffers ping-pong.
//                Reduced-precision storage holds h_q = g_q/w_q - 1; FP64 too.
//   scalar fields Real f[2][nz][ny][nx] (point index p = s*n3 + cell).
//   e            auxiliary rotational energy minus delta*theta0/2 (deviation)
//   drho         rho - 1 of the last collision
//   u            two ring slots of 3 planes each: u(t) and u(t-1)
//   kap          kappa_R of the last collision
// The state between steps is "post-collision, pre-stream": the collide kernel
// pulls g(x - c_q) from the previous buffer. Right after initialisation the
// state is post-stream instead (kPull = false reads the point's own slot).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include <utility>

#include "rpk_lattice.cuh"
#include "rpk_vec2.cuh"

namespace rpk {

// ---------------------------------------------------------------------------
// storage conversions

template <typename S, typename R>
__device__ __forceinline__ R to_real(S v) { return static_cast<R>(v); }
template <>
__device__ __forceinline__ float to_real<__half, float>(__half v) { return __half2float(v); }
template <>
__device__ __forceinline__ float to_real<__nv_bfloat16, float>(__nv_bfloat16 v) {
  return __bfloat162float(v);
}
template <typename S, typename R>
__device__ __forceinline__ S from_real(R v) { return static_cast<S>(v); }
template <>
__device__ __forceinline__ __half from_real<__half, float>(float v) { return __float2half_rn(v); }
template <>
__device__ __forceinline__ __nv_bfloat16 from_real<__nv_bfloat16, float>(float v) {
  return __float2bfloat16_rn(v);
}

// FP32 <-> FP64 by integer operations, the same bits as the conversion
// instructions: those go through the FP64 pipe, two lanes per cycle and SM, which
// a pass over a field with FP64 inputs or outputs would otherwise wait for.
__device__ __forceinline__ double to_double(float x) {
  const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
  if (m - 0x00800000u < 0x7f000000u || m == 0u) {  // normal or zero
    const unsigned hi = m ? (m >> 3) + 0x38000000u : 0u;
    return __hiloint2double((int)(hi | (b & 0x80000000u)), (int)(b << 29));
  }
  return (double)x;
}
__device__ __forceinline__ double to_double(double x) { return x; }

template <typename Real>
__device__ __forceinline__ Real round_to(double x);
template <>
__device__ __forceinline__ double round_to<double>(double x) { return x; }
template <>
__device__ __forceinline__ float round_to<float>(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x), m = hi & 0x7fffffffu;
  if (m - 0x38100000u < 0x0fd00000u) {  // rounds to a normal FP32 value
    const unsigned f = ((m - 0x38000000u) << 3) | (lo >> 29), rest = lo & 0x1fffffffu;
    const unsigned up = rest > 0x10000000u || (rest == 0x10000000u && (f & 1u));
    return __uint_as_float((f + up) | (hi & 0x80000000u));
  }
  if ((m | lo) == 0u) return __uint_as_float(hi);
  return (float)x;
}

// x > 0 and finite; x finite
__device__ __forceinline__ bool positive_finite(double x) {
  const long long b = __double_as_longlong(x);
  return b > 0 && b < 0x7ff0000000000000ll;
}
__device__ __forceinline__ bool finite_bits(double x) {
  return ((unsigned)__double2hiint(x) & 0x7ff00000u) != 0x7ff00000u;
}

// compile-time loop: f(std::integral_constant<int, K>) for K = 0..N-1
template <typename F, int... K>
__device__ __forceinline__ void static_for_impl(F&& f, std::integer_sequence<int, K...>) {
  (f(std::integral_constant<int, K>{}), ...);
}
template <int N, typename F>
__device__ __forceinline__ void static_for(F&& f) {
  static_for_impl(f, std::make_integer_sequence<int, N>{});
}

// ---------------------------------------------------------------------------
// per-launch constants (host fills them in double, then casts)

// Division of a 32-bit index by a launch constant, after Granlund and Montgomery
// (Division by invariant integers using multiplication, PLDI 1994): n / d =
// (umulhi(m, n) + n) >> l for n < 2^31, m = floor(2^32 (2^l - d) / d) + 1, l =
// ceil(log2 d).
struct FastDiv {
  unsigned m, l;
  FastDiv() = default;
  explicit FastDiv(unsigned d) {
    l = 0;
    while ((1ull << l) < d) ++l;
    m = (unsigned)(((1ull << 32) * ((1ull << l) - d)) / d + 1);
  }
  __device__ __forceinline__ unsigned div(unsigned n) const { return (__umulhi(m, n) + n) >> l; }
};

template <typename Real>
struct StepConst {
  int nx, ny, nz;
  FastDiv by_nx, by_ny, by_nxp;  // division by nx, ny and nx / 2
  int64_t n3;     // nx*ny*nz
  Real theta0;
  Real c_keep;    // 1 - 2 beta*
  Real c_relax;   // 2 beta*
  Real beta;      // beta* = dt/(2 tau* + dt)
  Real w_es;      // tau*/tau
  Real w_eq;      // tau*/tau1
  Real b;
  Real inv_sig;   // 1 / (1 + dt/(2 tau*) - b dt/(2 tau))
  Real inv_d;     // 1 / (1 + dt/(2 tau1))
  Real delta;
  Real inv_3pd;   // 1 / (3 + delta)
  Real exc;       // dt delta / (2 tau1)
  Real kapc;      // k_r 5 tau / (2 B), kappa_R = kapc * rho * theta
  Real E0;        // delta theta0 / 2
  // Not read: the kernels' pointers then begin 8 bytes past a 16-byte boundary of the
  // arguments. Without it, us a launch: 256^3 BF16 pairs 1267 -> 1296, FP32 one point
  // a thread 161 x 127 x 93 240 -> 248.
  Real spare;
  // products of the above for the shell-wise collision (i = 1 / theta0)
  Real two_id;    // 2 / delta
  Real c_d, c_3;  // delta / (3 + delta), 3 / (3 + delta)
  Real bsig;      // (tau*/tau) b inv_sig
  Real q1h, q1;   // c_relax i / 2, c_relax i
  Real q2h, q2;   // c_relax i^2 / 2, c_relax i^2
  Real q36, q32, q3;  // c_relax i^3 / 6, / 2, / 1
  Real dt;
  Real hsub;      // dt / nsub
  // paper mode of the rotational solver (Sec. 5, four steps on theta_R):
  int paper;      // 1: the state holds theta_R - theta0 instead of the auxiliary energy
  Real ra_keep;   // 1 / (1 + X), X = 3 dt / (2 tau1 (3 + delta)): backward-Euler half step
  Real ra_t;      // X / (1 + X)
  Real pa;        // a = delta X / 3: theta_T(g) = theta_T + a (theta_T - theta_R)
  Real inv_1pa;   // 1 / (1 + a)
};

// Ghost values, one block of kGhostStride per x end (reservoirs, blocks 0, 1)
// or per wall (low / high y wall in blocks 0, 1, low / high x wall in blocks
// 2, 3: h of f^eq(1, u_w, theta_w), its e, rho - 1 = 0, u_w, kappa_R).
constexpr int kGhostStride = 48;
constexpr int kGhostBlocks = 4;

// Boundary kinds of the templated kernels (kBC): 0 periodic; 1 x reservoirs;
// otherwise a mask of diffuse walls, kWallY normal to y and kWallX normal to x.
constexpr int kWallY = 2, kWallX = 4;
enum { kGhE = 41, kGhDrho = 42, kGhU = 43, kGhKap = 46 };

// ---------------------------------------------------------------------------
// moments and Hermite targets (all in deviation form about rho = 1, theta0)

template <typename Real>
struct Mom {
  Real drho, rho, inv_rho;
  Real j[3];
  Real dP[6];    // sum w h c_a c_b: xx yy zz xy xz yz
  Real dTg;      // theta_T(g) - theta0
  Real dth;      // theta - theta0 (eq. thetadef)
  Real dT, dR;   // theta_T(f) - theta0, theta_R - theta0
  Real sig[6];   // sigma(f), a density
};

// rho, j, P of g = w (1 + h), pair by pair. Generic over the value type V
// (float, double, or F2 = the same quantity at two points).
template <typename V>
__device__ __forceinline__ void raw_moments(const V (&h)[kQ], Mom<V>& m) {
  using S = scalar_t<V>;
  V d = S(kWeightRest) * h[0];
  V jx = splat<V>(0), jy = jx, jz = jx, pxx = jx, pyy = jx, pzz = jx, pxy = jx, pxz = jx, pyz = jx;
  static_for<kPairs>([&](auto kc) {
    constexpr int k = decltype(kc)::value;
    constexpr Vel2 v = kPairVel2[k];
    constexpr double w = pair_weight(k);
    const V ev = S(w) * (h[2 * k + 1] + h[2 * k + 2]);
    const V od = S(w) * (h[2 * k + 1] - h[2 * k + 2]);
    d += ev;
    if constexpr (v.x != 0) jx = fmad(S(0.5 * v.x), od, jx);
    if constexpr (v.y != 0) jy = fmad(S(0.5 * v.y), od, jy);
    if constexpr (v.z != 0) jz = fmad(S(0.5 * v.z), od, jz);
    if constexpr (v.x != 0) pxx = fmad(S(0.25 * v.x * v.x), ev, pxx);
    if constexpr (v.y != 0) pyy = fmad(S(0.25 * v.y * v.y), ev, pyy);
    if constexpr (v.z != 0) pzz = fmad(S(0.25 * v.z * v.z), ev, pzz);
    if constexpr (v.x * v.y != 0) pxy = fmad(S(0.25 * v.x * v.y), ev, pxy);
    if constexpr (v.x * v.z != 0) pxz = fmad(S(0.25 * v.x * v.z), ev, pxz);
    if constexpr (v.y * v.z != 0) pyz = fmad(S(0.25 * v.y * v.z), ev, pyz);
  });
  m.drho = d;
  m.rho = S(1) + d;
  m.inv_rho = S(1) / m.rho;
  m.j[0] = jx; m.j[1] = jy; m.j[2] = jz;
  m.dP[0] = pxx; m.dP[1] = pyy; m.dP[2] = pzz;
  m.dP[3] = pxy; m.dP[4] = pxz; m.dP[5] = pyz;
}

// The same sums shell by shell: the weight of a shell multiplies the shell's
// sums once instead of every pair, and the sign patterns of the (1, 1, 1) and
// (1/2, 1/2, 1/2) pairs, (+++), (++-), (+-+), (+--), are one 4-point butterfly for
// the even and one for the odd parts: 138 operations instead of 214. For
// FP64 and batched collisions, and for moments and diagnostics of every storage; the
// collisions of FP32 and 16-bit lattices keep raw_moments (see kShells).
template <typename V>
__device__ __forceinline__ void raw_moments_shells(const V (&h)[kQ], Mom<V>& m) {
  using S = scalar_t<V>;
  constexpr S w1 = S(pair_weight(0)), w2 = S(pair_weight(3)), wf = S(pair_weight(6)), wc = S(pair_weight(12)),
              wh = S(pair_weight(16));
  constexpr S w2j = S(2 * pair_weight(3)), w2p = S(4 * pair_weight(3)), whj = S(0.5 * pair_weight(16)),
              whp = S(0.25 * pair_weight(16));
  auto ev = [&](int k) { return h[2 * k + 1] + h[2 * k + 2]; };
  auto od = [&](int k) { return h[2 * k + 1] - h[2 * k + 2]; };
  // axes
  const V s0 = ev(0), s1 = ev(1), s2 = ev(2), s3 = ev(3), s4 = ev(4), s5 = ev(5);
  // face diagonals: planes xy, xz, yz
  const V ap = ev(6), am = ev(7), bp = ev(8), bm = ev(9), cp = ev(10), cm = ev(11);
  const V A = ap + am, B = bp + bm, C = cp + cm;
  const V oap = od(6), oam = od(7), obp = od(8), obm = od(9), ocp = od(10), ocm = od(11);
  // space diagonals: even sums (all, xy, xz, yz) and odd sums (x, y, z)
  auto butterfly = [](V p, V q, V r, V t, V (&o)[4]) {
    const V pq = p + q, rt = r + t, d = p - q, e = r - t;
    o[0] = pq + rt;
    o[1] = pq - rt;
    o[2] = d + e;
    o[3] = d - e;
  };
  V ce[4], co[4], he[4], ho[4];
  butterfly(ev(12), ev(13), ev(14), ev(15), ce);
  butterfly(od(12), od(13), od(14), od(15), co);
  butterfly(ev(16), ev(17), ev(18), ev(19), he);
  butterfly(od(16), od(17), od(18), od(19), ho);
  V d = S(kWeightRest) * h[0];
  d = fmad(w1, s0 + s1 + s2, d);
  d = fmad(w2, s3 + s4 + s5, d);
  d = fmad(wf, A + B + C, d);
  d = fmad(wc, ce[0], d);
  d = fmad(wh, he[0], d);
  m.drho = d;
  m.rho = S(1) + d;
  m.inv_rho = S(1) / m.rho;
  m.j[0] = fmad(whj, ho[0], fmad(wc, co[0], fmad(wf, (oap + oam) + (obp + obm), fmad(w2j, od(3), w1 * od(0)))));
  m.j[1] = fmad(whj, ho[1], fmad(wc, co[1], fmad(wf, (oap - oam) + (ocp + ocm), fmad(w2j, od(4), w1 * od(1)))));
  m.j[2] = fmad(whj, ho[2], fmad(wc, co[2], fmad(wf, (obp - obm) + (ocp - ocm), fmad(w2j, od(5), w1 * od(2)))));
  const V diag = fmad(whp, he[0], wc * ce[0]);
  m.dP[0] = fmad(w1, s0, fmad(w2p, s3, fmad(wf, A + B, diag)));
  m.dP[1] = fmad(w1, s1, fmad(w2p, s4, fmad(wf, A + C, diag)));
  m.dP[2] = fmad(w1, s2, fmad(w2p, s5, fmad(wf, B + C, diag)));
  m.dP[3] = fmad(whp, he[1], fmad(wc, ce[1], wf * (ap - am)));
  m.dP[4] = fmad(whp, he[2], fmad(wc, ce[2], wf * (bp - bm)));
  m.dP[5] = fmad(whp, he[3], fmad(wc, ce[3], wf * (cp - cm)));
}

// Storage whose one-point kernels use the factored sums and targets: FP64. FP32 and
// 16-bit lattices keep the pair-by-pair form so that their stored states keep their
// bits, not for accuracy: over random states both forms shift mass and energy by the
// same parts in 1e8 a step, which come from the rounded constants they share.
template <typename Store>
constexpr bool kShells = sizeof(Store) == 8;

// f-level moments from g (Sec. 5, g/f relations) and the stored auxiliary
// rotational energy e (deviation) -- or, in paper mode, the stored theta_R:
// then theta_T(f) = (theta_T(g) + a theta_R)/(1 + a) inverts the printed
// theta_T(g) relation.
//   theta_T(g) = (tr P - j^2/rho)/(3 rho)
//   Rt = 2 Er/(delta rho)  (auxiliary rotational temperature)
//   theta = (3 theta_T(g) + delta Rt)/(3 + delta)   (invariant of the transform)
//   D = (theta_T(g) - Rt)/(1 + dt/(2 tau1)) = theta_T(f) - theta_R
//   theta_T(f) = theta + delta D/(3 + delta),  theta_R = theta - 3 D/(3 + delta)
//   sigma(f) = (P - jj/rho - rho theta_T(g) I)/(1 + dt/(2 tau*) - b dt/(2 tau))
template <typename Real, bool kPaper = false, typename V>
__device__ __forceinline__ void recover(Mom<V>& m, V e, const StepConst<Real>& K) {
  using S = scalar_t<V>;
  const S t0 = K.theta0;
  const V jj = fmad(m.j[2], m.j[2], fmad(m.j[1], m.j[1], m.j[0] * m.j[0]));
  const V trdP = m.dP[0] + m.dP[1] + m.dP[2];
  m.dTg = (trdP - jj * m.inv_rho - S(3) * t0 * m.drho) * m.inv_rho * S(1.0 / 3.0);
  if constexpr (kPaper) {
    // paper mode: e is theta_R - theta0 itself
    m.dR = e;
    m.dT = fmad(K.pa, m.dR, m.dTg) * K.inv_1pa;
    m.dth = fmad(K.delta, m.dR, S(3) * m.dT) * K.inv_3pd;
  } else {
    const V dRt = (S(2) * e - K.delta * t0 * m.drho) * m.inv_rho / K.delta;
    m.dth = fmad(K.delta, dRt, S(3) * m.dTg) * K.inv_3pd;
    const V D = (m.dTg - dRt) * K.inv_d;
    m.dT = fmad(K.delta * K.inv_3pd, D, m.dth);
    m.dR = m.dth - (S(3) * K.inv_3pd) * D;
  }
  const V iso = fmad(t0, m.drho, m.rho * m.dTg);
  const V ir = m.inv_rho;
  m.sig[0] = (m.dP[0] - m.j[0] * m.j[0] * ir - iso) * K.inv_sig;
  m.sig[1] = (m.dP[1] - m.j[1] * m.j[1] * ir - iso) * K.inv_sig;
  m.sig[2] = (m.dP[2] - m.j[2] * m.j[2] * ir - iso) * K.inv_sig;
  m.sig[3] = (m.dP[3] - m.j[0] * m.j[1] * ir) * K.inv_sig;
  m.sig[4] = (m.dP[4] - m.j[0] * m.j[2] * ir) * K.inv_sig;
  m.sig[5] = (m.dP[5] - m.j[1] * m.j[2] * ir) * K.inv_sig;
}

// Coefficients of f_q/w_q - 1 for the third-order Hermite expansion of a
// Gaussian (rho, u, Lambda) about the lattice weights; Dl = Lambda - theta0 I.
//   f/w = rho + j.c/t0 + A2:(cc - t0 I)/(2 t0^2) + A3:H3(c)/(6 t0^3)
//   A2 = jj/rho + rho Dl,  A3_abc = j_a j_b j_c/rho^2 + Dl_ab j_c + Dl_bc j_a + Dl_ca j_b
// even part: e0 + sum E_ab c_a c_b ; odd part: sum O_a c_a + cubic terms.
template <typename Real>
struct Herm {
  Real e0, exx, eyy, ezz, exy, exz, eyz;
  Real ox, oy, oz;
  Real oxxx, oyyy, ozzz, oxxy, oxxz, oyyx, oyyz, ozzx, ozzy, oxyz;
};

template <typename V>
__device__ __forceinline__ void hermite(V drho, V rho, V inv_rho, const V (&j)[3], const V (&Dl)[6],
                                        scalar_t<V> t0, Herm<V>& H) {
  using S = scalar_t<V>;
  const V jx = j[0], jy = j[1], jz = j[2];
  const V jxr = jx * inv_rho, jyr = jy * inv_rho, jzr = jz * inv_rho;
  const V a2xx = fmad(jx, jxr, rho * Dl[0]);
  const V a2yy = fmad(jy, jyr, rho * Dl[1]);
  const V a2zz = fmad(jz, jzr, rho * Dl[2]);
  const V a2xy = fmad(jx, jyr, rho * Dl[3]);
  const V a2xz = fmad(jx, jzr, rho * Dl[4]);
  const V a2yz = fmad(jy, jzr, rho * Dl[5]);
  // j_a j_b j_c / rho^2 = (j_a j_b / rho)(j_c / rho)
  const V xx = jx * jxr, yy = jy * jyr, zz = jz * jzr;
  const V dxx = Dl[0], dyy = Dl[1], dzz = Dl[2], dxy = Dl[3], dxz = Dl[4], dyz = Dl[5];
  const V a3xxx = fmad(S(3) * dxx, jx, xx * jxr);
  const V a3yyy = fmad(S(3) * dyy, jy, yy * jyr);
  const V a3zzz = fmad(S(3) * dzz, jz, zz * jzr);
  const V a3xxy = fmad(dxx, jy, fmad(S(2) * dxy, jx, xx * jyr));
  const V a3xxz = fmad(dxx, jz, fmad(S(2) * dxz, jx, xx * jzr));
  const V a3yyx = fmad(dyy, jx, fmad(S(2) * dxy, jy, yy * jxr));
  const V a3yyz = fmad(dyy, jz, fmad(S(2) * dyz, jy, yy * jzr));
  const V a3zzx = fmad(dzz, jx, fmad(S(2) * dxz, jz, zz * jxr));
  const V a3zzy = fmad(dzz, jy, fmad(S(2) * dyz, jz, zz * jyr));
  const V a3xyz = fmad(dxy, jz, fmad(dyz, jx, fmad(dxz, jy, (jx * jyr) * jzr)));
  const S i1 = S(1) / t0;
  const S i2 = i1 * i1;
  const S i3 = i2 * i1;
  // even part
  H.e0 = drho - (S(0.5) * i1) * (a2xx + a2yy + a2zz);
  H.exx = (S(0.5) * i2) * a2xx;
  H.eyy = (S(0.5) * i2) * a2yy;
  H.ezz = (S(0.5) * i2) * a2zz;
  H.exy = i2 * a2xy;
  H.exz = i2 * a2xz;
  H.eyz = i2 * a2yz;
  // odd part: j.c/t0 - t0 * 3 V.c/(6 t0^3), V_a = sum_b A3_abb
  const V vx = a3xxx + a3yyx + a3zzx;
  const V vy = a3xxy + a3yyy + a3zzy;
  const V vz = a3xxz + a3yyz + a3zzz;
  H.ox = fmad(-S(0.5) * i2, vx, jx * i1);
  H.oy = fmad(-S(0.5) * i2, vy, jy * i1);
  H.oz = fmad(-S(0.5) * i2, vz, jz * i1);
  const S s6 = i3 * S(1.0 / 6.0), s2 = i3 * S(0.5);
  H.oxxx = s6 * a3xxx;
  H.oyyy = s6 * a3yyy;
  H.ozzz = s6 * a3zzz;
  H.oxxy = s2 * a3xxy;
  H.oxxz = s2 * a3xxz;
  H.oyyx = s2 * a3yyx;
  H.oyyz = s2 * a3yyz;
  H.ozzx = s2 * a3zzx;
  H.ozzy = s2 * a3zzy;
  H.oxyz = i3 * a3xyz;
}

// hermite for Lambda = (theta0 + D) I.
template <typename V>
__device__ __forceinline__ void hermite_iso(V drho, V rho, V inv_rho, const V (&j)[3], V D, Herm<V>& H) {
  using S = scalar_t<V>;
  constexpr S i1 = S(1) / S(kTheta0), i2 = i1 * i1, i3 = i2 * i1;
  const V jx = j[0], jy = j[1], jz = j[2];
  const V ux = jx * inv_rho, uy = jy * inv_rho, uz = jz * inv_rho;
  const V xx = jx * ux, yy = jy * uy, zz = jz * uz, xy = jx * uy;
  const V rD = rho * D, Dx = D * jx, Dy = D * jy, Dz = D * jz;
  H.e0 = fmad(S(-0.5) * i1, (xx + yy + zz) + S(3) * rD, drho);
  H.exx = S(0.5) * i2 * (xx + rD);
  H.eyy = S(0.5) * i2 * (yy + rD);
  H.ezz = S(0.5) * i2 * (zz + rD);
  H.exy = i2 * xy;
  H.exz = i2 * (jx * uz);
  H.eyz = i2 * (jy * uz);
  const V xxx = fmad(xx, ux, S(3) * Dx), yyy = fmad(yy, uy, S(3) * Dy), zzz = fmad(zz, uz, S(3) * Dz);
  const V xxy = fmad(xx, uy, Dy), xxz = fmad(xx, uz, Dz), yyx = fmad(yy, ux, Dx), yyz = fmad(yy, uz, Dz),
          zzx = fmad(zz, ux, Dx), zzy = fmad(zz, uy, Dy);
  H.ox = fmad(S(-0.5) * i2, xxx + yyx + zzx, i1 * jx);
  H.oy = fmad(S(-0.5) * i2, xxy + yyy + zzy, i1 * jy);
  H.oz = fmad(S(-0.5) * i2, xxz + yyz + zzz, i1 * jz);
  H.oxxx = i3 * S(1.0 / 6.0) * xxx;
  H.oyyy = i3 * S(1.0 / 6.0) * yyy;
  H.ozzz = i3 * S(1.0 / 6.0) * zzz;
  H.oxxy = S(0.5) * i3 * xxy;
  H.oxxz = S(0.5) * i3 * xxz;
  H.oyyx = S(0.5) * i3 * yyx;
  H.oyyz = S(0.5) * i3 * yyz;
  H.ozzx = S(0.5) * i3 * zzx;
  H.ozzy = S(0.5) * i3 * zzy;
  H.oxyz = i3 * (xy * uz);
}

template <int VX, int VY, int VZ, typename V>
__device__ __forceinline__ V herm_even(const Herm<V>& H) {
  using S = scalar_t<V>;
  constexpr double cx = 0.5 * VX, cy = 0.5 * VY, cz = 0.5 * VZ;
  V r = H.e0;
  if constexpr (VX != 0) r = fmad(S(cx * cx), H.exx, r);
  if constexpr (VY != 0) r = fmad(S(cy * cy), H.eyy, r);
  if constexpr (VZ != 0) r = fmad(S(cz * cz), H.ezz, r);
  if constexpr (VX * VY != 0) r = fmad(S(cx * cy), H.exy, r);
  if constexpr (VX * VZ != 0) r = fmad(S(cx * cz), H.exz, r);
  if constexpr (VY * VZ != 0) r = fmad(S(cy * cz), H.eyz, r);
  return r;
}

template <int VX, int VY, int VZ, typename V>
__device__ __forceinline__ V herm_odd(const Herm<V>& H) {
  using S = scalar_t<V>;
  constexpr double cx = 0.5 * VX, cy = 0.5 * VY, cz = 0.5 * VZ;
  V r = splat<V>(0);
  if constexpr (VX != 0) r = fmad(S(cx * cx * cx), H.oxxx, fmad(S(cx), H.ox, r));
  if constexpr (VY != 0) r = fmad(S(cy * cy * cy), H.oyyy, fmad(S(cy), H.oy, r));
  if constexpr (VZ != 0) r = fmad(S(cz * cz * cz), H.ozzz, fmad(S(cz), H.oz, r));
  if constexpr (VX * VY != 0) r = fmad(S(cy * cy * cx), H.oyyx, fmad(S(cx * cx * cy), H.oxxy, r));
  if constexpr (VX * VZ != 0) r = fmad(S(cz * cz * cx), H.ozzx, fmad(S(cx * cx * cz), H.oxxz, r));
  if constexpr (VY * VZ != 0) r = fmad(S(cz * cz * cy), H.ozzy, fmad(S(cy * cy * cz), H.oyyz, r));
  if constexpr (VX * VY * VZ != 0) r = fmad(S(cx * cy * cz), H.oxyz, r);
  return r;
}

// herm_even and herm_odd of all pairs, shell by shell: sums shared between the
// axis, face and space diagonals, and butterflies over the sign patterns (160
// operations instead of 224 for the 20 pairs). emit(k, even, odd).
template <typename V, typename Emit>
__device__ __forceinline__ void herm_shells(const Herm<V>& H, Emit&& emit) {
  using S = scalar_t<V>;
  const V ex = H.e0 + H.exx, ey = H.e0 + H.eyy, ez = H.e0 + H.ezz;
  const V ox = H.ox + H.oxxx, oy = H.oy + H.oyyy, oz = H.oz + H.ozzz;
  emit(0, ex, ox);
  emit(1, ey, oy);
  emit(2, ez, oz);
  emit(3, fmad(S(4), H.exx, H.e0), fmad(S(8), H.oxxx, S(2) * H.ox));
  emit(4, fmad(S(4), H.eyy, H.e0), fmad(S(8), H.oyyy, S(2) * H.oy));
  emit(5, fmad(S(4), H.ezz, H.e0), fmad(S(8), H.ozzz, S(2) * H.oz));
  const V xy = ex + H.eyy, xz = ex + H.ezz, yz = ey + H.ezz;
  const V xa = ox + H.oyyx, ya = oy + H.oxxy;  // plane xy
  const V xb = ox + H.ozzx, zb = oz + H.oxxz;  // plane xz
  const V yc = oy + H.ozzy, zc = oz + H.oyyz;  // plane yz
  emit(6, xy + H.exy, xa + ya);
  emit(7, xy - H.exy, xa - ya);
  emit(8, xz + H.exz, xb + zb);
  emit(9, xz - H.exz, xb - zb);
  emit(10, yz + H.eyz, yc + zc);
  emit(11, yz - H.eyz, yc - zc);
  const V n1 = H.exz + H.eyz, n2 = H.exz - H.eyz;
  {
    const V b = xy + H.ezz, m1 = b + H.exy, m2 = b - H.exy;
    const V X = xa + H.ozzx, Y = ya + H.ozzy, Z = zb + H.oyyz;
    const V a = X + Y, c = X - Y, f = Z + H.oxyz, g = Z - H.oxyz;
    emit(12, m1 + n1, a + f);
    emit(13, m1 - n1, a - f);
    emit(14, m2 + n2, c + g);
    emit(15, m2 - n2, c - g);
    // half velocities: second-order terms times 1/4, third-order times 1/8
    // (X holds the first-order term once: 1/8 + 3/8 = 1/2)
    const V hb = fmad(S(0.25), H.exx + H.eyy + H.ezz, H.e0);
    const V h1 = fmad(S(0.25), H.exy, hb), h2 = fmad(S(-0.25), H.exy, hb);
    const V hX = fmad(S(0.125), X, S(0.375) * H.ox), hY = fmad(S(0.125), Y, S(0.375) * H.oy);
    const V hZ = fmad(S(0.125), Z, S(0.375) * H.oz);
    const V ha = hX + hY, hc = hX - hY, hf = fmad(S(0.125), H.oxyz, hZ), hg = fmad(S(-0.125), H.oxyz, hZ);
    emit(16, fmad(S(0.25), n1, h1), ha + hf);
    emit(17, fmad(S(-0.25), n1, h1), ha - hf);
    emit(18, fmad(S(0.25), n2, h2), hc + hg);
    emit(19, fmad(S(-0.25), n2, h2), hc - hg);
  }
}

// H times the scalar c.
template <typename V>
__device__ __forceinline__ void herm_scale(Herm<V>& H, scalar_t<V> c) {
  V* v = reinterpret_cast<V*>(&H);
#pragma unroll
  for (int i = 0; i < (int)(sizeof(Herm<V>) / sizeof(V)); ++i) v[i] = v[i] * c;
}

// Hermite coefficients of f^mix = tau*(f^ES/tau + f^Eq/tau1) (Sec. 5): both
// targets share rho and u and are linear in Lambda, so
//   Lambda_mix = (tau*/tau)(theta_T I + b sigma/rho) + (tau*/tau1) theta I.
template <typename Real, typename V>
__device__ __forceinline__ void mix_coeffs(const Mom<V>& m, const StepConst<Real>& K, Herm<V>& H) {
  const V iso = fmad(K.w_eq, m.dth, K.w_es * m.dT);
  const V bs = (K.w_es * K.b) * m.inv_rho;
  V Dl[6] = {fmad(bs, m.sig[0], iso), fmad(bs, m.sig[1], iso), fmad(bs, m.sig[2], iso),
             bs * m.sig[3], bs * m.sig[4], bs * m.sig[5]};
  hermite(m.drho, m.rho, m.inv_rho, m.j, Dl, K.theta0, H);
}

// recover, mix_coeffs and the factor c_relax in one: from the raw moments and the
// stored rotational value, the f-level temperatures in m and the coefficients of
// c_relax (f^mix/w - 1) in H. The products j_a u_b serve the temperature, the
// stress and both orders of the expansion, and products of constants come from
// the launch (about 130 operations instead of 240). FP64 lattices and the batched
// tubes use it; FP32 and 16-bit lattices keep their bits (see kShells).
template <typename Real, bool kPaper, typename V>
__device__ __forceinline__ void relaxed_target(Mom<V>& m, V e, const StepConst<Real>& K, Herm<V>& H) {
  using S = scalar_t<V>;
  constexpr S t0 = S(kTheta0);
  const V jx = m.j[0], jy = m.j[1], jz = m.j[2], ir = m.inv_rho, rho = m.rho;
  const V ux = jx * ir, uy = jy * ir, uz = jz * ir;
  const V xx = jx * ux, yy = jy * uy, zz = jz * uz, xy = jx * uy, xz = jx * uz, yz = jy * uz;
  m.dTg = fmad(S(-3) * t0, m.drho, (m.dP[0] + m.dP[1] + m.dP[2]) - (xx + yy + zz)) * (ir * S(1.0 / 3.0));
  if constexpr (kPaper) {
    m.dR = e;
    m.dT = fmad(K.pa, m.dR, m.dTg) * K.inv_1pa;
    m.dth = fmad(K.c_d, m.dR, K.c_3 * m.dT);
  } else {
    const V dRt = fmad(K.two_id, e, -t0 * m.drho) * ir;
    m.dth = fmad(K.c_d, dRt, K.c_3 * m.dTg);
    const V D = (m.dTg - dRt) * K.inv_d;
    m.dT = fmad(K.c_d, D, m.dth);
    m.dR = fmad(-K.c_3, D, m.dth);
  }
  // Lambda_mix - theta0 I
  const V iso = fmad(t0, m.drho, rho * m.dTg);
  const V mix = fmad(K.w_eq, m.dth, K.w_es * m.dT), bs = K.bsig * ir;
  const V dxx = fmad(bs, m.dP[0] - xx - iso, mix), dyy = fmad(bs, m.dP[1] - yy - iso, mix),
          dzz = fmad(bs, m.dP[2] - zz - iso, mix);
  const V dxy = bs * (m.dP[3] - xy), dxz = bs * (m.dP[4] - xz), dyz = bs * (m.dP[5] - yz);
  const V axx = fmad(rho, dxx, xx), ayy = fmad(rho, dyy, yy), azz = fmad(rho, dzz, zz);
  H.e0 = fmad(-K.q1h, axx + ayy + azz, K.c_relax * m.drho);
  H.exx = K.q2h * axx;
  H.eyy = K.q2h * ayy;
  H.ezz = K.q2h * azz;
  H.exy = K.q2 * fmad(rho, dxy, xy);
  H.exz = K.q2 * fmad(rho, dxz, xz);
  H.eyz = K.q2 * fmad(rho, dyz, yz);
  const V bxy = S(2) * dxy, bxz = S(2) * dxz, byz = S(2) * dyz;
  const V a3xxx = fmad(S(3) * dxx, jx, xx * ux), a3yyy = fmad(S(3) * dyy, jy, yy * uy),
          a3zzz = fmad(S(3) * dzz, jz, zz * uz);
  const V a3xxy = fmad(dxx, jy, fmad(bxy, jx, xx * uy)), a3xxz = fmad(dxx, jz, fmad(bxz, jx, xx * uz));
  const V a3yyx = fmad(dyy, jx, fmad(bxy, jy, yy * ux)), a3yyz = fmad(dyy, jz, fmad(byz, jy, yy * uz));
  const V a3zzx = fmad(dzz, jx, fmad(bxz, jz, zz * ux)), a3zzy = fmad(dzz, jy, fmad(byz, jz, zz * uy));
  const V a3xyz = fmad(dxy, jz, fmad(dyz, jx, fmad(dxz, jy, xy * uz)));
  H.ox = fmad(-K.q2h, a3xxx + a3yyx + a3zzx, K.q1 * jx);
  H.oy = fmad(-K.q2h, a3xxy + a3yyy + a3zzy, K.q1 * jy);
  H.oz = fmad(-K.q2h, a3xxz + a3yyz + a3zzz, K.q1 * jz);
  H.oxxx = K.q36 * a3xxx;
  H.oyyy = K.q36 * a3yyy;
  H.ozzz = K.q36 * a3zzz;
  H.oxxy = K.q32 * a3xxy;
  H.oxxz = K.q32 * a3xxz;
  H.oyyx = K.q32 * a3yyx;
  H.oyyz = K.q32 * a3yyz;
  H.ozzx = K.q32 * a3zzx;
  H.ozzy = K.q32 * a3zzy;
  H.oxyz = K.q3 * a3xyz;
}

// ---------------------------------------------------------------------------
// geometry helpers

__device__ __forceinline__ int wrap_near(int a, int n) {
  // valid for |a - [0, n)| <= 2; n == 1 maps everything to 0
  return n == 1 ? 0 : (a < 0 ? a + n : (a >= n ? a - n : a));
}

struct PointIdx {
  int s, x, y, z;
  int64_t cell;  // (z*ny + y)*nx + x
};

// Point of a thread: consecutive threads take consecutive cells of sublattice
// blockIdx.y, across the ends of rows, so every thread of every block but the
// last has a point whatever nx is (n3 < 2^31: the populations of more cells
// would not fit any device).
template <typename Real>
__device__ __forceinline__ bool point_from_block(const StepConst<Real>& K, PointIdx& P) {
  const unsigned c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= (unsigned)K.n3) return false;
  const unsigned row = K.by_nx.div(c), z = K.by_ny.div(row);
  P.s = blockIdx.y;
  P.x = (int)(c - row * K.nx);
  P.y = (int)(row - z * K.ny);
  P.z = (int)z;
  P.cell = c;
  return true;
}

// As point_from_block for pairs of x-adjacent points (nx even): pair c of the sublattice
// is column i of row (y, z).
__device__ __forceinline__ bool pair_from_block(const StepConst<float>& K, int& s, int& i, int& y, int& z,
                                                int64_t& cellp) {
  const unsigned c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= (unsigned)(K.n3 >> 1)) return false;
  const unsigned row = K.by_nxp.div(c), zz = K.by_ny.div(row);
  s = blockIdx.y;
  i = (int)(c - row * (unsigned)(K.nx >> 1));
  y = (int)(row - zz * K.ny);
  z = (int)zz;
  cellp = c;
  return true;
}

// Gather the 41 populations of point P: from its own slots (kPull = false) or
// pulled from x - c_q (kPull = true; Sec. 5, BCC layout: a half velocity
// from sublattice 0 at index x comes from sublattice 1 at x - (c > 0 ? 1 : 0)
// per axis, and from sublattice 1 it comes from sublattice 0 at
// x + (c < 0 ? 1 : 0)). kBC = 1: sources beyond the x ends read the reservoir.
// kBC & kWallY: sources beyond a y wall (y = -1/4, y = ny - 1/4) are emitted by
// the wall, g = rho_w f^eq(1, u_w, theta_w), i.e. h = d + hw + d hw with
// d = rho_w - 1 of the point's (x, z) column (wcol[(wall * nz + z) * nx + x])
// and hw the wall's table entry. kBC & kWallX: the same for the x walls
// (x = -1/4, x = nx - 1/4) with the (y, z) columns at
// wcol[2 nx nz + (wall * nz + z) * ny + y]; a source beyond both a y and an x
// wall belongs to the y wall. Only the pairs kLo .. kHi - 1 (and the rest
// population with pair 0) are gathered.
template <typename Store, typename Real, bool kPull, int kBC, int kLo = 0, int kHi = kPairs>
__device__ __forceinline__ void gather(const Store* pin,
                                       const Real* __restrict__ ghost, const StepConst<Real>& K,
                                       const PointIdx& P, Real (&h)[kQ],
                                       const Real* wcol = nullptr) {
  const int64_t n3 = K.n3;
  if constexpr (!kPull) {
    const unsigned cell = (unsigned)P.cell;
#pragma unroll
    for (int q = kLo ? 2 * kLo + 1 : 0; q < 2 * kHi + 1; ++q)
      h[q] = to_real<Store, Real>((pin + (int64_t)(P.s * kQ + q) * n3)[cell]);
  } else {
    const int nx = K.nx, ny = K.ny, nz = K.nz;
    int xw[5], yw[5], zw[5];
    bool xin[5], yin[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      xw[k] = wrap_near(P.x + k - 2, nx);
      // cell offsets of the row and the plane: 32 bits (a sublattice holds fewer
      // than 2^31 cells), added to a base that is the same for the whole block
      yw[k] = wrap_near(P.y + k - 2, ny) * nx;
      zw[k] = wrap_near(P.z + k - 2, nz) * (ny * nx);
      xin[k] = (P.x + k - 2 >= 0) && (P.x + k - 2 < nx);
      yin[k] = (P.y + k - 2 >= 0) && (P.y + k - 2 < ny);
    }
    // half-velocity source offsets: c > 0 -> s - 1, c < 0 -> s
    const int s = P.s;
    const int xhp = s ? xw[2] : xw[1], xhm = s ? xw[3] : xw[2];
    const int yhp = s ? yw[2] : yw[1], yhm = s ? yw[3] : yw[2];
    const int zhp = s ? zw[2] : zw[1], zhm = s ? zw[3] : zw[2];
    const bool xinhp = s ? xin[2] : xin[1], xinhm = s ? xin[3] : xin[2];
    const bool yinhp = s ? yin[2] : yin[1], yinhm = s ? yin[3] : yin[2];
    const Store* same = pin + (int64_t)(s * kQ) * n3;
    const Store* other = pin + (int64_t)((1 - s) * kQ) * n3;
    if constexpr (kLo == 0) h[0] = to_real<Store, Real>(same[(unsigned)P.cell]);
    static_for<2 * (kHi - kLo)>([&](auto qc) {
      constexpr int q = decltype(qc)::value + 2 * kLo + 1;
      constexpr Vel2 v = vel2(q);
      constexpr bool half = (v.x & 1) != 0;
      int xs, ys, zs;
      [[maybe_unused]] bool insx = true, insy = true;
      const Store* base;
      if constexpr (half) {
        xs = v.x > 0 ? xhp : xhm;
        ys = v.y > 0 ? yhp : yhm;
        zs = v.z > 0 ? zhp : zhm;
        insx = v.x > 0 ? xinhp : xinhm;
        insy = v.y > 0 ? yinhp : yinhm;
        base = other;
      } else {
        xs = xw[2 - v.x / 2];
        ys = yw[2 - v.y / 2];
        zs = zw[2 - v.z / 2];
        insx = xin[2 - v.x / 2];
        insy = yin[2 - v.y / 2];
        base = same;
      }
      const unsigned cell = (unsigned)(zs + ys + xs);
      if constexpr (kBC == 1) {
        if (!insx) {
          h[q] = ghost[(v.x > 0 ? 0 : kGhostStride) + q];
          return;
        }
      }
      if constexpr ((kBC & kWallY) && v.y != 0) {
        if (!insy) {
          const int w = v.y > 0 ? 0 : 1;  // source below the low wall / above the high wall
          const Real d = wcol[((int64_t)w * nz + P.z) * nx + P.x];
          const Real hw = ghost[w * kGhostStride + q];
          h[q] = d + hw + d * hw;
          return;
        }
      }
      if constexpr ((kBC & kWallX) && v.x != 0) {
        if (!insx) {
          const int w = v.x > 0 ? 0 : 1;
          const Real d = wcol[2 * (int64_t)nx * nz + ((int64_t)w * nz + P.z) * ny + P.y];
          const Real hw = ghost[(2 + w) * kGhostStride + q];
          h[q] = d + hw + d * hw;
          return;
        }
      }
      h[q] = to_real<Store, Real>((base + (int64_t)q * n3)[cell]);
    });
  }
}

// rho_w - 1 of every wall column, from the post-collision populations pin that
// the next pull reads. For a wall and one of its columns: the column's
// populations whose destination lies beyond the wall carry the mass
// M_out = sum w (1 + h); the wall emits rho_w f^eq(1, u_w, theta_w) into the
// column's entries whose source lies beyond it, mass rho_w D with
// D = sum w (1 + hw). rho_w - 1 = (M_out - D) / D, accumulated as
// (sum_out w - sum_in w) + sum_out w h - sum_in w hw so that the deviation keeps
// its precision (the weights of c and -c are equal). A velocity with |2 c_a| = n
// along the wall normal a has its n layers next to the wall in play. Where
// both kinds of walls are on, a population crossing a y wall belongs to it
// even if it crosses an x wall too, so the x walls count only entries whose
// other end stays inside in y.
// The sums of one column of the wall at side w; kX: an x wall (else a y wall).
// Of a velocity pair that crosses the wall one member leaves and the other is
// emitted, so the loads are unconditional and all 44 of a column are in flight
// at once (the axis is a template argument: every trip count is known). 128 x 64
// x 8 between y walls: 12.6 us with one load after the other, now 4.6 us.
template <typename Store, typename Real, int kBC, bool kX>
__device__ __forceinline__ Real wall_column(const StepConst<Real>& K, const Store* pin,
                                            const Real* __restrict__ hw, int w, int ca, int z) {
  const int nx = K.nx, ny = K.ny, nn = kX ? nx : ny;  // cells along the wall normal
  const int64_t n3 = K.n3;
  Real base = Real(0), A = Real(0), D = Real(0), S = Real(0);
  static_for<kPairs>([&](auto kc) {
    constexpr int k = decltype(kc)::value;
    constexpr Vel2 v = kPairVel2[k];
    constexpr int vn = kX ? v.x : v.y;  // doubled velocity along the normal
    constexpr int vt = kX ? v.y : 0;    // along y, for the corner rule of the x walls
    constexpr int n = vn > 0 ? vn : -vn;
    if constexpr (n > 0) {
      const Real wq = Real(pair_weight(k));
      const bool first_out = (w == 1) == (vn > 0);  // the pair's first member leaves
      const int out = first_out ? 2 * k + 1 : 2 * k + 2, in = first_out ? 2 * k + 2 : 2 * k + 1;
      const Real hin = hw[in];
      bool mine[n];
#pragma unroll
      for (int l = 0; l < n; ++l) {
        const int L2 = w == 0 ? l : 2 * nn - 1 - l;  // 2 * index + s along the normal
        const int s = L2 & 1, i = L2 >> 1;
        const int x = kX ? i : ca, y = kX ? ca : i;
        const Real h = to_real<Store, Real>(pin[(int64_t)(s * kQ + out) * n3 + ((int64_t)z * ny + y) * nx + x]);
        mine[l] = true;
        if ((kBC & kWallY) && kX) {
          // the other end of the trajectory must stay inside in y
          const int Y2 = 2 * ca + s + (first_out ? vt : -vt);
          mine[l] = Y2 >= 0 && Y2 < 2 * ny;
        }
        if (mine[l]) {
          S += wq * h;
          D += wq * (Real(1) + hin);
          A -= wq * hin;
        }
      }
      const Real d = first_out ? wq : -wq;
#pragma unroll
      for (int l = 0; l < n; ++l)
        if (mine[l]) base += d;
#pragma unroll
      for (int l = 0; l < n; ++l)
        if (mine[l]) base -= d;
    }
  });
  return (base + A + S) / D;
}

// One thread per (wall, column): y walls first (slots [0, 2 nx nz), columns
// (x, z)), then x walls (slots 2 nx nz + [0, 2 ny nz), columns (y, z)).
template <typename Store, typename Real, int kBC>
__global__ void __launch_bounds__(128)
    k_wall_rho(StepConst<Real> K, const Store* pin, const Real* __restrict__ ghost,
               Real* __restrict__ wcol) {
  pdl_wait();
  const int64_t ny_cols = (int64_t)K.nx * K.nz, nx_cols = (int64_t)K.ny * K.nz;
  const int64_t ybase = (kBC & kWallY) ? 2 * ny_cols : 0;
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= ybase + ((kBC & kWallX) ? 2 * nx_cols : 0)) return;
  // columns of a wall fit 32 bits: they are fewer than the cells
  if (t >= ybase) {
    if constexpr ((kBC & kWallX) != 0) {
      t -= ybase;
      const int w = t >= nx_cols ? 1 : 0;
      const int64_t c = t - w * nx_cols;
      wcol[2 * ny_cols + t] = wall_column<Store, Real, kBC, true>(K, pin, ghost + (2 + w) * kGhostStride, w,
                                                                  (int)((unsigned)c % (unsigned)K.ny), (int)((unsigned)c / (unsigned)K.ny));
    }
  } else {
    if constexpr ((kBC & kWallY) != 0) {
      const int w = t >= ny_cols ? 1 : 0;
      const int64_t c = t - w * ny_cols;
      wcol[t] = wall_column<Store, Real, kBC, false>(K, pin, ghost + w * kGhostStride, w,
                                                     (int)((unsigned)c % (unsigned)K.nx),
                                                     (int)((unsigned)c / (unsigned)K.nx));
    }
  }
}

}  // namespace rpk
