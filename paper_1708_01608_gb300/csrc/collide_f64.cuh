// The FP64 collision of one cell, counted in FP64 instructions.
//
// GB300 issues two FP64 lanes per SM and cycle (1.25 TFLOP/s over 152 SMs),
// so an FP64 step is bound by that pipe long before HBM: at 128^3 the 304
// bytes of an update take 94 us per step at the copy bandwidth, the 549 FP64
// instructions of the former velocity-by-velocity form took 2.285 ms.  This
// form spends 174 (92 DADD, 14 DMUL, 67 DFMA, halo included): 0.781 ms, the
// pipe 79 % busy (ncu); D2Q9 at 1024^2 went from 0.599 to 0.201 ms.  (Without
// the mass terms of relax_pairs and the table's error in psi_f64, 169, 0.752 and
// 0.189 ms, but twice the former error.)  With w the edge weight (1/36), m = rho u
// and one value each per axis a
//   B_a = 3 omega w m_a,  v_a = 1.5 u_a,  Q_a = B_a v_a,
//   K = omega w rho - (Q_x + Q_y + Q_z)/3,
// omega f_eq of the rest, an axis and an edge velocity is
//   R0 K,  R (K + Q_a) +- R B_a,
//   K + Q_a + Q_b + c_a c_b B_a (2 v_b) +- (c_a B_a + c_b B_b)
// (R and R0 the weights' ratios 2 and 12, D2Q9 4 and 16), so opposite
// velocities share the even part, the four edges of a plane share
// K + Q_a + Q_b, relaxation is one FMA on (1 - omega) f_i, and the only
// division left is one reciprocal of rho.  Zero velocity components cost
// nothing (a product with 0.0 is not removable under IEEE rules) and the
// density is the psi phase's sum.
#pragma once

#include "internal.h"
#include "lattice.cuh"

namespace sclbm {

// {T, e}: T = 2^(k/64) rounded to nearest, k = 0 .. 63, and e = 2^(k/64)/T - 1
// rounded, what the rounding took
static __device__ const double2 EXP2_64TH[64] = {
    {0x1.0000000000000p+0, 0.0}, {0x1.02c9a3e778061p+0, -0x1.160139cd8dc5dp-56},
    {0x1.059b0d3158574p+0, 0x1.cd2523567f613p-55}, {0x1.0874518759bc8p+0, 0x1.0f74e61e6c861p-57},
    {0x1.0b5586cf9890fp+0, 0x1.79aa65d837b6cp-54}, {0x1.0e3ec32d3d1a2p+0, 0x1.ebe3d702f9cd1p-60},
    {0x1.11301d0125b51p+0, -0x1.556522a2fbd0ep-54}, {0x1.1429aaea92de0p+0, -0x1.1c923b9d5f416p-54},
    {0x1.172b83c7d517bp+0, -0x1.01b15eaa59348p-55}, {0x1.1a35beb6fcb75p+0, 0x1.b898c3f1353bfp-55},
    {0x1.1d4873168b9aap+0, 0x1.aecf73e3a2f5fp-54}, {0x1.2063b88628cd6p+0, 0x1.a6f4144a6c38cp-55},
    {0x1.2387a6e756238p+0, 0x1.68efde3a8a893p-54}, {0x1.26b4565e27cddp+0, 0x1.0472b981fe7f2p-55},
    {0x1.29e9df51fdee1p+0, 0x1.2f7e16d09ab31p-55}, {0x1.2d285a6e4030bp+0, 0x1.b3782720c0ab3p-55},
    {0x1.306fe0a31b715p+0, 0x1.34d754db0abb6p-55}, {0x1.33c08b26416ffp+0, 0x1.fdd395dd3f84ap-55},
    {0x1.371a7373aa9cbp+0, -0x1.24aedcc4b5069p-54}, {0x1.3a7db34e59ff7p+0, -0x1.1d1e83e9436d2p-56},
    {0x1.3dea64c123422p+0, 0x1.59f48a72a4c6cp-55}, {0x1.4160a21f72e2ap+0, -0x1.8a78f4817895bp-58},
    {0x1.44e086061892dp+0, 0x1.363ed60c2ac11p-59}, {0x1.486a2b5c13cd0p+0, 0x1.ecce1daa10379p-57},
    {0x1.4bfdad5362a27p+0, 0x1.690cebb7aafb0p-56}, {0x1.4f9b2769d2ca7p+0, -0x1.f94340071a38fp-55},
    {0x1.5342b569d4f82p+0, -0x1.8dec6bd0f3860p-56}, {0x1.56f4736b527dap+0, 0x1.3350518fdd78dp-54},
    {0x1.5ab07dd485429p+0, 0x1.063e1e21c5409p-54}, {0x1.5e76f15ad2148p+0, 0x1.432e62b64c035p-54},
    {0x1.6247eb03a5585p+0, -0x1.c33c53bef4da8p-55}, {0x1.6623882552225p+0, -0x1.3cedd78565858p-54},
    {0x1.6a09e667f3bcdp+0, -0x1.3b3efbf5e2229p-54}, {0x1.6dfb23c651a2fp+0, -0x1.367efb86da9eep-57},
    {0x1.71f75e8ec5f74p+0, -0x1.81f647e5a3ecfp-56}, {0x1.75feb564267c9p+0, -0x1.619321e55e68ap-55},
    {0x1.7a11473eb0187p+0, -0x1.b32dcb94da51dp-56}, {0x1.7e2f336cf4e62p+0, 0x1.5ebe1abd66c55p-57},
    {0x1.82589994cce13p+0, -0x1.369b6f13b3734p-54}, {0x1.868d99b4492edp+0, -0x1.4d450d872576ep-54},
    {0x1.8ace5422aa0dbp+0, 0x1.db72fc1f0eab4p-55}, {0x1.8f1ae99157736p+0, 0x1.bf68359f35f44p-56},
    {0x1.93737b0cdc5e5p+0, -0x1.da9b88b6c1e29p-58}, {0x1.97d829fde4e50p+0, -0x1.2434322f4f9aap-54},
    {0x1.9c49182a3f090p+0, 0x1.1affc2b91ce27p-56}, {0x1.a0c667b5de565p+0, -0x1.7c50422622263p-55},
    {0x1.a5503b23e255dp+0, -0x1.1bbd1d3bcbb15p-54}, {0x1.a9e6b5579fdbfp+0, 0x1.469846e735ab3p-55},
    {0x1.ae89f995ad3adp+0, 0x1.c1a7792cb3386p-55}, {0x1.b33a2b84f15fbp+0, -0x1.5c3d956dcaebap-58},
    {0x1.b7f76f2fb5e47p+0, -0x1.8d6f438ad9334p-57}, {0x1.bcc1e904bc1d2p+0, 0x1.4ffd70a5fddcdp-56},
    {0x1.c199bdd85529cp+0, 0x1.36eae30af0cb3p-56}, {0x1.c67f12e57d14bp+0, 0x1.4e08fd10959acp-55},
    {0x1.cb720dcef9069p+0, 0x1.76b2c6c921968p-57}, {0x1.d072d4a07897cp+0, -0x1.fad5d3ffffa6fp-55},
    {0x1.d5818dcfba487p+0, 0x1.4a385a63d07a7p-56}, {0x1.da9e603db3285p+0, 0x1.e5a50d5c192acp-55},
    {0x1.dfc97337b9b5fp+0, -0x1.2d52107b43e1fp-55}, {0x1.e502ee78b3ff6p+0, 0x1.4b604603a88d3p-56},
    {0x1.ea4afa2a490dap+0, -0x1.ff7128fd391f1p-55}, {0x1.efa1bee615a27p+0, 0x1.ec3bc41aa2008p-55},
    {0x1.f50765b6e4540p+0, 0x1.a64a931d185edp-55}, {0x1.fa7c1819e90d8p+0, 0x1.7893b4d91cd9cp-56}};

// psi(rho) = rho0 (1 - exp(-rho/rho0)) with the table-driven exponential of
// Tang (ACM TOMS 15, 1989): x = n ln2/64 + r with |r| <= ln2/128, e^x =
// 2^(n/64) (1 + r + r^2/2 + ... + r^5/120), the tail below 4e-17.  13 FP64
// instructions against about 20 with exp().  One of them adds the table entry's
// own error to r, which gives psi back the error that it has with exp(): of rho0,
// in units of 2^-53, rms and largest 0.31 and 0.89 (rho0 = 1; exp() 0.32 and
// 0.90, without e 0.34 and 1.24) and 0.38 and 1.27 (others; exp() 0.49 and
// 1.66).  The range test is on integers; outside it (and for NaN) exp()
// decides.
__device__ __forceinline__ double psi_f64(double rho, double rho0, double inv_rho0) {
  const double x = -rho * inv_rho0;
  if ((__double2hiint(x) & 0x7fffffff) >= 0x4085e000) return rho0 * (1.0 - exp(x));  // |x| >= 700
  const double t = fma(x, 0x1.71547652b82fep+6, 0x1.8p52);  // n in the low word
  const int n = __double2loint(t);
  const double nd = t - 0x1.8p52;
  const double2 T = __ldg(EXP2_64TH + (n & 63));
  const double r = fma(nd, -0x1.473de6af278edp-40, fma(nd, -0x1.62e42fefp-7, x));
  double q = fma(r, 1.0 / 120.0, 1.0 / 24.0);
  q = fma(q, r, 1.0 / 6.0);
  q = fma(q, r, 0.5);
  q = fma(q * r, r, r + T.y);  // e^r - 1, and T's error
  const double S = __hiloint2double(__double2hiint(T.x) + ((n >> 6) << 20), __double2loint(T.x));
  return fma(-rho0, fma(S, q, S), rho0);
}

// Whether the reciprocal of b may be infinite: |b| below the normal numbers
__device__ __forceinline__ bool rcp_overflows(double b) {
  return (__double2hiint(b) & 0x7fffffff) < 0x00100000;
}
__device__ __forceinline__ bool rcp_overflows(float b) {
  return fabsf(b) < 0x1p-126f;
}

// Density of one cell from its Q values, in two chains (half the latency of
// one; the owner and a neighbour's halo thread use the same order)
template <int Q, class Ld>
__device__ __forceinline__ auto rho_f64(Ld ld) {
  auto a = ld(0), b = ld(1);
#pragma unroll
  for (int i = 2; i + 1 < Q; i += 2) {
    a += ld(i);
    b += ld(i + 1);
  }
  if constexpr (Q % 2 == 1) a += ld(Q - 1);
  return a + b;
}

// Relaxation constants; w is the edge weight 1/36.
template <int LAT, class T>
struct RelaxK {
  static constexpr T R = LAT == D3Q19 ? 2 : 4;     // axis weight / edge weight
  static constexpr T R0 = LAT == D3Q19 ? 12 : 16;  // rest weight / edge weight
  T om1, wK, cB, eps;
  __device__ __forceinline__ RelaxK(T om1_, T wK_, T cB_, T eps_)
      : om1(om1_), wK(wK_), cB(cB_), eps(eps_) {}
};

template <int CC, class T>
__device__ __forceinline__ T cacc_t(T acc, T v) {
  if constexpr (CC > 0) return acc + v;
  else if constexpr (CC < 0) return acc - v;
  else return acc;
}

// sum_i w_i q(i) c_i / w over opposite pairs, q(i) given as the difference
// dq(i) = q(i) - q(opp i) of a representative
template <int LAT, bool WEIGHTED, class T, class Dq>
__device__ __forceinline__ void pair_moments(Dq dq, T (&m)[3]) {
  using L = Lattice<LAT>;
  // -0 is the additive identity, so a first term is no addition
  T ax[3] = {0, 0, 0}, ed[3] = {(T)-0.0, (T)-0.0, (T)-0.0};
  static_for<L::NP>([&](auto kc) {
    constexpr int i = L::rep(decltype(kc)::value);
    constexpr int cx = L::cx(i), cy = L::cy(i), cz = L::cz(i);
    const T d = dq(std::integral_constant<int, i>{});
    if constexpr (WEIGHTED && cx * cx + cy * cy + cz * cz == 1) {
      static_assert(cx + cy + cz == 1, "axis representatives point along +a");
      ax[cx ? 0 : (cy ? 1 : 2)] = d;
    } else {
      ed[0] = cacc_t<cx>(ed[0], d);
      ed[1] = cacc_t<cy>(ed[1], d);
      ed[2] = cacc_t<cz>(ed[2], d);
    }
  });
#pragma unroll
  for (int a = 0; a < 3; ++a)
    m[a] = WEIGHTED && (a != 1 || L::HAS_Y) ? fma(RelaxK<LAT, T>::R, ax[a], ed[a]) : ed[a];
}

// The relaxed populations of a cell: f(i) its populations, rho their sum,
// v = 1.5 u, B = 3 omega w rho u; out(integral_constant i, value).
//
// Mass.  The populations together carry om1 + 36 wK of rho, the same wrong
// factor in every cell and step by the rounding of the two constants, and 36
// times the rounding of K.  FP64 adds both to the rest population inside its
// FMA (added after it they would be rounded off): 4 of a cell's 174 FP64
// instructions.  Total mass after 300 steps against velocity by velocity, rms
// over 320 runs (D3Q19 and D2Q9, tau 0.6 to 1.4, with and without a bubble):
// without 1.5e-14, with eps alone 5.0e-15, with both 1.5e-15.  FP32 gives the
// rest population rho minus the moving ones, as the FP32 step kernels do: of
// the largest population after 400 steps, velocity by velocity 1.9e-6, from K
// 1.1e-5, this 7e-8 (two lattices, D2Q9, tau 0.6).
template <int LAT, class T, class F, class Out>
__device__ __forceinline__ void relax_pairs(const RelaxK<LAT, T> &q, F f, T rho, const T (&v)[3],
                                            const T (&B)[3], Out out) {
  using L = Lattice<LAT>;
  constexpr T R = RelaxK<LAT, T>::R, R0 = RelaxK<LAT, T>::R0;
  T Q[3], s = (T)-0.0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (a == 1 && !L::HAS_Y) continue;
    Q[a] = B[a] * v[a];
    s += Q[a];
  }
  const T ts = s * (T)(-1.0 / 3.0), K = fma(q.wK, rho, ts);
  constexpr bool REST = sizeof(T) == 4;
  T moved[2] = {(T)-0.0, (T)-0.0};  // in two chains: one of 18 additions is latency
  if constexpr (!REST)
    out(std::integral_constant<int, 0>{},
        fma(q.om1, f(0), fma(R0, K, fma((T)36, fma(q.wK, rho, ts - K), q.eps * rho))));
  auto put = [&](auto ic, T x, int chain) {
    if constexpr (REST) moved[chain] += x;
    out(ic, x);
  };
  static_for<L::NP>([&](auto kc) {
    constexpr int i = L::rep(decltype(kc)::value), o = L::opp(i);
    constexpr int cx = L::cx(i), cy = L::cy(i), cz = L::cz(i);
    constexpr int c[3] = {cx, cy, cz};
    constexpr int a = cx ? 0 : (cy ? 1 : 2);
    if constexpr (cx * cx + cy * cy + cz * cz == 1) {
      const T A = R * (K + Q[a]);
      put(std::integral_constant<int, i>{}, fma(R, B[a], fma(q.om1, f(i), A)), 0);
      put(std::integral_constant<int, o>{}, fma(-R, B[a], fma(q.om1, f(o), A)), 1);
    } else {
      constexpr int b = cz ? 2 : 1;
      const T D = (K + Q[a]) + Q[b], v2 = v[b] + v[b];
      const T A = c[a] * c[b] > 0 ? fma(B[a], v2, D) : fma(-B[a], v2, D);
      // c_a B_a + c_b B_b up to the sign of c_a
      const T t = c[a] * c[b] > 0 ? B[a] + B[b] : B[a] - B[b];
      const T hi = fma(q.om1, f(i), A), ho = fma(q.om1, f(o), A);
      put(std::integral_constant<int, i>{}, c[a] > 0 ? hi + t : hi - t, 0);
      put(std::integral_constant<int, o>{}, c[a] > 0 ? ho - t : ho + t, 1);
    }
  });
  if constexpr (REST) out(std::integral_constant<int, 0>{}, rho - (moved[0] + moved[1]));
}

// The FP64 collision of one cell.  f(i): its populations, rho their sum,
// psi0 and psi(i) the pseudopotential here and at x + c_i, fG = -tau G w;
// put(i, v) takes the collided population (integral_constant i).  SITE adds
// w_i dm to every population.
template <int LAT, bool SITE, class F, class Psi, class Put>
__device__ __forceinline__ void collide_f64(const RelaxK<LAT, double> &q, double fG, F f,
                                            double rho, double psi0, Psi psi, Put put, double dm) {
  using L = Lattice<LAT>;
  double j[3], s[3];
  pair_moments<LAT, false, double>(
      [&](auto ic) { return f(decltype(ic)::value) - f(L::opp(decltype(ic)::value)); }, j);
  pair_moments<LAT, true, double>(
      [&](auto ic) { return psi(decltype(ic)::value) - psi(L::opp(decltype(ic)::value)); }, s);
  const double gp = fG * psi0, ir = 1.5 * __drcp_rn(rho);
  double v[3], B[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (a == 1 && !L::HAS_Y) continue;
    const double m = fma(gp, s[a], j[a]);
    v[a] = rcp_overflows(rho) ? 1.5 * (m / rho) : m * ir;
    B[a] = q.cB * m;
  }
  relax_pairs<LAT, double>(q, f, rho, v, B, [&](auto ic, double x) {
    put(ic, SITE ? x + L::w(decltype(ic)::value) * dm : x);
  });
}

}  // namespace sclbm
