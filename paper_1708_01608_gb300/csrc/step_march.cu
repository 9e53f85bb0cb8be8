// One-launch step on plain loads, for lattices the TMA march cannot take:
// rows that are no multiple of 16 bytes (any nx of a context, any buffer of
// the allocation-free step).  Push form, as everywhere: stored_i(x) =
// f_i(x, t).
//
// What bounds it: the two kernels of the two-pass step (psi field, then
// collision) move 3 Q S + 2 sizeof(psi) bytes per update.  Here a CTA owns a
// column of the lattice and marches along z as the TMA march does, so that a
// population leaves HBM once per step: 2 Q S bytes.
//
// The thread block covers the column with its one-cell halo ring (TX x TY
// threads, (TX - 2) x (TY - 2) cells): every thread sums one cell per plane
// into a four-plane psi ring in shared memory, the inner ones collide the
// plane before it.  Rings cost loads (L2 hits) in place of a divergent halo
// pass.  The next plane's populations are in flight, in registers, over the
// barrier and the collision; the colliding plane's wait in shared memory, each
// thread in its own slots (read a second time instead they came from L2, 2 %
// of them from L1: 49.0 us at 127x101x90 against 43.5; in a third set of
// registers, with two CTAs per SM, 44.0).  FP64, which the pipe bounds, reads
// them twice.
//
// FP32 arithmetic repeats the two-pass kernels rounding for rounding and
// gives their bits (the state after a step, and so every label and census
// that depends on it, is that of the two-pass step).  FP64 takes the
// collision of collide_f64.cuh.
//
// us per step, two-pass / this: 201x150x99 FP32 168 / 121, FP16 164 / 97;
// 33x35x31 FP32 10.3 / 4.9; 93^3 FP64 772 / 461; D2Q9 201^2 FP32 10.3 / 3.0,
// 1401x1203 68 / 25, 129^2 FP64 27 / 11.5; the allocation-free step at
// 127x101x90 54 / 43.5.  Blocks of 32 x 8 threads, three per SM, against 32 x
// 12, two per SM (124 and 105 at 201x150x99) and 32 x 24 (144 and 118);
// without the plane in flight 129 and 112.
#include <algorithm>
#include <cmath>

#include "collide_f64.cuh"
#include "internal.h"
#include "lattice.cuh"

namespace sclbm {

namespace {

// acc + c v, rounded and never contracted, for c in {-1, 0, 1}
template <int CC>
__device__ __forceinline__ float cacc_rn(float acc, float v) {
  if constexpr (CC > 0) return __fadd_rn(acc, v);
  else if constexpr (CC < 0) return __fsub_rn(acc, v);
  else return acc;
}

// The FP32 collision of one cell on its offsets g (R their sum): every
// rounding written out, as the two-pass kernels have it; the relaxation of
// opposite velocities runs as paired instructions.
template <int LAT, int ST, class Psi, class Dst>
__device__ __forceinline__ void collide_rn(float (&g)[Lattice<LAT>::Q], float R, float rho_ref,
                                           float tau, float omega, float G, Psi psi_at, Dst dst) {
  using L = Lattice<LAT>;
  using S = Storage<ST>;
  constexpr int Q = L::Q;
  float sx = 0, sy = 0, sz = 0, jx = 0, jy = 0, jz = 0;
  static_for<Q>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    if constexpr (i > 0) {
      const float wp = __fmul_rn((float)L::w(i), psi_at(i));
      sx = cacc_rn<L::cx(i)>(sx, wp);
      sy = cacc_rn<L::cy(i)>(sy, wp);
      sz = cacc_rn<L::cz(i)>(sz, wp);
      jx = cacc_rn<L::cx(i)>(jx, g[i]);
      jy = cacc_rn<L::cy(i)>(jy, g[i]);
      jz = cacc_rn<L::cz(i)>(jz, g[i]);
    }
  });
  const float rho = __fadd_rn(rho_ref, R), ir = __fdiv_rn(1.0f, rho);
  const float tg = __fmul_rn(tau, -G * psi_at(0));
  const float ux = __fmul_rn(__fmaf_rn(tg, sx, jx), ir), uy = __fmul_rn(__fmaf_rn(tg, sy, jy), ir),
              uz = __fmul_rn(__fmaf_rn(tg, sz, jz), ir);
  const float uu = __fmaf_rn(uz, uz, __fmaf_rn(ux, ux, __fmul_rn(uy, uy)));
  const float K = __fmaf_rn(-__fmul_rn(1.5f, rho), uu, R);
  static_for<L::NP>([&](auto kc) {
    constexpr int i = L::rep(decltype(kc)::value), o = L::opp(i);
    constexpr float w = (float)L::w(i);
    const float cu = cdot<L::cx(i), L::cy(i), L::cz(i)>(ux, uy, uz);
    const float q = __fmul_rn(__fmul_rn(4.5f, cu), cu);
    const float2 g2 = make_float2(g[i], g[o]);
    const float2 e2 = make_float2(__fmaf_rn(3.0f, cu, q), __fmaf_rn(-3.0f, cu, q));
    const float2 X = __ffma2_rn(make_float2(rho, rho), e2, make_float2(K, K));
    const float2 t = __ffma2_rn(make_float2(-w, -w), X, g2);
    const float2 r = __ffma2_rn(make_float2(-omega, -omega), t, g2);
    g[i] = r.x;
    g[o] = r.y;
  });
  float moved = 0;
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    moved = __fadd_rn(moved, g[i]);
    *dst(i) = S::store(g[i]);
  }
  *dst(0) = S::store(__fsub_rn(R, moved));
}

template <int LAT, int ST, int TX, int TY, int MINB>
__global__ void __launch_bounds__(TX *TY, MINB)
    march_step_kernel(const StepArgs a, const int tiles_x, const int tiles_y, const int zlen) {
  using L = Lattice<LAT>;
  using S = Storage<ST>;
  using T = typename S::T;
  using C = typename S::C;
  constexpr int Q = L::Q, HY = L::HAS_Y ? 1 : 0, BX = TX - 2, BY = TY - 2 * HY;
  constexpr bool F64 = sizeof(C) == 8;
  static_assert(BX > 0 && BY > 0 && (HY || TY == 1), "a cell inside the halo ring");
  static_assert(!S::RESID, "psi reads neighbours' residuals, which the collision rewrites");
  __shared__ C ring[4][TY][TX];
  __shared__ T held[F64 ? 1 : 2][Q][F64 ? 1 : TX * TY];  // planes P and P - 1

  const int NX = (int)a.NX, NY = (int)a.NY, NZ = (int)a.NZ;
  const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;
  const int ntiles = tiles_x * tiles_y;
  const int zc = blockIdx.x / ntiles, tt = blockIdx.x % ntiles;
  const int x0 = (tt % tiles_x) * BX, y0 = (tt / tiles_x) * BY;
  const int BXe = min(BX, NX - x0), BYe = min(BY, NY - y0);
  const int zs = zc * zlen, ze = min(NZ, zs + zlen);
  const int npl = ze - zs + 2;  // planes zs - 1 .. ze
  const bool covers = tx <= BXe + 1 && (!HY || ty <= BYe + 1);
  const bool inner = tx >= 1 && tx <= BXe && (!HY || (ty >= 1 && ty <= BYe));
  // this thread's cell, wrapped, and its neighbours'
  const int xr = x0 - 1 + tx, yr = HY ? y0 - 1 + ty : 0;
  const int x = xr < 0 ? NX - 1 : (xr >= NX ? 0 : xr), y = yr < 0 ? NY - 1 : (yr >= NY ? 0 : yr);
  const int ox[3] = {x == 0 ? NX - 1 : x - 1, x, x + 1 >= NX ? 0 : x + 1};
  const int px = (int)a.px, plane = px * NY;  // padded cells fit 32 bits
  const int oy[3] = {(y == 0 ? NY - 1 : y - 1) * px, y * px, (y + 1 >= NY ? 0 : y + 1) * px};
  const int64_t pop = (int64_t)plane * NZ;
  const T *fin = static_cast<const T *>(a.fin);
  auto wrap_z = [&](int z) { return z < 0 ? z + NZ : (z >= NZ ? z - NZ : z); };

  const C rho0 = F64 ? (C)a.rho0 : (C)a.rho0_f;
  const C inv_rho0 = F64 ? (C)a.relax.inv_rho0 : (C)a.inv_rho0_f;
  const C G = (C)a.G_f, tau = (C)a.tau_f, omega = (C)a.omega_f, rho_ref = (C)a.rho_ref_f;

  // launched as a programmatic dependent: nothing of the lattices is touched
  // before the previous step is complete
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  T next[Q];
  auto load_plane = [&](int P) {
    const T *p = fin + (wrap_z(P) * plane + oy[1] + x);
#pragma unroll
    for (int i = 0; i < Q; ++i) next[i] = p[i * pop];
  };
  C r1 = 0, r2 = 0;  // sums of planes P and P - 1 (without rho_ref)
  if (!F64 && covers) load_plane(zs - 1);
  for (int k = 0; k < npl; ++k) {
    const int P = zs - 1 + k;
    r2 = r1;
    if (covers) {
      if constexpr (F64) {
        // the FP64 pipe bounds this form, not the loads: nothing is held
        load_plane(P);
        r1 = rho_f64<Q>([&](int i) { return next[i]; });
        ring[k & 3][ty][tx] = psi_f64(r1, rho0, inv_rho0);
      } else {
        C r = 0;
#pragma unroll
        for (int i = 0; i < Q; ++i) r += S::load(next[i]);
        r1 = r;
        ring[k & 3][ty][tx] = psi_of(r + rho_ref, rho0, inv_rho0);
#pragma unroll
        for (int i = 0; i < Q; ++i) held[k & 1][i][threadIdx.x] = next[i];
        if (k + 1 < npl) load_plane(P + 1);
      }
    }
    __syncthreads();
    if (k < 2 || !inner) continue;

    // ---- collide plane P - 1 (psi of P - 2, P - 1, P in the ring) and push
    const int Pc = P - 1;
    const int oz[3] = {(Pc == 0 ? NZ - 1 : Pc - 1) * plane, Pc * plane,
                       (Pc + 1 >= NZ ? 0 : Pc + 1) * plane};
    auto psi_at = [&](int i) -> C {
      return ring[(k - 1 + L::cz(i)) & 3][ty + L::cy(i)][tx + L::cx(i)];
    };
    auto dst = [&](int i) -> T * {
      return static_cast<T *>(a.out_pop[i]) +
             (oz[L::cz(i) + 1] + oy[L::cy(i) + 1] + ox[L::cx(i) + 1]);
    };
    if constexpr (F64) {
      const T *own = fin + (oz[1] + oy[1] + x);
      T f[Q];
#pragma unroll
      for (int i = 0; i < Q; ++i) f[i] = own[i * pop];
      const RelaxK<LAT, double> relax(a.relax.om1, a.relax.wK, a.relax.cB, a.relax.eps);
      collide_f64<LAT, false>(
          relax, a.relax.fG, [&](int i) { return f[i]; }, r2, psi_at(0), psi_at,
          [&](auto ic, C v) { *dst(decltype(ic)::value) = v; }, 0.0);
    } else {
      C g[Q];
#pragma unroll
      for (int i = 0; i < Q; ++i) g[i] = S::load(held[(k - 1) & 1][i][threadIdx.x]);
      collide_rn<LAT, ST>(g, r2, rho_ref, tau, omega, G, psi_at, dst);
    }
  }
}

// ---- the box form -----------------------------------------------------------
// Lattices on which most of a march's threads would idle: rows or columns far
// narrower than its tile, or one plane, which it stages three times.  A CTA
// takes a box of cells, forms psi on it and its one-cell halo in shared memory
// (no halo on an axis the box covers: it wraps in place) and collides; the
// populations are read a second time, from L1 or L2.  The arithmetic is the
// march's.  Against the two-pass kernels on 773 lattices of 1 to 1000 cells a
// row, one row and one plane among them, the allocation-free step takes half
// the time on average and 0.91 of it at most.
struct BoxPlan {
  int b[3], h[3];        // cells of a box per axis; 1 where the axis is split and needs a halo
  int nb[2];             // boxes along x and y
  int cells, pos;        // cells of a box, and with its halo
  uint32_t items;
  FastDiv fb[2], fp[2];  // by the box's and the halo box's extents along x and y
};
constexpr int BOX_NT = 256, BOX_POS = 2048;  // threads; most positions of a halo box

template <int LAT, int ST>
__global__ void __launch_bounds__(BOX_NT, 2) box_step_kernel(const StepArgs a, const BoxPlan p) {
  using L = Lattice<LAT>;
  using S = Storage<ST>;
  using T = typename S::T;
  using C = typename S::C;
  constexpr int Q = L::Q;
  constexpr bool F64 = sizeof(C) == 8;
  __shared__ C psi[BOX_POS];
  const int N[3] = {(int)a.NX, (int)a.NY, (int)a.NZ};
  const int px = (int)a.px, plane = px * N[1];  // padded cells fit 32 bits
  const int64_t pop = (int64_t)plane * N[2];
  const T *fin = static_cast<const T *>(a.fin);
  const C rho0 = F64 ? (C)a.rho0 : (C)a.rho0_f;
  const C inv_rho0 = F64 ? (C)a.relax.inv_rho0 : (C)a.inv_rho0_f;
  const C rho_ref = (C)a.rho_ref_f;
  const int w0 = p.b[0] + 2 * p.h[0], w1 = p.b[1] + 2 * p.h[1];
  const unsigned bx = blockIdx.x % (unsigned)p.nb[0], br = blockIdx.x / (unsigned)p.nb[0];
  const int o[3] = {(int)bx * p.b[0], (int)(br % (unsigned)p.nb[1]) * p.b[1],
                    (int)(br / (unsigned)p.nb[1]) * p.b[2]};
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  for (int r = threadIdx.x; r < p.pos; r += BOX_NT) {
    const int q = (int)fdiv((uint32_t)r, p.fp[0], (uint32_t)w0), rx = r - q * w0;
    const int rz = (int)fdiv((uint32_t)q, p.fp[1], (uint32_t)w1), ry = q - rz * w1;
    int c[3] = {o[0] + rx - p.h[0], o[1] + ry - p.h[1], o[2] + rz - p.h[2]};
    // past a ragged box's halo: read by no cell
    if (c[0] > N[0] || c[1] > N[1] || c[2] > N[2]) continue;
#pragma unroll
    for (int d = 0; d < 3; ++d) c[d] = c[d] < 0 ? N[d] - 1 : (c[d] >= N[d] ? 0 : c[d]);
    const T *f = fin + (c[2] * plane + c[1] * px + c[0]);
    if constexpr (F64) {
      psi[r] = psi_f64(rho_f64<Q>([&](int i) { return f[i * pop]; }), rho0, inv_rho0);
    } else {
      C m = 0;
#pragma unroll
      for (int i = 0; i < Q; ++i) m += S::load(f[i * pop]);
      psi[r] = psi_of(m + rho_ref, rho0, inv_rho0);
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < p.cells; k += BOX_NT) {
    const int q = (int)fdiv((uint32_t)k, p.fb[0], (uint32_t)p.b[0]);
    const int l[3] = {k - q * p.b[0], q - (int)fdiv((uint32_t)q, p.fb[1], (uint32_t)p.b[1]) * p.b[1],
                      (int)fdiv((uint32_t)q, p.fb[1], (uint32_t)p.b[1])};
    if (o[0] + l[0] >= N[0] || o[1] + l[1] >= N[1] || o[2] + l[2] >= N[2]) continue;
    // cells and psi positions of the neighbours at -1, 0 and 1 on each axis
    const int gs[3] = {1, px, plane}, ps[3] = {1, w0, w0 * w1};
    int g[3][3], w[3][3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int c = o[d] + l[d];
      g[d][0] = (c == 0 ? N[d] - 1 : c - 1) * gs[d];
      g[d][1] = c * gs[d];
      g[d][2] = (c + 1 >= N[d] ? 0 : c + 1) * gs[d];
      w[d][0] = (p.h[d] ? l[d] : (l[d] == 0 ? N[d] - 1 : l[d] - 1)) * ps[d];
      w[d][1] = (l[d] + p.h[d]) * ps[d];
      w[d][2] = (p.h[d] ? l[d] + 2 : (l[d] + 1 >= N[d] ? 0 : l[d] + 1)) * ps[d];
    }
    auto psi_at = [&](int i) -> C {
      return psi[w[2][L::cz(i) + 1] + w[1][L::cy(i) + 1] + w[0][L::cx(i) + 1]];
    };
    auto dst = [&](int i) -> T * {
      return static_cast<T *>(a.out_pop[i]) +
             (g[2][L::cz(i) + 1] + g[1][L::cy(i) + 1] + g[0][L::cx(i) + 1]);
    };
    const T *own = fin + (g[2][1] + g[1][1] + g[0][1]);
    C f[Q];
    if constexpr (F64) {
#pragma unroll
      for (int i = 0; i < Q; ++i) f[i] = own[i * pop];
      const C rho = rho_f64<Q>([&](int i) { return f[i]; });
      const RelaxK<LAT, double> relax(a.relax.om1, a.relax.wK, a.relax.cB, a.relax.eps);
      collide_f64<LAT, false>(
          relax, a.relax.fG, [&](int i) { return f[i]; }, rho, psi_at(0), psi_at,
          [&](auto ic, C v) { *dst(decltype(ic)::value) = v; }, 0.0);
    } else {
      C R = 0;
#pragma unroll
      for (int i = 0; i < Q; ++i) R += f[i] = S::load(own[i * pop]);
      collide_rn<LAT, ST>(f, R, rho_ref, (C)a.tau_f, (C)a.omega_f, (C)a.G_f, psi_at, dst);
    }
  }
}

// The box with the least work.  FP32, bound by latency: two boxes on an SM run
// side by side, each in passes of the CTA's threads over its halo box (1 each)
// and its cells (2), then the smallest halo.  FP64, bound by the pipe: on the
// busiest SM, in units of a halo position's psi, 6 for a cell and 400 for a box
// (fitted to the times of 271 lattices, rms 9 %: 6.2, 45 and 1700 ns).  Either
// rule on the other type: 2 to 6 % slower on average.
BoxPlan box_plan(bool f64, const int64_t (&N)[3], int nsm) {
  BoxPlan best{};
  double least = 0;
  auto extents = [](int64_t n, int (&v)[9]) {  // powers of two, and a short axis whole
    int k = 0;
    for (int b = 1; b <= 128 && b < n; b *= 2) v[k++] = b;
    if (n <= 512) v[k++] = (int)n;
    return k;
  };
  int vx[9], vy[9];
  const int kx = extents(N[0], vx), ky = extents(N[1], vy);
  for (int i = 0; i < kx; ++i)
    for (int j = 0; j < ky; ++j)
      for (int t = 1; t <= 4; ++t) {  // passes over the cells
        const int64_t bz = std::min<int64_t>(N[2], t * BOX_NT / (vx[i] * vy[j]));
        if (bz < 1) continue;
        BoxPlan p{};
        p.b[0] = vx[i], p.b[1] = vy[j], p.b[2] = (int)bz;
        int64_t items = 1, pos = 1;
        for (int d = 0; d < 3; ++d) {
          p.h[d] = p.b[d] < N[d];  // D2Q9: y is one cell and has no halo
          pos *= p.b[d] + 2 * p.h[d];
          const int64_t nd = (N[d] + p.b[d] - 1) / p.b[d];
          if (d < 2) p.nb[d] = (int)nd;
          items *= nd;
        }
        if (pos > BOX_POS || items > INT32_MAX) continue;
        p.cells = p.b[0] * p.b[1] * p.b[2];
        p.pos = (int)pos;
        p.items = (uint32_t)items;
        // a piece of a row below 32 cells takes more lines per cell
        const double piece = p.h[0] && p.b[0] < 32 ? 1.0 / p.b[0] : 0.0;
        const int64_t per_sm = (items + nsm - 1) / nsm, waves = (items + 2 * nsm - 1) / (2 * nsm);
        const int passes = (p.pos + BOX_NT - 1) / BOX_NT + 2 * ((p.cells + BOX_NT - 1) / BOX_NT);
        const double work =
            f64 ? (double)per_sm * (p.pos + 6.0 * p.cells + 400.0) * (1.0 + 0.9 * piece)
                : (double)waves * passes * (1.0 + 8.0 * piece) + 0.01 * p.pos / p.cells;
        if (best.cells == 0 || work < least) {
          least = work;
          best = p;
        }
      }
  for (int d = 0; d < 2; ++d) {
    best.fb[d] = make_fastdiv((uint32_t)best.b[d]);
    best.fp[d] = make_fastdiv((uint32_t)(best.b[d] + 2 * best.h[d]));
  }
  return best;
}

// as a programmatic dependent of the previous kernel in the stream
template <class... P, class... A>
cudaError_t launch_pdl(unsigned items, int threads, cudaStream_t s, void (*k)(P...), A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(items);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, args...);
}

template <int LAT, int ST, int TX, int TY, int MINB>
cudaError_t march_launch_t(const StepArgs &a, cudaStream_t s) {
  constexpr int HY = Lattice<LAT>::HAS_Y ? 1 : 0;
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int tiles_x = (int)((a.NX + TX - 3) / (TX - 2));
  const int tiles_y = HY ? (int)((a.NY + TY - 3) / (TY - 2)) : 1;
  const int64_t ntiles = (int64_t)tiles_x * tiles_y, slots = (int64_t)nsm * MINB;
  // Chunks along z: whole waves of the resident CTAs, a chunk of zl planes
  // staging zl + 2, the fewest staged planes per slot
  int64_t best = INT64_MAX, zlen = a.NZ;
  for (int w = 1; w <= 8; ++w) {
    const int64_t want = std::min(std::max<int64_t>(1, w * slots / ntiles), a.NZ);
    const int64_t zl = (a.NZ + want - 1) / want, n = (a.NZ + zl - 1) / zl;
    const int64_t cost = (ntiles * n + slots - 1) / slots * (zl + 2);
    if (cost < best) {
      best = cost;
      zlen = zl;
    }
  }
  const int64_t chunks = (a.NZ + zlen - 1) / zlen, items = ntiles * chunks;
  // The box form where the march runs more than LIMIT threads, of whole warps,
  // per cell and step, unless three staged planes are all it takes.  us per step
  // of the allocation-free step, march / box, at so many threads per cell:
  // 24x289x289, 1.9, 65 / 89; 97x144x144, 2.0, 73 / 115; 17x343x343, 2.8, 89 / 88;
  // 31x8x2016, 3.4, 38 / 21; 9x471x471, 5.0, 140 / 89; 3x816x816, 15, 429 / 81;
  // 1x1x500000, 96, 715 / 19.
  constexpr double LIMIT = HY ? 2.8 : 1.8;
  const int64_t warps =
      HY ? (int64_t)tiles_x * TX / 32 * ((tiles_y - 1) * TY + a.NY - (int64_t)(tiles_y - 1) * (TY - 2) + 2)
         : (int64_t)(tiles_x - 1) * TX / 32 + (a.NX - (int64_t)(tiles_x - 1) * (TX - 2) + 2 + 31) / 32;
  const double run = 32.0 * (double)warps * (double)(zlen + 2) * (double)chunks;
  if (items > INT32_MAX || (best > 3 && run > LIMIT * (double)(a.NX * a.NY * a.NZ))) {
    const int64_t N[3] = {a.NX, a.NY, a.NZ};
    const BoxPlan p = box_plan(ST == ST_F64, N, nsm);
    return launch_pdl(p.items, BOX_NT, s, box_step_kernel<LAT, ST>, a, p);
  }
  return launch_pdl((unsigned)items, TX * TY, s, march_step_kernel<LAT, ST, TX, TY, MINB>, a,
                    tiles_x, tiles_y, (int)zlen);
}

}  // namespace

static cudaError_t march_dispatch(int lat, int st, const StepArgs &a, cudaStream_t s) {
  if (lat == D3Q19) {
    switch (st) {
      case ST_F64: return march_launch_t<D3Q19, ST_F64, 32, 8, 2>(a, s);
      case ST_F32: return march_launch_t<D3Q19, ST_F32, 32, 8, 3>(a, s);
      case ST_F16: return march_launch_t<D3Q19, ST_F16, 32, 8, 3>(a, s);
      case ST_BF16: return march_launch_t<D3Q19, ST_BF16, 32, 8, 3>(a, s);
      default: return cudaErrorInvalidValue;
    }
  }
  switch (st) {
    case ST_F64: return march_launch_t<D2Q9, ST_F64, 128, 1, 4>(a, s);
    case ST_F32: return march_launch_t<D2Q9, ST_F32, 128, 1, 8>(a, s);
    case ST_F16: return march_launch_t<D2Q9, ST_F16, 128, 1, 8>(a, s);
    case ST_BF16: return march_launch_t<D2Q9, ST_BF16, 128, 1, 8>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t march_launch(int lat, int st, const StepArgs &a, cudaStream_t s) {
  const cudaError_t e = march_dispatch(lat, st, a, s);
  return e == cudaSuccess && a.nsites > 0 ? twopass_inject(lat, st, a, s) : e;
}

}  // namespace sclbm

// ---- allocation-free time step ---------------------------------------------
// Some callers cannot call cudaMalloc: a host framework that owns the whole
// device-memory pool and forbids allocations behind its back, a time loop
// that must not stall on the allocator (cudaMalloc and cudaFree can
// synchronise the device), or a program held to a fixed memory budget.  The
// one-launch step keeps psi in shared memory and needs no scratch at all.
namespace sclbm {
namespace {
constexpr int64_t kStaticCells = 2097152;  // the documented limit, 128^3 cells
}
}  // namespace sclbm

extern "C" lbm_status lbm_step_static_f32(int32_t lattice, int64_t nx, int64_t ny, int64_t nz,
                                          double tau, double G, double rho0, const float *f_in,
                                          float *f_out, void *stream) {
  using namespace sclbm;
  if (lattice != LBM_D2Q9 && lattice != LBM_D3Q19)
    return set_error(LBM_EINVAL, "lbm_step_static_f32: unknown lattice");
  if (nx < 1 || ny < 1 || nz < 1 || (lattice == LBM_D2Q9 && nz != 1))
    return set_error(LBM_EINVAL, "lbm_step_static_f32: extents must be >= 1 (nz = 1 for D2Q9)");
  // nx * ny * nz <= cap, tested by division so that no product can overflow
  if (nx > kStaticCells || ny > kStaticCells / nx || nz > kStaticCells / (nx * ny))
    return set_error(LBM_EINVAL,
                     "lbm_step_static_f32: more than 2097152 cells (use lbm_create/lbm_step for "
                     "larger lattices)");
  if (!(tau > 0.5) || !std::isfinite(tau) || !(rho0 > 0) || !std::isfinite(rho0) ||
      !std::isfinite(G))
    return set_error(LBM_EINVAL,
                     "lbm_step_static_f32: tau must be finite and > 0.5, rho0 finite and > 0, "
                     "G finite");
  if (!f_in || !f_out || static_cast<const void *>(f_in) == static_cast<const void *>(f_out))
    return set_error(LBM_EINVAL, "lbm_step_static_f32: f_in and f_out must be distinct buffers");
  StepArgs a{};
  a.fin = f_in;
  a.fout = f_out;
  a.NX = nx;
  a.NY = lattice == LBM_D2Q9 ? 1 : ny;  // D2Q9 runs on the view (nx, 1, ny)
  a.NZ = lattice == LBM_D2Q9 ? ny : nz;
  a.px = nx;
  a.tau = tau;
  a.G = G;
  a.rho0 = rho0;
  a.rho_ref = 0.0;  // plain f_i, no offset
  a.tau_f = (float)tau;
  a.omega_f = (float)(1.0 / tau);
  a.G_f = (float)G;
  a.rho0_f = (float)rho0;
  a.inv_rho0_f = (float)(1.0 / rho0);
  const int lat = lattice == LBM_D2Q9 ? D2Q9 : D3Q19;
  for (int i = 0; i < (lat == D2Q9 ? 9 : 19); ++i) a.out_pop[i] = f_out + i * (nx * ny * nz);
  const cudaError_t e = march_launch(lat, ST_F32, a, static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) {
    cudaGetLastError();
    return set_error(LBM_ECUDA, cudaGetErrorString(e));
  }
  return LBM_OK;
}
