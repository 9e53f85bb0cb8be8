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
// 33x35x31 FP32 10.3 / 4.9; 93^3 FP64 772 / 451; D2Q9 201^2 FP32 10.3 / 3.0,
// 1401x1203 68 / 25, 129^2 FP64 27 / 11; the allocation-free step at
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
      // every rounding written out, as the two-pass kernels have it; the
      // relaxation of opposite velocities runs as paired instructions
      C sx = 0, sy = 0, sz = 0, jx = 0, jy = 0, jz = 0;
      static_for<Q>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        if constexpr (i > 0) {
          const C wp = __fmul_rn((C)L::w(i), psi_at(i));
          sx = cacc_rn<L::cx(i)>(sx, wp);
          sy = cacc_rn<L::cy(i)>(sy, wp);
          sz = cacc_rn<L::cz(i)>(sz, wp);
          jx = cacc_rn<L::cx(i)>(jx, g[i]);
          jy = cacc_rn<L::cy(i)>(jy, g[i]);
          jz = cacc_rn<L::cz(i)>(jz, g[i]);
        }
      });
      const C R = r2, rho = __fadd_rn(rho_ref, R), ir = __fdiv_rn((C)1, rho);
      const C tg = __fmul_rn(tau, -G * psi_at(0));
      const C ux = __fmul_rn(__fmaf_rn(tg, sx, jx), ir), uy = __fmul_rn(__fmaf_rn(tg, sy, jy), ir),
              uz = __fmul_rn(__fmaf_rn(tg, sz, jz), ir);
      const C uu = __fmaf_rn(uz, uz, __fmaf_rn(ux, ux, __fmul_rn(uy, uy)));
      const C K = __fmaf_rn(-__fmul_rn((C)1.5, rho), uu, R);
      static_for<L::NP>([&](auto kc) {
        constexpr int i = L::rep(decltype(kc)::value), o = L::opp(i);
        constexpr float w = (float)L::w(i);
        const C cu = cdot<L::cx(i), L::cy(i), L::cz(i)>(ux, uy, uz);
        const C q = __fmul_rn(__fmul_rn((C)4.5, cu), cu);
        const float2 g2 = make_float2(g[i], g[o]);
        const float2 e2 = make_float2(__fmaf_rn((C)3, cu, q), __fmaf_rn((C)-3, cu, q));
        const float2 X = __ffma2_rn(make_float2(rho, rho), e2, make_float2(K, K));
        const float2 t = __ffma2_rn(make_float2(-w, -w), X, g2);
        const float2 r = __ffma2_rn(make_float2(-omega, -omega), t, g2);
        g[i] = r.x;
        g[o] = r.y;
      });
      C moved = 0;
#pragma unroll
      for (int i = 1; i < Q; ++i) {
        moved = __fadd_rn(moved, g[i]);
        *dst(i) = S::store(g[i]);
      }
      *dst(0) = S::store(__fsub_rn(R, moved));
    }
  }
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
  const int64_t items = ntiles * ((a.NZ + zlen - 1) / zlen);
  if (items > INT32_MAX) return cudaErrorInvalidConfiguration;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)items);
  cfg.blockDim = dim3((unsigned)(TX * TY));
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, march_step_kernel<LAT, ST, TX, TY, MINB>, a, tiles_x, tiles_y,
                            (int)zlen);
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
