// Multi-lattice Shan-Chen model: a reading of the modified model of Sec. 3.1
// and Fig. 1 ("each bubble in its own lattice and fluid in a separate
// lattice"; the lattices are coupled and their interactions computed; eta_m
// switches the barrier off at the rupture criterion and the bubbles merge).
//
// Lattice 0 holds the fluid, lattice k = 1 .. nl-1 the gas of bubble k.
// They interact through the multicomponent Shan-Chen force
//   F_s(x) = -psi_s(x) sum_t Gm[s][t] sum_i w_i psi_t(x + c_i) c_i
// with the coupling matrix Gm[0][0] = G (the fluid's own attraction, the
// single-component model of the hot path), Gm[0][k] = Gm[k][0] = G_x (fluid
// and gas), Gm[k][k] = 0 and Gm[k][l] = eta_m(k, l) G_b between two bubbles.
// Every lattice relaxes with one tau towards f_eq(rho_s, u_s),
//   u' = sum_s j_s / sum_s rho_s,   u_s = u' + tau F_s / rho_s
// (u_s = u' where the lattice is empty: f_eq is 0 there).  eta_m(k, l) = 0
// merges lattice l into k (f_k += f_l, f_l = 0) and removes their coupling.
//
// GB300 form: one launch per step for D2Q9 (psi of a tile and its halo in
// shared memory), psi into a field first for D3Q19; one thread per (cell,
// lattice); populations f[s][i][z][y][x] unpadded, plain values (no offset),
// FP64 or FP32.  The blowing
// agent of site k deposits w_i dm into lattice k (one thread walks the
// sites in order after the step, on the pushed populations at x_k + c_i).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "collide_f64.cuh"
#include "internal.h"
#include "lattice.cuh"
#include "lbm.h"

using namespace sclbm;

namespace {

constexpr int ML_MAX = 8;  // lattices: the fluid and up to seven bubbles
constexpr int TPB = 256;
constexpr int ML_TPB = 256;  // threads of a step CTA at most: two or three CTAs per SM

// (T: the constants in the arithmetic type of the kernel.  Converting them per
// thread would run on the FP64 pipe: with nl^2 couplings per cell that alone
// was a tenth of an FP32 step.)
template <class T>
struct MlArgs {
  const void *fin;
  void *fout;
  int64_t NX, NY, NZ;  // view extents (D2Q9 on (nx, 1, ny))
  int nl;
  T rho0, inv_rho0;
  T om1, wK, cB, eps, fG;  // RelaxArgs
  T Gm[ML_MAX * ML_MAX];
};

inline int nblocks(int64_t n) {
  const int64_t b = (n + TPB - 1) / TPB;
  return (int)std::min<int64_t>(std::max<int64_t>(b, 1), 262144);
}

__device__ __forceinline__ int wrapv(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

// psi = rho0 (1 - exp(-rho/rho0)) in the oracle's operation order
__device__ __forceinline__ double ml_psi(double rho, double rho0) {
  return rho0 * (1.0 - exp(-rho / rho0));
}
__device__ __forceinline__ float ml_psi(float rho, float rho0) {
  return rho0 * (1.0f - expf(-rho / rho0));
}
// the step kernels' psi, density and reciprocal
__device__ __forceinline__ double ml_psi_fast(double rho, double rho0, double inv_rho0) {
  return psi_f64(rho, rho0, inv_rho0);
}
__device__ __forceinline__ float ml_psi_fast(float rho, float rho0, float) {
  return ml_psi(rho, rho0);
}
template <int Q, class T>
__device__ __forceinline__ T ml_rho(const T *f, int64_t N) {
  return rho_f64<Q>([&](int i) { return f[i * N]; });
}
__device__ __forceinline__ double ml_rcp(double v) { return __drcp_rn(v); }
__device__ __forceinline__ float ml_rcp(float v) { return 1.0f / v; }
// a / b.  The front of every gas lattice runs through the subnormal densities
// into cells that are empty, and psi is 0 there while the reciprocal of a
// density below 2^-1024 (FP32: 2^-128) is infinite.  FP64 takes the reciprocal
// where it is finite: a division for every cell cost 2 % of a step (104^2,
// three lattices).
__device__ __forceinline__ double ml_quot(double a, double b) {
  return rcp_overflows(b) ? a / b : a * __drcp_rn(b);
}
__device__ __forceinline__ float ml_quot(float a, float b) { return a / b; }

// What the step kernels need beside MlArgs: the work split (ml_tile).  A CTA
// takes tx x tz cells of every lattice, one thread per (cell, lattice); on the
// field form tx cells of a row or, where rows would leave threads idle, tx that
// follow one another in memory.
struct MlTile {
  int tx, tz;       // cells of a CTA along x and along the view's z (D2Q9)
  int hx;           // 1: the psi tile has a halo along x; 0: tx is the whole row
  int row;          // field form: 1: cells of one row (ML_ROW), else ML_RUN
  int threads, smem;
  unsigned gx, gy;  // grid
  FastDiv fcells, ftx, fpw, fnx, fny;  // by tx tz, tx, tx + 2 hx, NX, NY
};

// psi of every lattice into a field, one thread per (cell, lattice): D3Q19,
// where a tile's one-cell halo would cost as much psi as the tile itself
template <int LAT, class T>
__global__ void __launch_bounds__(TPB) k_ml_psi(const MlArgs<T> a, T *psi) {
  using L = Lattice<LAT>;
  const int64_t N = a.NX * a.NY * a.NZ;
  const T *f = static_cast<const T *>(a.fin);
  const T rho0 = a.rho0, inv_rho0 = a.inv_rho0;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int s = blockIdx.y;
  for (int64_t k = blockIdx.x * (int64_t)TPB + threadIdx.x; k < N; k += (int64_t)gridDim.x * TPB)
    psi[(int64_t)s * N + k] =
        ml_psi_fast(ml_rho<L::Q>(f + (int64_t)s * L::Q * N + k, N), rho0, inv_rho0);
}

// One step of every lattice.  In small lattices (104^2 of the bubble-size
// sweep: 71 cells per SM) the FP64 pipe is the bound only if every SM has
// work, so a CTA holds one thread per (cell, lattice) and ml_tile picks the
// tile that spreads the cells evenly over the SMs; the per-lattice parts
// (density, momentum, psi gradient, relaxation) run side by side and meet in
// shared memory for the two sums over lattices.  Operations follow
// collide_f64.cuh.  Us per step with three lattices, a launch of one thread
// per cell for psi and one for the collision of all lattices (844 FP64
// instructions per cell, 43 CTAs at 104^2) against this form: FP64 104^2 96.9
// / 12.3, 500^2 698 / 218, D3Q19 64x64x48 912 / 244; FP32 104^2 16.4 / 3.4,
// 1000^2 161 / 113, 64x64x48 66.6 / 27.1.
//
// Forms: psi of the tile and a one-cell halo formed in shared memory, one launch
// per step (ML_TILE, D2Q9); psi from k_ml_psi, the CTA's cells of one row
// (ML_ROW) or in memory order (ML_RUN; D3Q19).
enum { ML_TILE = 0, ML_ROW = 1, ML_RUN = 2 };
template <int LAT, class T, int FORM>
__global__ void __launch_bounds__(ML_TPB, sizeof(T) == 8 ? 2 : 3)
    k_ml_step(const MlArgs<T> a, const MlTile tl, const T *psi_field) {
  using L = Lattice<LAT>;
  constexpr int Q = L::Q;
  constexpr bool FIELD = FORM != ML_TILE;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nl = a.nl, cells = tl.tx * tl.tz;
  const int PW = tl.tx + 2 * tl.hx, PC = FIELD ? 0 : PW * (tl.tz + 2);
  T *sG = reinterpret_cast<T *>(smem_raw);  // coupling matrix
  T *mom = sG + ML_MAX * ML_MAX;            // [lattice][rho, j (3), S (3)][cell]
  T *psis = mom + nl * 7 * cells;           // [lattice][PC]
  const int NX = (int)a.NX, NY = (int)a.NY, NZ = (int)a.NZ;
  const int64_t N = a.NX * a.NY * a.NZ;
  const T *f = static_cast<const T *>(a.fin);
  const int tid = threadIdx.x, x0 = blockIdx.y * tl.tx;
  for (int k = tid; k < ML_MAX * ML_MAX; k += blockDim.x) sG[k] = a.Gm[k];
  const RelaxK<LAT, T> relax(a.om1, a.wK, a.cB, a.eps);
  const T rho0 = a.rho0, inv_rho0 = a.inv_rho0;
  const int s = (int)fdiv((uint32_t)tid, tl.fcells, (uint32_t)cells), c = tid - s * cells;
  const int cz_ = FIELD ? 0 : (int)fdiv((uint32_t)c, tl.ftx, (uint32_t)tl.tx);
  const int cx_ = c - cz_ * tl.tx;
  int x = x0 + cx_;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  const T *fs = f + (int64_t)s * Q * N;
  const uint32_t rows = FORM == ML_ROW ? (uint32_t)(a.NY * a.NZ) : gridDim.x;
  for (uint32_t row = FIELD ? blockIdx.x : 0; row < (FIELD ? rows : 1u); row += gridDim.x) {
    int z0, y;
    if constexpr (FORM == ML_RUN) {  // a run of cells; a lattice has fewer than 2^32
      const uint32_t k = (uint32_t)min((uint64_t)row * (uint64_t)cells + (uint64_t)c, (uint64_t)N);
      const uint32_t r = fdiv(k, tl.fnx, (uint32_t)NX);
      x = (int)(k - r * (uint32_t)NX);
      z0 = (int)fdiv(r, tl.fny, (uint32_t)NY);  // NZ past the last cell
      y = (int)(r - (uint32_t)z0 * (uint32_t)NY);
    } else {
      z0 = FIELD ? (int)fdiv(row, tl.fny, (uint32_t)NY) : (int)blockIdx.x * tl.tz;
      y = FIELD ? (int)(row - (uint32_t)z0 * (uint32_t)NY) : 0;
    }
    const int z = z0 + cz_;
    const bool on = s < nl && x < NX && z < NZ;
    if constexpr (!FIELD) {
      if (s < nl)
        for (int r = c; r < PC; r += cells) {
          const int rz = (int)fdiv((uint32_t)r, tl.fpw, (uint32_t)PW);
          // cells past a ragged tile's halo are not read by anyone
          const int hx = x0 + r - rz * PW - tl.hx, hz = z0 + rz - 1;
          if (hx > NX || hz > NZ) continue;
          const uint32_t k = (uint32_t)wrapv(hz, NZ) * (uint32_t)NX + (uint32_t)wrapv(hx, NX);
          psis[s * PC + r] = ml_psi_fast(ml_rho<Q>(fs + k, N), rho0, inv_rho0);
        }
      __syncthreads();
    }
    T fi[Q], rho = 0, psi0 = 0;
    uint32_t nb[Q];  // a lattice has fewer than 2^32 cells (lbm_ml_create)
    if (on) {
      const int xs[3] = {wrapv(x - 1, NX), x, wrapv(x + 1, NX)};
      const int ys[3] = {wrapv(y - 1, NY), y, wrapv(y + 1, NY)};
      const int zs[3] = {wrapv(z - 1, NZ), z, wrapv(z + 1, NZ)};
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        nb[i] = ((uint32_t)zs[L::cz(i) + 1] * (uint32_t)NY + (uint32_t)ys[L::cy(i) + 1]) *
                    (uint32_t)NX + (uint32_t)xs[L::cx(i) + 1];
      }
#pragma unroll
      for (int i = 0; i < Q; ++i) fi[i] = fs[i * N + nb[0]];
      rho = rho_f64<Q>([&](int i) { return fi[i]; });
      const T *pf = FIELD ? psi_field + (int64_t)s * N
                          : psis + s * PC + (cz_ + 1) * PW + cx_ + tl.hx;
      const int xm = tl.hx || cx_ > 0 ? -1 : NX - 1, xp = tl.hx || cx_ + 1 < NX ? 1 : 1 - NX;
      auto psi = [&](int i) -> T {
        return FIELD ? pf[nb[i]]
                     : pf[L::cz(i) * PW + (L::cx(i) > 0 ? xp : (L::cx(i) < 0 ? xm : 0))];
      };
      psi0 = psi(0);
      T j[3], S[3];
      pair_moments<LAT, false, T>(
          [&](auto ic) { return fi[decltype(ic)::value] - fi[L::opp(decltype(ic)::value)]; }, j);
      pair_moments<LAT, true, T>(
          [&](auto ic) { return psi(decltype(ic)::value) - psi(L::opp(decltype(ic)::value)); }, S);
      T *m = mom + s * 7 * cells + c;
      m[0] = rho;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        m[(1 + d) * cells] = j[d];
        m[(4 + d) * cells] = S[d];
      }
    }
    __syncthreads();
    if (on) {
      // common velocity sum j / sum rho and the force sum over lattices
      T rt = 0, jt[3] = {0, 0, 0}, A[3] = {0, 0, 0};
      for (int t = 0; t < nl; ++t) {
        const T *m = mom + t * 7 * cells + c;
        const T g = sG[s * ML_MAX + t];
        rt += m[0];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          if (d == 1 && !L::HAS_Y) continue;
          jt[d] += m[(1 + d) * cells];
          A[d] = fma(g, m[(4 + d) * cells], A[d]);
        }
      }
      const T ir = ml_rcp(rt);
      // u_s = u' + tau F_s / rho_s where the lattice is not empty (fG: -tau w)
      const T h = rho != (T)0 ? ml_quot(a.fG * psi0, rho) : (T)0;
      T v[3], B[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        if (d == 1 && !L::HAS_Y) continue;
        const T u = fma(h, A[d], rcp_overflows(rt) ? jt[d] / rt : jt[d] * ir);
        v[d] = (T)1.5 * u;
        B[d] = relax.cB * (rho * u);
      }
      T *g = static_cast<T *>(a.fout) + (int64_t)s * Q * N;
      relax_pairs<LAT, T>(
          relax, [&](int i) { return fi[i]; }, rho, v, B,
          [&](auto ic, T val) { g[decltype(ic)::value * N + nb[decltype(ic)::value]] = val; });
    }
    if (FORM == ML_ROW) __syncthreads();  // the moments are read before the next row writes them
  }
}

// the blowing agent, site by site in order (one thread): dm = min(rate,
// budget) into lattice site_lat[m] at the pushed destinations x_m + c_i
template <int LAT, class T>
__global__ void k_ml_inject(const MlArgs<T> a, int n, const int32_t *sx, const int32_t *sy,
                            const int32_t *sz, const int32_t *slat, const double *rate,
                            double *budget) {
  using L = Lattice<LAT>;
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const int64_t N = a.NX * a.NY * a.NZ;
  T *g = static_cast<T *>(a.fout);
  for (int m = 0; m < n; ++m) {
    const double b = budget[m];
    if (b <= 0.0) continue;
    const double dm = rate[m] < b ? rate[m] : b;
    budget[m] = b - dm;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
      const int64_t cell =
          ((int64_t)wrapv(sz[m] + L::cz(i), (int)a.NZ) * a.NY + wrapv(sy[m] + L::cy(i), (int)a.NY)) *
              a.NX +
          wrapv(sx[m] + L::cx(i), (int)a.NX);
      T *o = g + ((int64_t)slat[m] * L::Q + i) * N + cell;
      *o = *o + (T)(L::w(i) * dm);
    }
  }
}

// eta_m(k, l) = 0: lattice l merged into lattice k
template <class T>
__global__ void __launch_bounds__(TPB) k_ml_merge(T *f, int64_t QN, int k, int l) {
  for (int64_t m = blockIdx.x * (int64_t)TPB + threadIdx.x; m < QN;
       m += (int64_t)gridDim.x * TPB) {
    f[(int64_t)k * QN + m] = f[(int64_t)k * QN + m] + f[(int64_t)l * QN + m];
    f[(int64_t)l * QN + m] = (T)0;
  }
}

// FP64 fields: densities of every lattice (rho: nl x N, may be null) and the
// pressure of the coupled lattices, p = rho_total/3 + 1/6 sum_s sum_t
// Gm[s][t] psi_s psi_t (p may be null)
template <int LAT, class T>
__global__ void __launch_bounds__(64) k_ml_fields(const MlArgs<double> a, double *rho_out, double *p) {
  using L = Lattice<LAT>;
  const int64_t N = a.NX * a.NY * a.NZ;
  const T *f = static_cast<const T *>(a.fin);
  for (int64_t k = blockIdx.x * (int64_t)64 + threadIdx.x; k < N; k += (int64_t)gridDim.x * 64) {
    double rho[ML_MAX];
    double rt = 0.0;
    for (int s = 0; s < a.nl; ++s) {
      double r = 0.0;
#pragma unroll
      for (int i = 0; i < L::Q; ++i) r += (double)f[((int64_t)s * L::Q + i) * N + k];
      rho[s] = r;
      rt += r;
      if (rho_out) rho_out[(int64_t)s * N + k] = r;
    }
    if (p) {
      double e = 0.0, ps[ML_MAX];
      for (int s = 0; s < a.nl; ++s) ps[s] = ml_psi(rho[s], a.rho0);
      for (int s = 0; s < a.nl; ++s)
        for (int t = 0; t < a.nl; ++t) e += a.Gm[s * ML_MAX + t] * ps[s] * ps[t];
      p[k] = rt / 3.0 + e / 6.0;
    }
  }
}

// f (device, storage type) <-> doubles f[(s*Q + i)*N + user cell]; the
// view's cell order equals the user's (D2Q9: (x, 1, y) has the same linear
// index as (x, y))
template <class T>
__global__ void __launch_bounds__(TPB) k_ml_to_double(const T *f, int64_t n, double *out) {
  for (int64_t m = blockIdx.x * (int64_t)TPB + threadIdx.x; m < n; m += (int64_t)gridDim.x * TPB)
    out[m] = (double)f[m];
}
template <class T>
__global__ void __launch_bounds__(TPB) k_ml_from_double(const double *in, int64_t n, T *f) {
  for (int64_t m = blockIdx.x * (int64_t)TPB + threadIdx.x; m < n; m += (int64_t)gridDim.x * TPB)
    f[m] = (T)in[m];
}
// f = w_i rho (at rest) for one lattice from an FP64 density field
template <int LAT, class T>
__global__ void __launch_bounds__(TPB) k_ml_rest(const double *rho, int64_t N, T *f) {
  using L = Lattice<LAT>;
  for (int64_t k = blockIdx.x * (int64_t)TPB + threadIdx.x; k < N; k += (int64_t)gridDim.x * TPB)
#pragma unroll
    for (int i = 0; i < L::Q; ++i) f[(int64_t)i * N + k] = (T)(L::w(i) * rho[k]);
}

thread_local std::string g_ml_err;

}  // namespace

struct lbm_ml_ctx {
  lbm_ml_config cfg;
  int lat = 0, Q = 0, nl = 0;
  bool f64 = true;
  View v{};
  int64_t N = 0;
  cudaStream_t s = nullptr;
  void *fA = nullptr, *fB = nullptr, *psi = nullptr;
  size_t lat_bytes = 0;
  double *d_rho = nullptr, *d_p = nullptr, *d_tmp = nullptr, *d_bub = nullptr;
  double *d_rate = nullptr, *d_budget = nullptr;
  int32_t *d_site = nullptr;  // x, y, z, lattice per site (view coordinates)
  double *h_mail = nullptr;   // pinned: the film probe's result
  int32_t nsites = 0;
  std::vector<int32_t> site_xyz;
  MlTile tile{};
  int cur = 0;
  bool seeded = false;
  int64_t steps = 0;
  double Gm[ML_MAX * ML_MAX] = {};
  std::vector<std::pair<void **, size_t>> owned;
};

namespace {

lbm_status ml_fail(lbm_status st, const std::string &m) {
  sclbm::set_error(st, m.c_str());
  return st;
}

#define MLCK(call)                                                                   \
  do {                                                                               \
    cudaError_t e_ = (call);                                                         \
    if (e_ != cudaSuccess) {                                                         \
      cudaGetLastError();                                                            \
      return ml_fail(LBM_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    }                                                                                \
  } while (0)
#define MLCKS(expr)              \
  do {                           \
    lbm_status s_ = (expr);      \
    if (s_ != LBM_OK) return s_; \
  } while (0)

lbm_status ml_alloc(lbm_ml_ctx *c, void **p, size_t bytes) {
  if (bytes == 0) bytes = 16;
  if (c->cfg.alloc) {
    *p = c->cfg.alloc(bytes, c->cfg.stream, c->cfg.alloc_user);
    if (!*p) return ml_fail(LBM_ENOMEM, "device allocation failed");
  } else if (cudaMalloc(p, bytes) != cudaSuccess) {
    cudaGetLastError();
    *p = nullptr;
    return ml_fail(LBM_ENOMEM, "cudaMalloc of " + std::to_string(bytes) + " bytes failed");
  }
  c->owned.push_back({p, bytes});
  return LBM_OK;
}

void ml_free_all(lbm_ml_ctx *c) {
  for (auto &o : c->owned)
    if (*o.first) {
      if (c->cfg.free)
        c->cfg.free(*o.first, o.second, c->cfg.stream, c->cfg.alloc_user);
      else
        cudaFree(*o.first);
      *o.first = nullptr;
    }
  c->owned.clear();
}

// a device staging buffer released when it goes out of scope (through the
// context's allocator when it has one)
struct MlTemp {
  lbm_ml_ctx *c;
  void *p = nullptr;
  size_t bytes = 0;
  MlTemp(lbm_ml_ctx *c_, size_t b) : c(c_), bytes(b) {
    if (c->cfg.alloc) {
      p = c->cfg.alloc(bytes, c->cfg.stream, c->cfg.alloc_user);
    } else if (cudaMalloc(&p, bytes) != cudaSuccess) {
      cudaGetLastError();
      p = nullptr;
    }
  }
  ~MlTemp() {
    if (!p) return;
    cudaStreamSynchronize(c->s);
    if (c->cfg.free)
      c->cfg.free(p, bytes, c->cfg.stream, c->cfg.alloc_user);
    else
      cudaFree(p);
  }
};

template <class T>
MlArgs<T> ml_args(const lbm_ml_ctx *c) {
  MlArgs<T> a{};
  a.fin = c->cur == 0 ? c->fA : c->fB;
  a.fout = c->cur == 0 ? c->fB : c->fA;
  a.NX = c->v.NX;
  a.NY = c->v.NY;
  a.NZ = c->v.NZ;
  a.nl = c->nl;
  const RelaxArgs r = make_relax(c->cfg.tau, 1.0, c->cfg.rho0);  // the couplings are in Gm
  a.rho0 = (T)c->cfg.rho0;
  a.inv_rho0 = (T)r.inv_rho0;
  a.om1 = (T)r.om1;
  a.wK = (T)r.wK;
  a.cB = (T)r.cB;
  a.eps = (T)r.eps;
  a.fG = (T)r.fG;
  for (int k = 0; k < ML_MAX * ML_MAX; ++k) a.Gm[k] = (T)c->Gm[k];
  return a;
}

// launched as a programmatic dependent of the previous kernel in the stream
template <class... P, class... A>
void ml_launch(const lbm_ml_ctx *c, dim3 grid, int threads, int smem, void (*k)(P...), A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = c->s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k, args...);  // the error stays for cudaGetLastError
}

// The tile of the step kernel.  D2Q9: the tx x tz with the least work on the
// busiest SM, a cell counting 5 (collision) and a halo position 1 (psi), plus
// 40 for the launch's fixed latency per CTA.  D3Q19: 64 cells (32 from five
// lattices on).
MlTile ml_tile(int lat, int nl, int ts, int64_t NX, int64_t NY, int64_t NZ, int nsm) {
  MlTile best{};
  auto fill = [&](MlTile &t) {
    const int cells = t.tx * t.tz;
    t.threads = (cells * nl + 31) / 32 * 32;
    t.fcells = make_fastdiv((uint32_t)cells);
    t.ftx = make_fastdiv((uint32_t)t.tx);
    t.hx = t.tx < NX || t.tx > NX;
    t.fpw = make_fastdiv((uint32_t)(t.tx + 2 * t.hx));
    t.fnx = make_fastdiv((uint32_t)NX);
    t.fny = make_fastdiv((uint32_t)NY);
    t.smem = ts * (ML_MAX * ML_MAX +
                   nl * (7 * cells + (lat == D2Q9 ? (t.tx + 2 * t.hx) * (t.tz + 2) : 0)));
  };
  if (lat == D3Q19) {
    best.tx = nl > 4 ? 32 : 64;
    best.tz = 1;
    // Rows where they keep 0.8 of the threads busy, in FP64 0.9 of the lanes of
    // the warps that have any (an idle warp costs the pipe nothing); elsewhere
    // cells in memory order, whose two more divisions cost 10 % of an FP32 step
    // on full rows.  us per step, rows / memory order, FP32, one lattice: 1x707x707
    // 781 / 26, 33x8x1894 34 / 26, 64x977x8 22 / 25.
    const int64_t unit = ts == 8 ? 32 : best.tx;
    best.row = NY * NZ <= INT32_MAX &&
               (double)NX >= (ts == 8 ? 0.9 : 0.8) * (double)((NX + unit - 1) / unit * unit);
    best.gx = (unsigned)(best.row ? NY * NZ : (NX * NY * NZ + best.tx - 1) / best.tx);
    best.gy = best.row ? (unsigned)((NX + best.tx - 1) / best.tx) : 1;
    fill(best);
    return best;
  }
  double cost = 0;
  for (int tx0 = 0; tx0 <= 64; tx0 += 8)
    for (int tz = 1; tz <= std::max(32, ML_TPB / std::max(tx0, 1)); ++tz) {
      if (tx0 == 0 && NX > 64) break;
      const int tx = tx0 == 0 ? (int)NX : tx0;  // first: whole rows
      MlTile t{};
      t.tx = tx;
      t.tz = tz;
      fill(t);
      const int64_t gx = (NZ + tz - 1) / tz, gy = (NX + tx - 1) / tx;
      if (t.threads > ML_TPB || t.smem > 48 * 1024 || gy > 65535) continue;
      // beyond a few tiles per SM rows of whole 128-byte lines
      if (gx * gy > 4 * nsm && tx * ts < 128 && tx < NX) continue;
      t.gx = (unsigned)gx;
      t.gy = (unsigned)gy;
      const double w = (double)((gx * gy + nsm - 1) / nsm) *
                       (5.0 * tx * tz + (double)(tx + 2 * t.hx) * (tz + 2) + 40.0);
      if (best.tx == 0 || w < cost) {
        cost = w;
        best = t;
      }
    }
  return best;
}

template <class Fn>
cudaError_t ml_dispatch(const lbm_ml_ctx *c, Fn fn) {
  if (c->lat == D3Q19) {
    if (c->f64)
      fn(std::integral_constant<int, D3Q19>{}, double{});
    else
      fn(std::integral_constant<int, D3Q19>{}, float{});
  } else {
    if (c->f64)
      fn(std::integral_constant<int, D2Q9>{}, double{});
    else
      fn(std::integral_constant<int, D2Q9>{}, float{});
  }
  return cudaGetLastError();
}

lbm_status ml_sync(lbm_ml_ctx *c) {
  MLCK(cudaStreamSynchronize(c->s));
  return LBM_OK;
}

}  // namespace

extern "C" {

void lbm_ml_config_default(lbm_ml_config *cfg) {
  if (!cfg) return;
  std::memset(cfg, 0, sizeof(*cfg));
  cfg->lattice = LBM_D2Q9;
  cfg->storage = LBM_F64;
  cfg->nx = cfg->ny = 128;
  cfg->nz = 1;
  cfg->nl = 3;
  cfg->tau = 1.0;
  cfg->rho0 = 1.0;
  cfg->G = -5.0;
  cfg->G_x = 1.0;
  cfg->G_b = 0.0;
}

lbm_status lbm_ml_create(const lbm_ml_config *cfg, lbm_ml_ctx **out) {
  if (!out) return ml_fail(LBM_EINVAL, "out is NULL");
  *out = nullptr;
  if (!cfg) return ml_fail(LBM_EINVAL, "cfg is NULL");
  if (cfg->lattice != LBM_D2Q9 && cfg->lattice != LBM_D3Q19)
    return ml_fail(LBM_EINVAL, "unknown lattice");
  if (cfg->storage != LBM_F64 && cfg->storage != LBM_F32)
    return ml_fail(LBM_EINVAL, "the multi-lattice model stores FP64 or FP32 populations");
  if (cfg->nl < 1 || cfg->nl > ML_MAX) return ml_fail(LBM_EINVAL, "nl must be 1..8");
  if (cfg->nx < 1 || cfg->ny < 1 || cfg->nz < 1 || (cfg->lattice == LBM_D2Q9 && cfg->nz != 1))
    return ml_fail(LBM_EINVAL, "extents must be >= 1 (nz = 1 for D2Q9)");
  if (cfg->nx > (1 << 20) || cfg->ny > (1 << 20) || cfg->nz > (1 << 20) ||
      cfg->nx * cfg->ny > ((int64_t)1 << 40) / cfg->nz)
    return ml_fail(LBM_EINVAL, "lattice too large");
  if (!(cfg->tau > 0.5) || !std::isfinite(cfg->tau) || !(cfg->rho0 > 0) ||
      !std::isfinite(cfg->rho0) || !std::isfinite(cfg->G) || !std::isfinite(cfg->G_x) ||
      !std::isfinite(cfg->G_b))
    return ml_fail(LBM_EINVAL, "tau finite and > 0.5, rho0 finite and > 0, couplings finite");
  if ((cfg->alloc == nullptr) != (cfg->free == nullptr))
    return ml_fail(LBM_EINVAL, "alloc and free callbacks must be given together");
  lbm_ml_ctx *c = new lbm_ml_ctx();
  c->cfg = *cfg;
  c->lat = cfg->lattice == LBM_D2Q9 ? D2Q9 : D3Q19;
  c->Q = c->lat == D3Q19 ? 19 : 9;
  c->nl = cfg->nl;
  c->f64 = cfg->storage == LBM_F64;
  c->s = static_cast<cudaStream_t>(cfg->stream);
  c->v.lat = c->lat;
  c->v.st = c->f64 ? ST_F64 : ST_F32;
  c->v.NX = cfg->nx;
  c->v.NY = c->lat == D2Q9 ? 1 : cfg->ny;
  c->v.NZ = c->lat == D2Q9 ? cfg->ny : cfg->nz;
  c->v.px = c->v.NX;
  c->v.rho_ref = 0.0;
  view_prepare(c->v);
  c->N = c->v.NX * c->v.NY * c->v.NZ;
  if (c->N > (int64_t)UINT32_MAX) {  // at least 96 bytes a cell: beyond the card's memory
    delete c;
    return ml_fail(LBM_ENOMEM, "device allocation failed");
  }
  // coupling matrix of the reading above; eta_m = 1 for every pair
  for (int s = 0; s < c->nl; ++s)
    for (int t = 0; t < c->nl; ++t)
      c->Gm[s * ML_MAX + t] =
          (s == 0 && t == 0) ? cfg->G : ((s == 0 || t == 0) ? cfg->G_x : (s == t ? 0.0 : cfg->G_b));
  const size_t ts = c->f64 ? 8 : 4;
  int dev = 0, nsm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();  // the allocations below report a missing device
    nsm = 1;
  }
  c->tile = ml_tile(c->lat, c->nl, (int)ts, c->v.NX, c->v.NY, c->v.NZ, nsm);
  c->lat_bytes = ts * (size_t)c->nl * c->Q * c->N;
  lbm_status st;
  auto bail = [&](lbm_status e) {
    lbm_ml_destroy(c);
    return e;
  };
  if ((st = ml_alloc(c, &c->fA, c->lat_bytes)) != LBM_OK) return bail(st);
  if ((st = ml_alloc(c, &c->fB, c->lat_bytes)) != LBM_OK) return bail(st);
  if (c->lat == D3Q19 && (st = ml_alloc(c, &c->psi, ts * (size_t)c->nl * c->N)) != LBM_OK)
    return bail(st);
  if ((st = ml_alloc(c, (void **)&c->d_rho, sizeof(double) * (size_t)c->nl * c->N)) != LBM_OK)
    return bail(st);
  if ((st = ml_alloc(c, (void **)&c->d_p, sizeof(double) * (size_t)c->N)) != LBM_OK) return bail(st);
  if ((st = ml_alloc(c, (void **)&c->d_tmp, sizeof(double) * (size_t)std::max<int64_t>(c->N, 8))) !=
      LBM_OK)
    return bail(st);
  if ((st = ml_alloc(c, (void **)&c->d_bub, sizeof(double) * 4 * ML_MAX)) != LBM_OK) return bail(st);
  if ((st = ml_alloc(c, (void **)&c->d_rate, sizeof(double) * ML_MAX)) != LBM_OK) return bail(st);
  if ((st = ml_alloc(c, (void **)&c->d_budget, sizeof(double) * ML_MAX)) != LBM_OK) return bail(st);
  if ((st = ml_alloc(c, (void **)&c->d_site, sizeof(int32_t) * 4 * ML_MAX)) != LBM_OK)
    return bail(st);
  if (cudaMemsetAsync(c->fA, 0, c->lat_bytes, c->s) != cudaSuccess ||
      cudaMemsetAsync(c->fB, 0, c->lat_bytes, c->s) != cudaSuccess) {
    cudaGetLastError();
    return bail(ml_fail(LBM_ECUDA, "memset failed"));
  }
  *out = c;
  return LBM_OK;
}

void lbm_ml_destroy(lbm_ml_ctx *c) {
  if (!c) return;
  cudaStreamSynchronize(c->s);
  cudaGetLastError();
  ml_free_all(c);
  if (c->h_mail) cudaFreeHost(c->h_mail);
  delete c;
}

lbm_status lbm_ml_coupling(const lbm_ml_ctx *c, double *Gm) {
  if (!c || !Gm) return ml_fail(LBM_EINVAL, "NULL argument");
  for (int s = 0; s < c->nl; ++s)
    for (int t = 0; t < c->nl; ++t) Gm[s * c->nl + t] = c->Gm[s * ML_MAX + t];
  return LBM_OK;
}

lbm_status lbm_ml_seed(lbm_ml_ctx *c, const lbm_bubble *b, double rho_l, double rho_v,
                       double rho_gas, double width, double noise_amp, uint64_t seed) {
  if (!c) return ml_fail(LBM_EINVAL, "ctx is NULL");
  const int nb = c->nl - 1;
  if (nb > 0 && !b) return ml_fail(LBM_EINVAL, "need nl - 1 bubbles");
  if (!(width > 0) || !std::isfinite(rho_l) || !std::isfinite(rho_v) || !std::isfinite(rho_gas) ||
      !std::isfinite(noise_amp))
    return ml_fail(LBM_EINVAL, "width > 0, densities finite");
  std::vector<double> vb(4 * ML_MAX, 0.0);
  c->site_xyz.assign(4 * ML_MAX, 0);
  for (int k = 0; k < nb; ++k) {
    if (!std::isfinite(b[k].x) || !std::isfinite(b[k].y) || !std::isfinite(b[k].z) ||
        !std::isfinite(b[k].r))
      return ml_fail(LBM_EINVAL, "non-finite bubble");
    double vx = b[k].x, vy = b[k].y, vz = b[k].z;
    if (c->lat == D2Q9) {
      vz = b[k].y;
      vy = 0.0;
    }
    vb[4 * k + 0] = vx;
    vb[4 * k + 1] = vy;
    vb[4 * k + 2] = vz;
    vb[4 * k + 3] = b[k].r;
    auto wr = [](double p, int64_t n) {
      int64_t q = (int64_t)std::floor(p + 0.5) % n;
      return (int32_t)(q < 0 ? q + n : q);
    };
    c->site_xyz[4 * k + 0] = wr(vx, c->v.NX);
    c->site_xyz[4 * k + 1] = wr(vy, c->v.NY);
    c->site_xyz[4 * k + 2] = wr(vz, c->v.NZ);
    c->site_xyz[4 * k + 3] = k + 1;
  }
  MLCK(cudaMemcpyAsync(c->d_bub, vb.data(), sizeof(double) * vb.size(), cudaMemcpyHostToDevice, c->s));
  c->cur = 0;
  double *rho = c->d_tmp;
  const int64_t QN = (int64_t)c->Q * c->N;
  // the fluid: every bubble, liquid rho_l, its vapour rho_v inside, noise
  MLCK(diag_init_rho(c->v, c->d_bub, nb, rho_l, rho_v, width, noise_amp, seed, rho, c->s));
  MLCK(ml_dispatch(c, [&](auto L, auto T) {
    using TT = decltype(T);
    k_ml_rest<decltype(L)::value, TT><<<nblocks(c->N), TPB, 0, c->s>>>(rho, c->N,
                                                                        static_cast<TT *>(c->fA));
  }));
  // bubble k's gas: rho_gas inside bubble k, zero far outside, no noise
  for (int k = 0; k < nb; ++k) {
    MLCK(diag_init_rho(c->v, c->d_bub + 4 * k, 1, 0.0, rho_gas, width, 0.0, seed, rho, c->s));
    MLCK(ml_dispatch(c, [&](auto L, auto T) {
      using TT = decltype(T);
      k_ml_rest<decltype(L)::value, TT><<<nblocks(c->N), TPB, 0, c->s>>>(
          rho, c->N, static_cast<TT *>(c->fA) + (int64_t)(k + 1) * QN);
    }));
  }
  // every pair's barrier back on
  for (int s = 0; s < c->nl; ++s)
    for (int t = 0; t < c->nl; ++t)
      if (s != t && s > 0 && t > 0) c->Gm[s * ML_MAX + t] = c->cfg.G_b;
  c->nsites = 0;
  c->steps = 0;
  c->seeded = true;
  return ml_sync(c);
}

lbm_status lbm_ml_write_f(lbm_ml_ctx *c, const double *f, size_t bytes) {
  if (!c || !f) return ml_fail(LBM_EINVAL, "NULL argument");
  const int64_t n = (int64_t)c->nl * c->Q * c->N;
  if (bytes != (size_t)n * sizeof(double)) return ml_fail(LBM_EINVAL, "bytes must be nl*Q*N*8");
  MlTemp tmp(c, bytes);
  if (!tmp.p) return ml_fail(LBM_ENOMEM, "staging allocation failed");
  double *d = static_cast<double *>(tmp.p);
  MLCK(cudaMemcpyAsync(d, f, bytes, cudaMemcpyHostToDevice, c->s));
  void *dst = c->cur == 0 ? c->fA : c->fB;
  MLCK(ml_dispatch(c, [&](auto, auto T) {
    using TT = decltype(T);
    k_ml_from_double<TT><<<nblocks(n), TPB, 0, c->s>>>(d, n, static_cast<TT *>(dst));
  }));
  MLCKS(ml_sync(c));
  c->seeded = true;
  return LBM_OK;
}

lbm_status lbm_ml_read_f(lbm_ml_ctx *c, double *f, size_t bytes) {
  if (!c || !f) return ml_fail(LBM_EINVAL, "NULL argument");
  if (!c->seeded) return ml_fail(LBM_ESTATE, "seed the lattices first");
  const int64_t n = (int64_t)c->nl * c->Q * c->N;
  if (bytes != (size_t)n * sizeof(double)) return ml_fail(LBM_EINVAL, "bytes must be nl*Q*N*8");
  MlTemp tmp(c, bytes);
  if (!tmp.p) return ml_fail(LBM_ENOMEM, "staging allocation failed");
  double *d = static_cast<double *>(tmp.p);
  const void *src = c->cur == 0 ? c->fA : c->fB;
  MLCK(ml_dispatch(c, [&](auto, auto T) {
    using TT = decltype(T);
    k_ml_to_double<TT><<<nblocks(n), TPB, 0, c->s>>>(static_cast<const TT *>(src), n, d);
  }));
  MLCK(cudaMemcpyAsync(f, d, bytes, cudaMemcpyDeviceToHost, c->s));
  return ml_sync(c);
}

lbm_status lbm_ml_inject(lbm_ml_ctx *c, const double *rate, const double *budget, int32_t n) {
  if (!c) return ml_fail(LBM_EINVAL, "ctx is NULL");
  if (!c->seeded) return ml_fail(LBM_ESTATE, "seed the lattices first");
  if (n == 0) {
    c->nsites = 0;
    return LBM_OK;
  }
  if (n != c->nl - 1 || !rate || !budget)
    return ml_fail(LBM_EINVAL, "n must be 0 or the number of bubbles (nl - 1)");
  for (int k = 0; k < n; ++k)
    if (!(rate[k] >= 0) || !(budget[k] >= 0) || !std::isfinite(rate[k]) || !std::isfinite(budget[k]))
      return ml_fail(LBM_EINVAL, "rates and budgets must be finite and >= 0");
  MLCK(cudaMemcpyAsync(c->d_rate, rate, sizeof(double) * n, cudaMemcpyHostToDevice, c->s));
  MLCK(cudaMemcpyAsync(c->d_budget, budget, sizeof(double) * n, cudaMemcpyHostToDevice, c->s));
  // site lists x, y, z, lattice as four arrays of ML_MAX
  std::vector<int32_t> sites(4 * ML_MAX, 0);
  for (int k = 0; k < n; ++k)
    for (int q = 0; q < 4; ++q) sites[q * ML_MAX + k] = c->site_xyz[4 * k + q];
  MLCK(cudaMemcpyAsync(c->d_site, sites.data(), sizeof(int32_t) * sites.size(),
                       cudaMemcpyHostToDevice, c->s));
  MLCKS(ml_sync(c));
  c->nsites = n;
  return LBM_OK;
}

lbm_status lbm_ml_read_budgets(lbm_ml_ctx *c, double *budget, int32_t n) {
  if (!c || !budget) return ml_fail(LBM_EINVAL, "NULL argument");
  if (n != c->nsites) return ml_fail(LBM_EINVAL, "n must equal the number of injecting sites");
  if (n == 0) return LBM_OK;
  MLCK(cudaMemcpyAsync(budget, c->d_budget, sizeof(double) * n, cudaMemcpyDeviceToHost, c->s));
  return ml_sync(c);
}

lbm_status lbm_ml_step(lbm_ml_ctx *c, int64_t nsteps) {
  if (!c) return ml_fail(LBM_EINVAL, "ctx is NULL");
  if (nsteps < 0) return ml_fail(LBM_EINVAL, "nsteps < 0");
  if (!c->seeded) return ml_fail(LBM_ESTATE, "seed the lattices first");
  for (int64_t t = 0; t < nsteps; ++t) {
    cudaError_t e = ml_dispatch(c, [&](auto L, auto T) {
      using TT = decltype(T);
      constexpr int lat = decltype(L)::value;
      const MlArgs<TT> a = ml_args<TT>(c);
      TT *psi = static_cast<TT *>(c->psi);
      if constexpr (lat == D3Q19)
        ml_launch(c, dim3((unsigned)nblocks(c->N), (unsigned)c->nl), TPB, 0, k_ml_psi<lat, TT>, a,
                  psi);
      auto step = [&](auto form) {
        ml_launch(c, dim3(c->tile.gx, c->tile.gy), c->tile.threads, c->tile.smem,
                  k_ml_step<lat, TT, decltype(form)::value>, a, c->tile,
                  static_cast<const TT *>(psi));
      };
      if constexpr (lat == D2Q9)
        step(std::integral_constant<int, ML_TILE>{});
      else if (c->tile.row)
        step(std::integral_constant<int, ML_ROW>{});
      else
        step(std::integral_constant<int, ML_RUN>{});
    });
    if (e == cudaSuccess && c->nsites > 0) e = ml_dispatch(c, [&](auto L, auto T) {
      using TT = decltype(T);
      constexpr int lat = decltype(L)::value;
      const MlArgs<TT> a = ml_args<TT>(c);
      k_ml_inject<lat, TT><<<1, 32, 0, c->s>>>(a, c->nsites, c->d_site, c->d_site + ML_MAX,
                                                c->d_site + 2 * ML_MAX, c->d_site + 3 * ML_MAX,
                                                c->d_rate, c->d_budget);
    });
    if (e != cudaSuccess) {
      cudaGetLastError();
      return ml_fail(LBM_ECUDA, std::string("multi-lattice step: ") + cudaGetErrorString(e));
    }
    c->cur = 1 - c->cur;
    ++c->steps;
  }
  return LBM_OK;
}

int64_t lbm_ml_step_count(const lbm_ml_ctx *c) { return c ? c->steps : -1; }

lbm_status lbm_ml_merge(lbm_ml_ctx *c, int32_t k, int32_t l) {
  if (!c) return ml_fail(LBM_EINVAL, "ctx is NULL");
  if (!c->seeded) return ml_fail(LBM_ESTATE, "seed the lattices first");
  if (k < 1 || l < 1 || k >= c->nl || l >= c->nl || k == l)
    return ml_fail(LBM_EINVAL, "k and l must be two different bubble lattices (1 .. nl-1)");
  const int64_t QN = (int64_t)c->Q * c->N;
  void *f = c->cur == 0 ? c->fA : c->fB;
  MLCK(ml_dispatch(c, [&](auto, auto T) {
    using TT = decltype(T);
    k_ml_merge<TT><<<nblocks(QN), TPB, 0, c->s>>>(static_cast<TT *>(f), QN, k, l);
  }));
  c->Gm[k * ML_MAX + l] = c->Gm[l * ML_MAX + k] = 0.0;
  return ml_sync(c);
}

// densities and pressure of the current state into d_rho and d_p (enqueued)
static lbm_status ml_enqueue_fields(lbm_ml_ctx *c) {
  const MlArgs<double> a = ml_args<double>(c);
  MLCK(ml_dispatch(c, [&](auto L, auto T) {
    k_ml_fields<decltype(L)::value, decltype(T)>
        <<<(int)std::min<int64_t>((c->N + 63) / 64, 1 << 20), 64, 0, c->s>>>(a, c->d_rho, c->d_p);
  }));
  return LBM_OK;
}

lbm_status lbm_ml_fields(lbm_ml_ctx *c, double *rho, double *p) {
  if (!c) return ml_fail(LBM_EINVAL, "ctx is NULL");
  if (!c->seeded) return ml_fail(LBM_ESTATE, "seed the lattices first");
  MLCKS(ml_enqueue_fields(c));
  if (rho)
    MLCK(cudaMemcpyAsync(rho, c->d_rho, sizeof(double) * (size_t)c->nl * c->N,
                         cudaMemcpyDeviceToHost, c->s));
  if (p) MLCK(cudaMemcpyAsync(p, c->d_p, sizeof(double) * (size_t)c->N, cudaMemcpyDeviceToHost, c->s));
  return ml_sync(c);
}

lbm_status lbm_ml_run_until_rupture(lbm_ml_ctx *c, const int64_t *line, double rho_mid,
                                     double eps_arm, double h_max, int64_t diag_every,
                                     int64_t max_steps, int32_t k, int32_t l, lbm_rupture *out) {
  if (!c || !line || !out) return ml_fail(LBM_EINVAL, "NULL argument");
  if (!c->seeded) return ml_fail(LBM_ESTATE, "seed the lattices first");
  const int dims = c->lat == D2Q9 ? 2 : 3;
  if (line[3] < 0 || line[3] >= dims || line[4] < 2)
    return ml_fail(LBM_EINVAL, "line = {x, y, z, axis (< dims), len >= 2}");
  if (diag_every < 1 || max_steps < 0 || !(eps_arm >= 0) || !(h_max > 0))
    return ml_fail(LBM_EINVAL, "diag_every >= 1, max_steps >= 0, eps_arm >= 0, h_max > 0");
  if (k < 1 || l < 1 || k >= c->nl || l >= c->nl || k == l)
    return ml_fail(LBM_EINVAL, "k and l must be two different bubble lattices (1 .. nl-1)");
  std::memset(out, 0, sizeof(*out));
  auto vaxis = [&](int a) { return c->lat == D2Q9 ? (a == 0 ? 0 : 2) : a; };
  int e[3] = {0, 0, 0}, ep[3] = {0, 0, 0};
  e[vaxis((int)line[3])] = 1;
  ep[vaxis(((int)line[3] + 1) % dims)] = 1;
  int64_t x0 = line[0], y0 = line[1], z0 = line[2];
  if (c->lat == D2Q9) {
    z0 = y0;
    y0 = 0;
  }
  auto wr = [](int64_t a, int64_t n) {
    const int64_t r = a % n;
    return r < 0 ? r + n : r;
  };
  bool armed = false;
  double h_prev = 0.0, d_prev = 0.0;
  if (!c->h_mail) MLCK(cudaMallocHost(reinterpret_cast<void **>(&c->h_mail), 6 * sizeof(double)));
  double *h = c->h_mail;
  int64_t t = 0;
  while (t < max_steps) {
    const int64_t n = std::min(diag_every, max_steps - t);
    MLCKS(lbm_ml_step(c, n));
    t += n;
    // the film on the fluid lattice's density, with the coupled pressure
    MLCKS(ml_enqueue_fields(c));
    MLCK(diag_film_probe(c->v, c->d_rho, c->d_p, wr(x0, c->v.NX), wr(y0, c->v.NY), wr(z0, c->v.NZ),
                         e, ep, line[4], rho_mid, h, FilmRule{0, armed, eps_arm, h_max}, c->s));
    MLCKS(ml_sync(c));
    out->steps = t;
    const bool found = h[0] != 0.0;
    const double hh = h[3], d2 = h[4];
    if (!found) {  // the film is gone before the criterion fired
      out->merged = 1;
      return LBM_OK;
    }
    if (hh > h_max) {
      armed = false;
    } else if (d2 < -eps_arm) {
      armed = true;
    } else if (armed && d2 >= 0.0) {
      // eta_m = 0: the barrier goes and the pair's lattices merge
      out->fired = 1;
      out->h_c = h_prev + (hh - h_prev) * (-d_prev / (d2 - d_prev));
      out->h_probe = hh;
      out->r_d = h[5];
      return lbm_ml_merge(c, k, l);
    }
    h_prev = hh;
    d_prev = d2;
  }
  return LBM_OK;
}

}  // extern "C"
