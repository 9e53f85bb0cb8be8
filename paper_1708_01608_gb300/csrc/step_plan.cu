// Host side of the fused step: tile table, launch plan, TMA descriptors and
// dispatch to the per-storage translation units.
#include <climits>
#include <algorithm>

#include "step_fused.cuh"

namespace sclbm {

bool fused_tile_shape(int lat, int st, int tile, int *bx, int *by, int *nstage, int *xc) {
  int cells = 1;
#define SCLBM_T(id, BX, BY, NS) \
  case id:                      \
    *bx = BX;                   \
    *by = BY;                   \
    *nstage = NS;               \
    if (xc) *xc = cells;        \
    return true;
  if (lat == D3Q19) {
    switch (tile) { SCLBM_D3Q19_TILES(SCLBM_T) }
  } else {
    switch (tile) { SCLBM_D2Q9_TILES(SCLBM_T) }
  }
  if (st == ST_F64) return false;  // the x-pair kernel computes in FP32
  cells = 2;
  if (lat == D3Q19) {
    switch (tile) { SCLBM_D3Q19_X2_TILES(SCLBM_T) }
  } else {
    switch (tile) { SCLBM_D2Q9_X2_TILES(SCLBM_T) }
  }
#undef SCLBM_T
  return false;
}

static int fused_smem_bytes(int lat, int st, int tile, int xc) {
  if (xc == 2) {
    switch (st) {
      case ST_F32: return fused_x2_smem_f32(lat, tile);
      case ST_F16:
      case ST_F16R: return fused_x2_smem_f16(lat, tile);
      case ST_BF16:
      case ST_BF16R: return fused_x2_smem_bf16(lat, tile);
      default: return -1;
    }
  }
  switch (st) {
    case ST_F64: return fused_smem_f64(lat, tile);
    case ST_F32: return fused_smem_f32(lat, tile);
    default: return fused_smem_h16(lat, st, tile);
  }
}

// The plan of a lattice whose tile the caller leaves open: the tile and chunk
// count with the least time in this model (lbm_autotune measures instead).  A
// CTA of a chunk of zl planes stages zl + 2 planes one after the other; a
// plane takes max(floor, ns * cells * co), with co CTAs resident on an SM
// (they share its issue slots and its memory path), and the step no less than
// its populations take at the copy bandwidth.  The constants are fitted to the
// times of every tile at 32^3 to 256^3 and 64^2 to 2000^2.  Every tile gives a
// lattice the same bits.
namespace {
struct TileCost {
  int tile;
  // a plane in us: at least floor, ns per cell and resident CTA; with both
  // lattices in L2, and beyond (one plane's HBM latency bounds a lone CTA)
  float floor_l2, ns_l2, floor_hbm, ns_hbm;
};
// Us per step, former default (tile 1, at least 4 planes per chunk) / now.
// FP32: 32^3 7.8 / 4.3, 64^3 11.8 / 9.9, 128^3 65.4 / 53.3, 256^3 464 / 394,
// 512^3 4218 / 3178.  Tile 25 is for lattices it splits into one even wave
// (128^3: 152 CTAs); in several waves it is the slower one (512^3: 3341).
constexpr TileCost COST_F32[] = {{16, 1.1f, 2.45f, 1.35f, 3.03f}, {14, 1.1f, 2.45f, 1.35f, 3.03f},
                                 {25, 1.1f, 2.45f, 1.35f, 3.03f}, {2, 0.5f, 4.0f, 1.35f, 6.0f}};
// 16-bit: 32^3 7.9 / 4.4, 128^3 49.0 / 36.5, 256^3 379 / 238, 512^3 2848 / 1794
constexpr TileCost COST_H16[] = {{24, 1.0f, 1.75f, 1.2f, 1.95f}, {23, 1.0f, 1.75f, 1.2f, 1.95f},
                                 {2, 0.5f, 4.0f, 1.2f, 4.0f}};
// 16-bit with the rounding residual: 256^3 460 / 283
constexpr TileCost COST_H16R[] = {{23, 1.2f, 2.1f, 1.7f, 2.4f}, {24, 1.2f, 2.1f, 1.7f, 2.4f},
                                  {2, 0.55f, 4.5f, 1.7f, 4.5f}};
// FP64 is bound by the FP64 pipe, which the CTAs of an SM share: 32^3 64 / 24
constexpr TileCost COST_F64[] = {{6, 0.0f, 49.0f, 0.0f, 49.0f}, {7, 0.0f, 49.0f, 0.0f, 49.0f},
                                 {2, 0.0f, 54.0f, 0.0f, 54.0f}};
// D2Q9, FP32 and 16-bit (the floor adds here: co-resident rows overlap):
// 64^2 4.6 / 2.7, 200^2 4.9 / 3.2, 512^2 7.4 / 5.6, 2000^2 56.5 / 50.5
constexpr TileCost COST_2D[] = {{4, 0.35f, 0.5f, 0.35f, 0.5f}, {6, 0.35f, 0.6f, 0.35f, 0.6f},
                                {3, 0.33f, 0.8f, 0.33f, 0.8f}};
// D2Q9 FP64: 64^2 21.1 / 9.2, 128^2 22.0 / 9.7, 512^2 60 / 56.5
constexpr TileCost COST_2D_F64[] = {{1, 2.6f, 25.5f, 2.6f, 25.5f}, {3, 2.6f, 25.5f, 2.6f, 25.5f}};

// Narrow lattices with D3Q19 and FP32 arithmetic: rows of 4 to 48 cells, fewer
// than 8 rows, in FP32 also up to 8 planes.  The copies of a box go row by row
// and the columns past the lattice are filled in, so that a plane takes nearly
// as long as a full one, which the model above, in cells of the lattice, does
// not know (8x250000x1 FP32: its plan, tile 14, 975 us, tile 1 437).  There its
// plan is compared with tile 1 and the chunks of lbm_config.tile = 1 in a second
// model: a plane takes max(floor, base + co row rows) us, rows the box's rows in
// the lattice and its two halo rows, the two halo planes count as `planes`
// planes, and a CTA takes start us besides.  Fitted to 6700 times on 591 such
// lattices (rms 7 to 14 %; the tiles then scaled by up to 14 % for the choice).
// Time against the better of the two plans, first model alone / now, mean and
// largest: FP32 1.13, 2.23 / 1.01, 1.17; 16-bit 1.06, 1.56 / 1.01, 1.09.
struct RowCost {
  int tile;
  float start, base, row, planes, floor;
};
constexpr RowCost ROW_F32[] = {{1, 2.92f, 0.840f, 0.0432f, 0.00f, 0.49f},
                               {2, 1.69f, 0.524f, 0.0646f, 0.87f, 0.84f},
                               {14, 1.70f, 0.952f, 0.0590f, 1.18f, 1.17f},
                               {16, 0.55f, 0.348f, 0.0500f, 2.47f, 1.02f},
                               {25, 3.02f, 0.754f, 0.0591f, 0.11f, 0.99f}};
constexpr RowCost ROW_H16[] = {{1, 1.31f, 1.168f, 0.0524f, 1.14f, 1.32f},
                               {2, 0.15f, 0.711f, 0.0465f, 2.81f, 0.94f},
                               {23, 1.73f, 0.738f, 0.0674f, 1.01f, 1.03f},
                               {24, 2.71f, 0.823f, 0.0558f, 0.41f, 0.66f}};
constexpr RowCost ROW_H16R[] = {{1, 1.41f, 1.232f, 0.0606f, 0.96f, 1.50f},
                                {2, 0.00f, 0.904f, 0.0487f, 2.42f, 1.15f},
                                {23, 1.00f, 0.983f, 0.0734f, 1.06f, 1.35f},
                                {24, 0.01f, 0.277f, 0.1149f, 1.91f, 1.60f}};

// us of a plan in that model; < 0: the tile is not in it
template <size_t N>
double row_us(const RowCost (&cand)[N], const FusedPlan &q, int st, int64_t NX, int64_t NY,
              int64_t NZ, int nsm) {
  int per_sm = 0;
  if (fused_prepare(D3Q19, st, q, &per_sm) != cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    return -1.0;
  }
  for (const RowCost &c : cand) {
    if (c.tile != q.tile) continue;
    const double zl = (double)q.zlen, bytes = (double)NX * NY * NZ * 38 * (double)storage_bytes(st);
    const double us = c.row * (double)(std::min<int64_t>(q.by, NY) + 2);
    auto wave = [&](int64_t co) {
      return c.start + (zl + c.planes) * std::max<double>(c.floor, c.base + us * (double)co);
    };
    const int64_t m = (q.items + nsm - 1) / nsm;  // CTAs of the busiest SM
    const double t = (double)(m / per_sm) * wave(per_sm) + (m % per_sm ? wave(m % per_sm) : 0.0);
    const double mem = bytes < 100e6 ? 0.0 : bytes * (1.0 + 0.35 / zl) / 6.7e6;
    const double far = bytes < 100e6 ? 1.0 : 1.0 + 0.02 * std::max(0.0, zl / 64 - 1.0);
    return (std::max(t, mem) + 0.05 * t) * far;
  }
  return -1.0;
}

template <size_t N>
cudaError_t pick_plan(const TileCost (&cand)[N], int lat, int st, int64_t NX, int64_t NY,
                      int64_t NZ, bool rows, FusedPlan *p) {
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const double bytes =
      (double)NX * NY * NZ * 2 * (lat == D3Q19 ? 19 : 9) * (double)storage_bytes(st);
  const bool in_l2 = bytes < 100e6;
  const double psi_only = st == ST_F64 ? 0.6 : 2.0;  // the two halo planes, in whole planes
  double best = 0;
  bool found = false;
  for (const TileCost &c : cand) {
    FusedPlan q;
    if (fused_make_plan(lat, st, c.tile, NX, NY, NZ, 1, &q, rows) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    int per_sm = 0;
    if (fused_prepare(lat, st, q, &per_sm) != cudaSuccess || per_sm < 1) {
      cudaGetLastError();
      continue;
    }
    const int64_t ntiles = (int64_t)q.tiles_x * q.tiles_y;
    // a ragged last tile takes a plane as long as a full one
    const double width = (double)std::min<int64_t>(q.bx, lat == D2Q9 ? (NX + 31) / 32 * 32 : NX);
    const double ns = (in_l2 ? c.ns_l2 : c.ns_hbm) * 1e-3 * width * q.by;
    const double floor_us = in_l2 ? c.floor_l2 : c.floor_hbm;
    // every chunk count that can be formed (about 2 sqrt(NZ) of them)
    for (int64_t zl = NZ; zl >= 1; --zl) {
      const int64_t n = (NZ + zl - 1) / zl;
      zl = (NZ + n - 1) / n;
      if (ntiles * n > INT_MAX) break;
      const int64_t m = (ntiles * n + nsm - 1) / nsm;  // CTAs of the busiest SM
      if (q.tile == 25 && lat == D3Q19 && m > per_sm) continue;
      auto plane = [&](int64_t co) {
        if (lat == D3Q19) return std::max(floor_us, ns * (double)co);
        return st == ST_F64 ? std::max(floor_us, 0.6 + ns * (double)co) : floor_us + ns * (double)co;
      };
      const double t = ((double)zl + psi_only) * ((double)(m / per_sm) * plane(per_sm) +
                                                  (m % per_sm ? plane(m % per_sm) : 0.0));
      const double mem = in_l2 ? 0.0 : bytes * (1.0 + 0.35 / (double)zl) / 6.7e6;
      // long chunks of a lattice beyond L2 lose the overlap of neighbouring
      // columns' halo rows (512^3 FP32: 3264 us in 2 chunks, 3160 in 8)
      const double far = in_l2 ? 1.0 : 1.0 + 0.02 * std::max(0.0, (double)zl / 64 - 1.0);
      const double cost = (std::max(t, mem) + 0.05 * t) * far;
      if (!found || cost < best) {
        best = cost;
        *p = q;
        p->zlen = (int)zl;
        p->nzc = (int)n;
        p->items = (int)(ntiles * n);
        found = true;
      }
    }
  }
  if (!found) return cudaErrorInvalidValue;
  FusedPlan q;
  if (lat == D3Q19 && st != ST_F64 && !rows && (NX <= 48 || NY < 8 || (st == ST_F32 && NZ <= 8)) &&
      fused_make_plan(lat, st, 1, NX, NY, NZ, 0, &q) == cudaSuccess) {
    auto us = [&](const FusedPlan &r) {
      return st == ST_F32 ? row_us(ROW_F32, r, st, NX, NY, NZ, nsm)
             : st == ST_F16R || st == ST_BF16R ? row_us(ROW_H16R, r, st, NX, NY, NZ, nsm)
                                               : row_us(ROW_H16, r, st, NX, NY, NZ, nsm);
    };
    if (us(q) >= 0.0 && us(q) < us(*p)) *p = q;
  }
  return cudaSuccess;
}
}  // namespace

cudaError_t fused_make_plan(int lat, int st, int tile, int64_t NX, int64_t NY, int64_t NZ,
                            int nzc, FusedPlan *p, bool rows) {
  int bx, by, ns, xc;
  if (tile <= 0) {
    if (lat == D2Q9)
      return st == ST_F64 ? pick_plan(COST_2D_F64, lat, st, NX, NY, NZ, rows, p)
                          : pick_plan(COST_2D, lat, st, NX, NY, NZ, rows, p);
    return st == ST_F64   ? pick_plan(COST_F64, lat, st, NX, NY, NZ, rows, p)
           : st == ST_F32 ? pick_plan(COST_F32, lat, st, NX, NY, NZ, rows, p)
           : st == ST_F16R || st == ST_BF16R ? pick_plan(COST_H16R, lat, st, NX, NY, NZ, rows, p)
                                             : pick_plan(COST_H16, lat, st, NX, NY, NZ, rows, p);
  }
  if (!fused_tile_shape(lat, st, tile, &bx, &by, &ns, &xc)) return cudaErrorInvalidValue;
  p->tile = tile;
  p->bx = bx;
  p->by = by;
  p->nstage = ns;
  p->xc = xc;
  p->threads = bx * by / xc;
  p->hx = (int)(16 / storage_bytes(st));
  p->smem = fused_smem_bytes(lat, st, tile, xc);
  p->rows = rows;
  if (rows && xc != 2) return cudaErrorInvalidValue;
  if (!rows && NX % p->hx != 0) return cudaErrorInvalidValue;  // halo boxes must start on 16 bytes
  int dev = 0, nsm = 0, smem_optin = 0, smem_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  if (p->smem <= 0 || p->smem > smem_optin) return cudaErrorInvalidValue;
  p->tiles_x = (int)((NX + bx - 1) / bx);
  p->tiles_y = (int)((NY + by - 1) / by);
  const int ntiles = p->tiles_x * p->tiles_y;
  if (nzc <= 0) {
    // resident CTA slots: SMs x the kernel's occupancy (registers, shared
    // memory and threads)
    int per_sm = 0;
    if (fused_prepare(lat, st, *p, &per_sm) != cudaSuccess || per_sm < 1) {
      cudaGetLastError();
      per_sm = std::max(1, std::min(smem_sm / (p->smem + 1024), 2048 / p->threads));
    }
    // Time model: CTAs run in waves of `slots`, a chunk of zlen planes
    // stages zlen + 2; pick the number of chunks (at least 4 planes each)
    // with the fewest staged planes per slot, the smaller one on ties.
    const int64_t slots = (int64_t)nsm * per_sm;
    const int64_t max_nzc = std::max<int64_t>(1, NZ / 4);
    int64_t best_cost = INT64_MAX;
    if (nzc < 0)  // one wave: as many chunks as fill every slot once
      best_cost = 0, nzc = (int)std::min<int64_t>(std::max<int64_t>(1, slots / ntiles), max_nzc);
    for (int64_t c = 1; c <= max_nzc && best_cost > 0; ++c) {
      const int64_t zl = (NZ + c - 1) / c;
      const int64_t n = (NZ + zl - 1) / zl;  // chunks actually formed
      const int64_t waves = (ntiles * n + slots - 1) / slots;
      const int64_t cost = waves * (zl + 2);
      if (cost < best_cost) {
        best_cost = cost;
        nzc = (int)n;
      }
    }
  }
  nzc = (int)std::min<int64_t>(std::max(nzc, 1), NZ);
  p->zlen = (int)((NZ + nzc - 1) / nzc);
  p->nzc = (int)((NZ + p->zlen - 1) / p->zlen);
  p->items = ntiles * p->nzc;
  return cudaSuccess;
}

int fused_item_of(const FusedPlan &p, int64_t x, int64_t y, int64_t z) {
  const int tx = (int)(x / p.bx), ty = (int)(y / p.by), zc = (int)(z / p.zlen);
  return (zc * p.tiles_y + ty) * p.tiles_x + tx;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn get_encode() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void *ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
  }
  return fn;
}

CUresult fused_encode_maps(int lat, int st, const FusedPlan &p, const void *base, int64_t NX,
                           int64_t NY, int64_t NZ, int64_t px, FusedMaps *tm) {
  EncodeTiledFn enc = get_encode();
  if (!enc) return CUDA_ERROR_NOT_FOUND;
  const int Q = lat == D3Q19 ? 19 : 9;
  const size_t sz = storage_bytes(st);
  CUtensorMapDataType dt = st == ST_F64   ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64
                           : st == ST_F32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                           : st == ST_F16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16
                                          : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  cuuint64_t dims[4] = {(cuuint64_t)NX, (cuuint64_t)NY, (cuuint64_t)NZ, (cuuint64_t)Q};
  cuuint64_t strides[3] = {(cuuint64_t)(px * sz), (cuuint64_t)(px * NY * sz),
                           (cuuint64_t)(px * NY * NZ * sz)};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  const cuuint32_t bx = p.bx, by = p.by, hx = p.hx, q = Q;
  const cuuint32_t boxes[4][4] = {{bx, by, 1, q}, {hx, by, 1, q}, {bx, 1, 1, q}, {hx, 1, 1, q}};
  CUtensorMap *maps[4] = {&tm->main, &tm->col, &tm->row, &tm->crn};
  for (int m = 0; m < 4; ++m) {
    CUresult r = enc(maps[m], dt, 4, const_cast<void *>(base), dims, strides, boxes[m], estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return r;
  }
  return CUDA_SUCCESS;
}

cudaError_t fused_launch(int lat, int st, const FusedPlan &p, const StepArgs &a,
                         const FusedMaps &tm, cudaStream_t s) {
  if (p.xc == 2) {
    switch (st) {
      case ST_F32: return fused_x2_launch_f32(lat, p, a, tm, s);
      case ST_F16: return fused_x2_launch_f16(lat, p, a, tm, s);
      case ST_BF16: return fused_x2_launch_bf16(lat, p, a, tm, s);
      case ST_F16R:
      case ST_BF16R: return fused_x2_launch_h16r(lat, st, p, a, tm, s);
      default: return cudaErrorInvalidValue;
    }
  }
  switch (st) {
    case ST_F64:
      return fused_launch_f64(lat, p, a, tm, s);
    case ST_F32:
      return fused_launch_f32(lat, p, a, tm, s);
    case ST_F16R:
    case ST_BF16R:
      return fused_launch_h16r(lat, st, p, a, tm, s);
    default:
      return fused_launch_h16(lat, st, p, a, tm, s);
  }
}

cudaError_t fused_prepare(int lat, int st, const FusedPlan &p, int *blocks_per_sm) {
  if (p.xc == 2) {
    switch (st) {
      case ST_F32: return fused_x2_prepare_f32(lat, p, blocks_per_sm);
      case ST_F16: return fused_x2_prepare_f16(lat, p, blocks_per_sm);
      case ST_BF16: return fused_x2_prepare_bf16(lat, p, blocks_per_sm);
      case ST_F16R:
      case ST_BF16R: return fused_x2_prepare_h16r(lat, st, p, blocks_per_sm);
      default: return cudaErrorInvalidValue;
    }
  }
  switch (st) {
    case ST_F64:
      return fused_prepare_f64(lat, p, blocks_per_sm);
    case ST_F32:
      return fused_prepare_f32(lat, p, blocks_per_sm);
    case ST_F16R:
    case ST_BF16R:
      return fused_prepare_h16r(lat, st, p, blocks_per_sm);
    default:
      return fused_prepare_h16(lat, st, p, blocks_per_sm);
  }
}

}  // namespace sclbm
