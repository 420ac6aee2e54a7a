// rk_direct_launch.cuh -- the choice between the operators by direct sums (rk_direct.cuh,
// rk_cells.cuh) and their launch configurations; one translation unit per precision, degree and reach
// (rk_direct_<type>_<degree>_<reach>.cu) instantiates direct_sr.
#pragma once

#include <algorithm>
#include <cmath>

#include "rk_cells.cuh"
#include "rk_direct.cuh"
#include "rk_internal.cuh"

namespace rk {

constexpr int kSMs = 152;

// How a launch is cut: the tile and the planes per block.
struct DirectPlan {
  bool small_tile;
  int zc, tiles_x, tiles_y;
  long long blocks;
  double cost;
  int steps, occ;   // steps of a block, blocks that an SM holds
  double lat, col;  // cycles of a step: its latency, its issue time
};

// Cost of a launch in SM cycles: every block walks its planes plus those of its halo, an SM
// runs `occ` blocks at a time, a step of a block takes at least the latency of its chain of
// stages (lat), and its columns take issue time (col cycles each: FP64 multiply-adds issue
// at 2 per cycle and SM).  Both are fits to the measured times of boxes of 16^3 to 256^3.
// A block's planes lie in one cell or are whole cells (twos: powers of two).
template <int TX, int TY>
inline DirectPlan walk_plan(bool small_tile, int nx, int ny, int nz, int zmin, int halo, int occ, double lat, double col,
                            bool twos = false) {
  DirectPlan best{small_tile, 0, (nx + TX - 1) / TX, (ny + TY - 1) / TY, 0, 0.0, 0, occ, lat, col};
  const long long tiles = (long long)best.tiles_x * best.tiles_y;
  for (int zc = zmin; zc <= 256; zc += twos || zc < kCell ? zc : kCell) {
    const int c = std::min(zc, nz);
    const long long blocks = tiles * ((nz + c - 1) / c);
    const int steps = c + halo;
    const long long per_sm = (blocks + kSMs - 1) / kSMs;
    const long long waves = (per_sm + occ - 1) / occ;
    const double t = std::max((double)waves * steps * lat, (double)per_sm * steps * col);
    if (best.blocks == 0 || t < best.cost) {
      best.zc = c;
      best.blocks = blocks;
      best.cost = t;
      best.steps = steps;
    }
    if (c == nz) break;
  }
  return best;
}

// Times in microseconds, for the choice between direct sums and transform passes.  The costs
// above order the ways to the direct sums; these are fits to measured calls (boxes of 36^3 to
// 256^3, cubic and not, a cube or spheres in them; 10 % off at most places): the walk of a plan
// with its empty cells left out (their blocks end at once; the others hold some of them), times
// and plus what the fits give per kernel.  K with r <= 2 in FP64 and every u^h were faster than
// the passes on all of these boxes (0.2 to 0.95 times) and are not estimated, nor is K in FP32
// outside CG.
inline double walk_us(const DirectPlan& p, double active) {
  const double per_sm = (double)((p.blocks + kSMs - 1) / kSMs) * std::sqrt(active);
  return std::max(std::max(1.0, per_sm / p.occ) * p.steps * p.lat, per_sm * p.steps * p.col) / 2000.0;
}
// a CG step in FP32 by k_direct (the longer walks of the quadratic basis gain more from empty cells)
template <int S, int R>
double direct_cg_us(const DirectPlan& p, double share) {
  const double active = S == 4 ? share : std::pow(share, 1.4);
  const double k = R <= 2 ? (S == 4 ? 1.35 : 1.1) : (R == 3 ? 2.0 : (S == 4 ? 1.16 : 2.25));
  return (R <= 2 ? 5.0 : 0.0) + k * walk_us(p, active);
}
template <typename T, int S, int R>
double regular_us(const DirectPlan& q, double active, int ncells, int ocells) {
  if constexpr (sizeof(T) == 8) {
    // (few cells leave as many long blocks: the 0.3rd power of their share)
    const double cells = (ncells + ocells) / (2.0 * kSMs), w = walk_us(q, std::pow(active, 0.6));
    if (R == 3) return S == 4 ? 154.0 + 1.45 * w + 11.6 * cells : 115.0 + w + 67.0 * cells;
    if (R == 4) return S == 4 ? 94.0 + 0.89 * w + 76.0 * cells : 85.0 + 0.82 * w + 131.0 * cells;
  }
  return 0.0;
}

// The regular stencil: cycles per step of a tile (its columns) and its latency.  Measured at
// r = 2: FP32 a step of 32 x 16 columns takes 1080 cycles alone on an SM and 700 of two; of
// 32 x 8 columns 900 and 540.  FP64: 30 cycles per column of a 32 x 32 tile, 40 of a 32 x 8
// one (the halo of the x sums).  The smaller tile wins where blocks are few: at 32^3 and 64^3
// in FP32 7.5 and 9.9 us against 8.5 and 10.6 us, at 128^3 26 against 22 us; in FP64 at 64^3
// 90 against 180 us, at 128^3 394 against 427 us.  FP32 with r = 4: 32 x 32 and 32 x 16
// columns, at r = 4 on a 256^3 cube 184 against 260 us, on 162 x 100 x 144 77 against 69 us.
template <typename T, int R>
inline DirectPlan regular_plan(int nx, int ny, int nz) {
  using DB = RTile<T, R, false>;
  using DS = RTile<T, R, true>;
  constexpr bool F64 = sizeof(T) == 8;
  const double h = DB::H / 4.0;
  const double cb = F64 ? 6.5 + 23.5 * h : 0.55 + 0.82 * h, cs = F64 ? 8.0 + 32.0 * h : 1.0 + 1.1 * h;
  const DirectPlan b = walk_plan<DB::TX, DB::TY>(false, nx, ny, nz, 2, 2 * DB::H + 1, DB::MINB, F64 ? 2100.0 : 1080.0, DB::TX * DB::TY * cb);
  const DirectPlan q = walk_plan<DS::TX, DS::TY>(true, nx, ny, nz, 2, 2 * DS::H + 1, DS::MINB, F64 ? 1450.0 : 900.0, DS::TX * DS::TY * cs);
  return q.cost < b.cost ? q : b;
}

template <typename T, int S, int R, int MODE>
DirectPlan direct_plan_mode(int nx, int ny, int nz) {
  using DB = DTile<T, S, R, MODE, false>;
  const double lat = sizeof(T) == 8 ? 2500.0 : 2300.0, col = (sizeof(T) == 8 ? 60.0 : 4.2) * DB::B::NG / 3.0;
  DirectPlan p = walk_plan<DB::TX, DB::TY>(false, nx, ny, nz, 1, 2 * DB::ZF + 2 * DB::ZO + 3, DB::MINB, lat, DB::GX * DB::GY * col, true);
  if constexpr (DB::B::DIM == 3) {
    using DS = DTile<T, S, R, MODE, true>;
    const DirectPlan q = walk_plan<DS::TX, DS::TY>(true, nx, ny, nz, 1, 2 * DS::ZF + 2 * DS::ZO + 3, DS::MINB, lat, DS::GX * DS::GY * col, true);
    if (q.cost < p.cost) p = q;
  }
  return p;
}

template <typename T, int S, int R, int MODE, bool SMALL, bool CG>
cudaError_t direct_launch(const DirectArgs<T>& a0, const DirectPlan& p, cudaStream_t s) {
  using D = DTile<T, S, R, MODE, SMALL>;
  auto kernel = k_direct<T, S, R, MODE, SMALL, CG>;
  const size_t smem = D::smem(CG);
  if (smem > 32 * 1024) {  // static and dynamic shared memory above 48 KB need the opt-in
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  DirectArgs<T> a = a0;
  a.tiles_x = p.tiles_x;
  a.tiles_y = p.tiles_y;
  a.zc = p.zc;
  count_launch();
  kernel<<<(unsigned)p.blocks, D::THREADS, smem, s>>>(a);
  return cudaGetLastError();
}

template <typename T, int R, bool SMALL, bool CG>
cudaError_t regular_launch(const DirectArgs<T>& a0, const DirectPlan& p, cudaStream_t s) {
  using D = RTile<T, R, SMALL>;
  auto kernel = k_regular<T, R, SMALL, CG>;
  const size_t smem = D::smem(CG);
  if (smem > 32 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  DirectArgs<T> a = a0;
  a.tiles_x = p.tiles_x;
  a.tiles_y = p.tiles_y;
  a.zc = p.zc;
  return launch_after(CG && a.after, kernel, dim3((unsigned)p.blocks), D::THREADS, smem, s, a);
}

// Blocks of k_correct in a CG step: a few per SM, so that few meet at the counter (128^3
// mixed solve 27.4 against 28.8 ms with one per cell, 96^3 adjoint 55.6 / 58.6 ms).
inline int correct_blocks(bool cg, int ocells) { return cg ? std::min(ocells, 5 * kSMs) : ocells; }

template <typename T, int S, int R, bool CG>
cudaError_t correct_launch(const DirectArgs<T>& a, cudaStream_t s) {
  auto k1 = k_delta<T, S, R, CG>;
  auto k2 = k_correct<T, S, R, CG>;
  constexpr size_t s1 = DeltaSize<T, S, R>::SMEM, s2 = CorrectSize<T, S, R>::SMEM;
  cudaError_t e = cudaSuccess;
  if (s1 > 32 * 1024) e = cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)s1);
  if (s2 > 32 * 1024 && e == cudaSuccess) e = cudaFuncSetAttribute(k2, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)s2);
  if (e != cudaSuccess) return e;
  if ((e = launch_after(a.after != 0, k1, dim3((unsigned)a.ncells), corr_threads<R>(), s1, s, a)) != cudaSuccess) return e;
  return launch_after(a.after != 0, k2, dim3((unsigned)correct_blocks(CG, a.ocells)), corr_threads<R>(), s2, s, a);
}

// The operators by blocks of nodes (rk_cells.cuh).  Cost in SM cycles as above: a kernel takes
// c0 however small, and each of an SM's blocks its multiply-adds.  Blocks of 4 along an axis
// put a small box on more SMs, at the price of more halo.
struct CellPlan {
  int b[3] = {0, 0, 0};
  long long blocks = 0;
  double cost = 0.0;
};
template <typename T, int S, int R, int MODE>
CellPlan cell_plan(int nx, int ny, int nz) {
  using B = DBasis<S>;
  constexpr bool F64 = sizeof(T) == 8, FWD = MODE != DM_TRANSPOSE_U, REFL = MODE != DM_EVAL_U;
  const double c0 = 7000.0, c1 = F64 ? 0.55 : 0.09;
  CellPlan best;
  for (int t = 0; t < 8; ++t) {
    const int b[3] = {t & 4 ? 4 : 8, t & 2 ? 4 : 8, t & 1 ? 4 : 8};
    const long long smem = std::max(FWD ? CellSmem<S, R>::sums(b[0], b[1], b[2]) : 0, REFL ? CellSmem<S, R>::spread(b[0], b[1], b[2]) : 0) * (long long)sizeof(T);
    if (smem > 200 * 1024) continue;
    const double x = b[0], y = b[1], z = b[2], wx = x + 2 * R, wy = y + 2 * R, wz = z + 2 * R, L = 2 * R + 1;
    const double fwd = L * (B::NX * x * wy * wz + B::NG * x * y * wz + S * x * y * z) + 6.0 * S * x * y * z;
    const double refl = L * (S * wx * wy * z + B::NG * wx * y * z + B::NX * x * y * z);
    const long long nb = (long long)((nx + b[0] - 1) / b[0]) * ((ny + b[1] - 1) / b[1]) * ((nz + b[2] - 1) / b[2]);
    const double per_sm = (double)((nb + kSMs - 1) / kSMs);
    // (one block per SM waits out each of its latencies: transpose of u^h on spheres in 144^3,
    // quadratic basis, 8^3 nodes in 189 KB 543 us, 4 x 8 x 8 in 104 KB 494 us)
    const double alone = smem > 112 * 1024 ? 1.6 : 1.0;
    const double c = alone * ((FWD ? c0 + per_sm * c1 * fwd : 0.0) + (REFL ? c0 + per_sm * c1 * refl : 0.0));
    if (best.blocks == 0 || c < best.cost) {
      for (int k = 0; k < 3; ++k) best.b[k] = b[k];
      best.blocks = nb;
      best.cost = c;
    }
  }
  return best;
}

template <typename T, int S, int R, int MODE>
double cells_us(const CellPlan& c, double active) {
  constexpr bool F64 = sizeof(T) == 8;
  const double t = c.cost / 2000.0;
  if constexpr (MODE == DM_TRANSPOSE_U) {
    if (!F64 || R < 3 || (R == 3 && S == 4)) return 0.0;
    const double w = t * std::pow(active, 0.7);
    return R == 3 ? 52.0 + 0.67 * w : (S == 4 ? 25.0 + 0.94 * w : 70.0 + 0.72 * w);
  }
  if constexpr (MODE == DM_STIFF) return F64 ? (R >= 3 ? 20.0 + 1.02 * t * std::pow(active, 0.7) : 0.0) : (R >= 2 ? 8.0 + 0.72 * t * std::sqrt(active) : 0.0);
  return 0.0;
}

template <typename T, int S, int R, int MODE, bool CG>
cudaError_t cell_launch(const DirectArgs<T>& a0, const CellPlan& p, cudaStream_t s) {
  DirectArgs<T> a = a0;
  a.bx = p.b[0];
  a.by = p.b[1];
  a.bz = p.b[2];
  const dim3 grid((a.nx + a.bx - 1) / a.bx, (a.ny + a.by - 1) / a.by, (a.nz + a.bz - 1) / a.bz);
  cudaError_t e = cudaSuccess;
  if constexpr (MODE != DM_TRANSPOSE_U) {
    auto k = k_cell_sums<T, S, R, MODE, CG>;
    const size_t smem = sizeof(T) * (size_t)CellSmem<S, R>::sums(a.bx, a.by, a.bz);
    if (smem > 32 * 1024 && (e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
    if ((e = launch_after(CG && a.after, k, grid, kBlockThreads, smem, s, a)) != cudaSuccess) return e;
  }
  if constexpr (MODE != DM_EVAL_U) {
    auto k = k_cell_spread<T, S, R, MODE == DM_MASS_STIFF ? DM_STIFF : MODE, CG>;
    const size_t smem = sizeof(T) * (size_t)CellSmem<S, R>::spread(a.bx, a.by, a.bz);
    if (smem > 32 * 1024 && (e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
    if ((e = launch_after(MODE != DM_TRANSPOSE_U && a.after, k, grid, kBlockThreads, smem, s, a)) != cudaSuccess) return e;
  }
  return e;
}

// Three ways to an operator on a 3D box, by their estimated costs:
//   blocks of nodes       small boxes, where walks along z leave SMs idle.  K, linear basis,
//                         against the better of the others: FP64 r = 1, 16^3 9.2 against
//                         23.3 us, 48^3 28 / 54, 64^3 52 / 79, 96^3 157 / 149 us; r = 2, 32^3
//                         24 / 59, 48^3 51 / 106, 64^3 113 / 149, 96^3 304 / 287 us; FP32
//                         r = 2, 16^3 7.0 / 12.1, 48^3 13.9 / 17.4, 64^3 21 / 23.4, 96^3 44 / 36.
//                         u^h and its transpose on every box, against k_direct: FP64,
//                         linear, r = 1, 48^3 12 / 60 and 14 / 46 us, 96^3 45 / 361 and
//                         55 / 130 us; quadratic, r = 2, 48^3 22 / 78 and 26 / 111, spheres
//                         in 144^3 192 / 347 and 494 / 538 us
//   regular + corrections K on larger boxes with regular nodes (a.corrected): the corrections
//                         cost two launches and a cell's share of an SM
//   k_direct              every node on its own, walking along z: K on large boxes without
//                         regular nodes
template <typename T, int S, int R, int MODE, bool CG>
cudaError_t direct_mode(const DirectArgs<T>& a0, cudaStream_t s, DirectQuery* query) {
  DirectArgs<T> a = a0;
  a.part0 = 0;
  if constexpr (DBasis<S>::DIM == 3) {
    const CellPlan c = cell_plan<T, S, R, MODE>(a.nx, a.ny, a.nz);
    bool cells = true;
    if constexpr (MODE == DM_STIFF) {
      // (the fits miss k_direct by up to a third on the low side, the corrections by less)
      const double direct = 1.2 * direct_plan_mode<T, S, R, MODE>(a.nx, a.ny, a.nz).cost;
      const DirectPlan q = regular_plan<T, R>(a.nx, a.ny, a.nz);
      const bool corr = a.ncells > 0 && a.ocells > 0;
      const double ccost = 5e3 + (corr ? 22e3 + (a.ncells + a.ocells) / (2.0 * kSMs) * (sizeof(T) == 8 ? 4e3 + 15e3 * R : 4e3) * S / 4.0 : 0.0);
      // A CG step in FP32 takes the sums of T and of its transpose one after the other for
      // r >= 2: the stencil's rounded coefficients are no longer a product B^T B, and where the
      // smallest eigenvalues lie near the rounding (a = 2.5: T_0 nearly vanishes at the highest
      // frequencies) CG needs more steps.  a = 2.5, 256^3 cube, mixed solve to 1e-10: 1625
      // iterations, 1.31 s, against 6675, 2.5 s (128^3 2250 / 2950); r = 1: as many both ways.
      // On such large boxes the transform passes are faster still (1825 iterations, 1.00 s;
      // choose_routes weighs them).
      constexpr bool product = CG && sizeof(T) == 4 && R >= 2;
      const bool regular = !product && a.corrected && q.cost + ccost < direct;
      cells = (query ? query->fields : a.gall != nullptr) && c.cost < (regular ? q.cost + ccost : direct);
      if (regular && !cells) {
        a.parts = (unsigned)(q.blocks + (corr ? correct_blocks(CG, a.ocells) : 0));
        if (query) {
          query->fields = false;
          query->blocks = a.parts;
          query->us = regular_us<T, S, R>(q, query->active, corr ? a.ncells : 0, corr ? a.ocells : 0);
          return cudaSuccess;
        }
        cudaError_t e = q.small_tile ? regular_launch<T, R, true, CG>(a, q, s) : regular_launch<T, R, false, CG>(a, q, s);
        if (e != cudaSuccess || !corr) return e;
        a.part0 = (unsigned)q.blocks;
        return correct_launch<T, S, R, CG>(a, s);
      }
    }
    if (cells) {
      a.parts = (unsigned)c.blocks;
      if (query) {
        query->fields = true;
        query->blocks = a.parts;
        query->us = cells_us<T, S, R, MODE>(c, query->active);
        return cudaSuccess;
      }
      return cell_launch<T, S, R, MODE, CG>(a, c, s);
    }
  }
  if constexpr (DBasis<S>::DIM == 2 || MODE == DM_STIFF) {
    const DirectPlan p = direct_plan_mode<T, S, R, MODE>(a.nx, a.ny, a.nz);
    a.parts = (unsigned)p.blocks;
    if (query) {
      query->fields = false;
      query->blocks = p.blocks;
      query->us = CG && sizeof(T) == 4 && R >= 2 ? direct_cg_us<S, R>(p, query->active) : 0.0;
      return cudaSuccess;
    }
    if constexpr (DBasis<S>::DIM == 3) {
      if (p.small_tile) return direct_launch<T, S, R, MODE, true, CG>(a, p, s);
    }
    return direct_launch<T, S, R, MODE, false, CG>(a, p, s);
  }
  return cudaErrorInvalidValue;
}

template <typename T, int S, int R>
cudaError_t direct_s(int mode, const DirectArgs<T>& a, cudaStream_t s, DirectQuery* query) {
  switch (mode) {
    case DM_STIFF: return a.cg || (query && query->cg) ? direct_mode<T, S, R, DM_STIFF, true>(a, s, query) : direct_mode<T, S, R, DM_STIFF, false>(a, s, query);
    case DM_MASS_STIFF:
      if constexpr (DBasis<S>::DIM == 3 && sizeof(T) == 8) {
        if (!a.gall || !a.cg || query) return cudaErrorInvalidValue;
        DirectArgs<T> b = a;
        const CellPlan c = cell_plan<T, S, R, DM_STIFF>(a.nx, a.ny, a.nz);
        b.part0 = 0;
        b.parts = (unsigned)c.blocks;
        return cell_launch<T, S, R, DM_MASS_STIFF, true>(b, c, s);
      }
      return cudaErrorInvalidValue;
    case DM_EVAL_U: return direct_mode<T, S, R, DM_EVAL_U, false>(a, s, query);
    case DM_TRANSPOSE_U: return direct_mode<T, S, R, DM_TRANSPOSE_U, false>(a, s, query);
    default: return cudaErrorInvalidValue;
  }
}

// basis sizes of one degree: 3D (4, 10) and 2D (3, 6)
template <typename T, int DEG, int R>
cudaError_t direct_sr(int mode, int dim, const DirectArgs<T>& a, cudaStream_t s, DirectQuery* query) {
  if (dim == 3) return direct_s<T, DEG == 1 ? 4 : 10, R>(mode, a, s, query);
  return direct_s<T, DEG == 1 ? 3 : 6, R>(mode, a, s, query);
}

#define RK_DIRECT_EACH(X) \
  X(float, 1, 1) X(float, 1, 2) X(float, 1, 3) X(float, 1, 4) X(float, 2, 1) X(float, 2, 2) X(float, 2, 3) X(float, 2, 4) \
  X(double, 1, 1) X(double, 1, 2) X(double, 1, 3) X(double, 1, 4) X(double, 2, 1) X(double, 2, 2) X(double, 2, 3) X(double, 2, 4)
#define RK_DIRECT_DECLARE(T, DEG, R) \
  extern template cudaError_t direct_sr<T, DEG, R>(int, int, const DirectArgs<T>&, cudaStream_t, DirectQuery*);
#define RK_DIRECT_INSTANTIATE(T, DEG, R) \
  template cudaError_t direct_sr<T, DEG, R>(int, int, const DirectArgs<T>&, cudaStream_t, DirectQuery*);

}  // namespace rk
