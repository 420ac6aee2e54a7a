// rk_cells.cuh -- the direct sums of rk_direct.cuh on small 3D boxes, a block of threads per
// block of nodes.
//
// Where a box has few nodes, walks along z (k_direct, k_regular) leave most SMs idle or spend
// their steps on the halo planes, and each step costs a chain of latencies.  Here a block
// takes bx x by x bz nodes (4 or 8 along each axis) with their halo at once, and the sums of
// an axis are one phase over all of them:
//   k_cell_sums     D_p by the forward sums along x, y and z, then g_p (K), u (Alg. 3), or
//                   the sum of both kinds of g_p that M + dt K spreads
//   k_cell_spread   the reflected sums of g_p along z, y and x: K (g_p of k_cell_sums,
//                   passed through memory that stays in L2) or Alg. 4 (g_p = b0_p y)
// Bounded by the FP64 pipe in FP64 (2 multiply-adds per cycle and SM), by latency below 48^3
// in FP32 and by instruction issue above.  FP64 48^3, linear basis, r = 1: K 16.4 + 12.0 us
// (k_direct 112 us), u^h 12.5 us (60), its transpose 15 us (46).
#pragma once

#include "rk_direct.cuh"

namespace rk {

// (against 128 threads: K at 96^3, FP32, r = 2, 44 against 50 us; FP64 64^3, r = 1, 52 / 59;
// u^h transposed on spheres in 144^3, quadratic basis, 675 / 877 us)
constexpr int kBlockThreads = 256;

// offsets of the nodes first .. first + w - 1 of an axis, continued periodically
RK_DEV void axis_offsets(long long* o, int first, int w, int n, long long stride) {
  for (int i = threadIdx.x; i < w; i += kBlockThreads) o[i] = stride * wrap_idx(first + i, n);
}

struct NodeBlock {
  int x0, y0, z0, nx, ny, nz;
};
template <typename T>
RK_DEV NodeBlock node_block(const DirectArgs<T>& a) {
  NodeBlock b;
  b.x0 = blockIdx.x * a.bx;
  b.y0 = blockIdx.y * a.by;
  b.z0 = blockIdx.z * a.bz;
  b.nx = min(a.bx, a.nx - b.x0);
  b.ny = min(a.by, a.ny - b.y0);
  b.nz = min(a.bz, a.nz - b.z0);
  return b;
}
// class of the cell that holds the block
template <typename T>
RK_DEV int block_class(const DirectArgs<T>& a, const NodeBlock& b) {
  const int cx = (a.nx + kCell - 1) / kCell, cy = (a.ny + kCell - 1) / kCell;
  return a.cls[b.x0 / kCell + cx * (b.y0 / kCell + (long long)cy * (b.z0 / kCell))];
}

// Shared memory (values of T) of a block of bx x by x bz nodes.
template <int S, int R>
struct CellSmem {
  using B = DBasis<S>;
  static constexpr RK_HD long long sums(int bx, int by, int bz) {
    const long long wx = bx + 2 * R, wy = by + 2 * R, wz = bz + 2 * R;
    const long long d = wx * wy * wz, e = (long long)B::NG * bx * by * wz;
    return (d > e ? d : e) + B::NX * bx * wy * wz;
  }
  static constexpr RK_HD long long spread(int bx, int by, int bz) {
    const long long wx = bx + 2 * R, wy = by + 2 * R, wz = bz + 2 * R;
    return S * wx * wy * wz + B::NG * wx * wy * bz;  // F takes the place of g
  }
};

// Where every node is regular b^0 is a constant of the even basis functions alone, and the
// sums of u = sum_p b0_p D_p (and of its transpose) collapse: with the quadratic basis two
// sums along x, three along y and two along z instead of 3, 6 and 10, with the linear one a
// single sum per axis.
template <typename T, int R>
RK_DEV T even_conv(int m, const T* in, int step, const T (*tab)[kDirectMaxReach + 1]) {
  T v[2 * R + 1];
#pragma unroll
  for (int j = 0; j <= 2 * R; ++j) v[j] = in[j * step];
  return conv1_m<R, 1>(m, v, R, tab);
}

template <typename T, int S, int R, int MODE, bool CG>
__global__ void __launch_bounds__(kBlockThreads) k_cell_sums(const __grid_constant__ DirectArgs<T> a) {
  using B = DBasis<S>;
  constexpr int W = kCell + 2 * R, CP = MODE == DM_EVAL_U ? S : ctab_pitch<T>(S);
  constexpr bool MASS = MODE == DM_MASS_STIFF;
  RK_DYN_SMEM(T, sm);
  __shared__ long long ox[W], oy[W], oz[W];
  const NodeBlock b = node_block(a);
  const int nx = b.nx, ny = b.ny, nz = b.nz;
  const int wx = nx + 2 * R, wy = ny + 2 * R, wz = nz + 2 * R;
  const unsigned rnx = box_inv(nx), rny = box_inv(ny), rwx = box_inv(wx), rwy = box_inv(wy);
  const long long ps = (long long)a.nx * a.ny;
  T* p_new = nullptr;
  const T* p_old = nullptr;
  T beta = (T)0;
  auto node = [&](int e) -> long long {  // of the block
    const int t = box_div(e, rnx), x = e - t * nx, z = box_div(t, rny), y = t - z * ny;
    return b.x0 + x + (long long)a.nx * (b.y0 + y) + ps * (b.z0 + z);
  };
  axis_offsets(ox, b.x0 - R, wx, a.nx, 1);
  axis_offsets(oy, b.y0 - R, wy, a.ny, a.nx);
  axis_offsets(oz, b.z0 - R, wz, a.nz, ps);
  const int cls = block_class(a, b);
  grid_wait();
  grid_trigger();
  if constexpr (CG) {
    const int par = a.cg->par;
    p_old = par ? a.p1 : a.p0;
    p_new = par ? a.p0 : a.p1;
    beta = (T)a.cg->beta;
  }
  if (cls == kCellZero) {  // (its g_p stay zero from the start)
    for (int e = threadIdx.x; e < nx * ny * nz; e += kBlockThreads) {
      if constexpr (CG) p_new[node(e)] = (T)0;
      if constexpr (MODE == DM_EVAL_U) a.out[node(e)] = (T)0;
    }
    return;
  }
  // the class and coefficients of a thread's first node are on their way during the sums
  int cl = -1;
  T co[CP], b0[MASS ? S : 1];
  auto load_node = [&](int e) {
    if (e >= nx * ny * nz) return;
    const long long i = node(e);
    cl = __ldg(a.cidx + i);
    if (cl <= 0) return;
    if constexpr (MASS) {
#pragma unroll
      for (int p = 0; p < S; ++p) b0[p] = __ldg(a.b0 + (long long)p * a.nbox + i);
    }
    if constexpr (MODE != DM_EVAL_U) {
      const Vec16<T>* src = reinterpret_cast<const Vec16<T>*>(a.ctab + (long long)(cl - 1) * CP);
#pragma unroll
      for (int k = 0; k < CP / (16 / (int)sizeof(T)); ++k) {
        const Vec16<T> raw = __ldg(src + k);
        memcpy(co + k * (16 / (int)sizeof(T)), &raw, 16);
      }
    } else {
#pragma unroll
      for (int p = 0; p < S; ++p) co[p] = __ldg(a.b0 + (long long)p * a.nbox + i);
    }
  };
  __syncthreads();
  const int nd = wx * wy * wz, ne = B::NG * nx * ny * wz;
  T *d = sm, *E = sm, *am = sm + (nd > ne ? nd : ne);  // E takes the place of d
#pragma unroll 4
  for (int e = threadIdx.x; e < nd; e += kBlockThreads) {
    const int t = box_div(e, rwx), x = e - t * wx, z = box_div(t, rwy), y = t - z * wy;
    const long long i = ox[x] + oy[y] + oz[z];
    T v;
    if constexpr (CG) {
      v = a.in[i] + beta * p_old[i];  // (not __ldg: the update that writes r may overlap this kernel)
      if ((unsigned)(x - R) < (unsigned)nx && (unsigned)(y - R) < (unsigned)ny && (unsigned)(z - R) < (unsigned)nz) p_new[i] = v;
    } else {
      v = __ldg(a.in + i);
      if (a.in_bits && !(__ldg(a.flags + i) & a.in_bits)) v = (T)0;
    }
    d[e] = v;
  }
  const int na = nx * wy * wz;
  if constexpr (MODE == DM_EVAL_U) {
    bool reg = a.diag0 != 0;
    for (int e = threadIdx.x; e < nx * ny * nz; e += kBlockThreads) reg = __ldg(a.cidx + node(e)) == 0 && reg;
    if (__syncthreads_and(reg)) {
      for (int e = threadIdx.x; e < na; e += kBlockThreads) {
        const int t = box_div(e, rnx), x = e - t * nx;
        T v[2 * R + 1];
#pragma unroll
        for (int j = 0; j <= 2 * R; ++j) v[j] = d[t * wx + x + j];
        am[e] = conv1<0, R, 1>(v, R, a.tab);
        if constexpr (S == 10) am[na + e] = conv1<2, R, 1>(v, R, a.tab);
      }
      __syncthreads();
      const int nxy = nx * ny, nE = nxy * wz;
      for (int e = threadIdx.x; e < nE; e += kBlockThreads) {
        const int t = box_div(e, rnx), x = e - t * nx, z = box_div(t, rny), y = t - z * ny;
        const T* c = am + x + nx * (y + wy * z);
        const T e0 = even_conv<T, R>(0, c, nx, a.tab);
        if constexpr (S == 10) {
          E[e] = a.b0reg[0] * e0 + a.b0reg[4] * even_conv<T, R>(0, c + na, nx, a.tab) + a.b0reg[7] * even_conv<T, R>(2, c, nx, a.tab);
          E[nE + e] = a.b0reg[9] * e0;
        } else {
          E[e] = a.b0reg[0] * e0;
        }
      }
      __syncthreads();
      for (int e = threadIdx.x; e < nxy * nz; e += kBlockThreads) {
        T u = even_conv<T, R>(0, E + e, nxy, a.tab);
        if constexpr (S == 10) u += even_conv<T, R>(2, E + nE + e, nxy, a.tab);
        a.out[node(e)] = u;
      }
      return;
    }
  }
  load_node(threadIdx.x);
  __syncthreads();
  for (int e = threadIdx.x; e < na; e += kBlockThreads) {
    const int t = box_div(e, rnx), x = e - t * nx;  // t = y + wy z
    T v[2 * R + 1];
#pragma unroll
    for (int j = 0; j <= 2 * R; ++j) v[j] = d[t * wx + x + j];
#pragma unroll
    for (int m = 0; m < B::NX; ++m) am[m * na + e] = conv1_m<R, 1>(m, v, R, a.tab);
  }
  __syncthreads();
  const int nxy = nx * ny, nE = nxy * wz;
  for (int e = threadIdx.x; e < nE; e += kBlockThreads) {
    const int t = box_div(e, rnx), x = e - t * nx, z = box_div(t, rny), y = t - z * ny;
#pragma unroll
    for (int m = 0; m < B::NX; ++m) {
      T v[2 * R + 1];
#pragma unroll
      for (int j = 0; j <= 2 * R; ++j) v[j] = am[m * na + x + nx * (y + j + wy * z)];
#pragma unroll
      for (int g = 0; g < B::NG; ++g)
        if (B::gmx(g) == m) E[g * nE + e] = conv1_m<R, 1>(B::gmy(g), v, R, a.tab);
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < nxy * nz; e += kBlockThreads) {
    if (e != (int)threadIdx.x) load_node(e);
    const long long i = node(e);
    T D[S];
#pragma unroll
    for (int gr = 0; gr < B::NG; ++gr) {
      T v[2 * R + 1];
#pragma unroll
      for (int j = 0; j <= 2 * R; ++j) v[j] = E[gr * nE + e + j * nxy];
#pragma unroll
      for (int p = 0; p < S; ++p)
        if (B::grp(p) == gr) D[p] = conv1_m<R, 1>(B::az(p), v, R, a.tab);
    }
    if constexpr (MODE != DM_EVAL_U) {
      T g[S];
      if (cl == 0 && a.diag) {
#pragma unroll
        for (int p = 0; p < S; ++p) g[p] = p >= 1 && p <= 3 ? a.creg[p - 1] * D[p] : (T)0;
      } else if (cl >= 0) {
        if (cl == 0) {
#pragma unroll
          for (int k = 0; k < 3 * S + 1; ++k) co[k] = a.breg[k];
        }
        pointwise_node<T, S>(co, cl, D, g);
      } else {
#pragma unroll
        for (int p = 0; p < S; ++p) g[p] = (T)0;
      }
      if constexpr (MASS) {
        // dt g_p + chi V b0_p u, u = sum_q b0_q D_q: one reflected sum for M and K
        const T w = cl > 0 ? co[3 * S] : a.vreg;
        T u = (T)0;
#pragma unroll
        for (int p = 0; p < S; ++p) u += (cl > 0 ? b0[p] : a.b0reg[p]) * D[p];
        u = cl >= 0 ? w * u : (T)0;
#pragma unroll
        for (int p = 0; p < S; ++p) g[p] = a.dt * g[p] + (cl > 0 ? b0[p] : a.b0reg[p]) * u;
      }
#pragma unroll
      for (int p = 0; p < S; ++p) a.gall[p * a.nbox + i] = g[p];
    } else {
      T u = (T)0;
      if (cl > 0) {
#pragma unroll
        for (int p = 0; p < S; ++p) u += co[p] * D[p];
      } else if (cl == 0) {
#pragma unroll
        for (int p = 0; p < S; ++p)
          if (!a.diag0 || even_p<S>(p)) u += a.b0reg[p] * D[p];
      }
      a.out[i] = u;
    }
  }
}

template <typename T, int S, int R, int MODE, bool CG>
__global__ void __launch_bounds__(kBlockThreads) k_cell_spread(const __grid_constant__ DirectArgs<T> a) {
  using B = DBasis<S>;
  constexpr int W = kCell + 2 * R;
  RK_DYN_SMEM(T, sm);
  __shared__ long long ox[W], oy[W], oz[W];
  const NodeBlock b = node_block(a);
  const int nx = b.nx, ny = b.ny, nz = b.nz;
  const int wx = nx + 2 * R, wy = ny + 2 * R, wz = nz + 2 * R;
  const unsigned rnx = box_inv(nx), rny = box_inv(ny), rwx = box_inv(wx), rwy = box_inv(wy);
  const long long ps = (long long)a.nx * a.ny;
  auto node = [&](int e) -> long long {
    const int t = box_div(e, rnx), x = e - t * nx, z = box_div(t, rny), y = t - z * ny;
    return b.x0 + x + (long long)a.nx * (b.y0 + y) + ps * (b.z0 + z);
  };
  axis_offsets(ox, b.x0 - R, wx, a.nx, 1);
  axis_offsets(oy, b.y0 - R, wy, a.ny, a.nx);
  axis_offsets(oz, b.z0 - R, wz, a.nz, ps);
  const int cls = block_class(a, b);
  grid_wait();
  grid_trigger();
  if (cls == kCellZero) {
    for (int e = threadIdx.x; e < nx * ny * nz; e += kBlockThreads) a.out[node(e)] = (T)0;
    if constexpr (CG) direct_pap_reduce<kBlockThreads>(DotAccPair<T>(), a);
    return;
  }
  __syncthreads();
  const int wxy = wx * wy, wn = wxy * wz, nG = wxy * nz, nF = wx * ny * nz;
  T *g = sm, *F = sm, *G = sm + S * wn;
  if constexpr (MODE == DM_STIFF) {
#pragma unroll 2
    for (int e = threadIdx.x; e < wn; e += kBlockThreads) {
      const int t = box_div(e, rwx), x = e - t * wx, z = box_div(t, rwy), y = t - z * wy;
      const long long i = ox[x] + oy[y] + oz[z];
#pragma unroll
      for (int p = 0; p < S; ++p) cp_async_value(g + p * wn + e, a.gall + p * a.nbox + i);
    }
    cp_async_commit();
    cp_async_wait<0>();
  } else {
    // Alg. 4: g_p = b0_p y.  Outside chi M is the identity: b0 = (1, 0, ...).
    int* C = reinterpret_cast<int*>(G);  // classes, until the z sums
    bool reg = a.diag0 != 0;
#pragma unroll 4
    for (int e = threadIdx.x; e < wn; e += kBlockThreads) {
      const int t = box_div(e, rwx), x = e - t * wx, z = box_div(t, rwy), y = t - z * wy;
      const long long i = ox[x] + oy[y] + oz[z];
      const int cl = __ldg(a.cidx + i);
      T v = __ldg(a.in + i);
      if (a.wfield) v *= __ldg(a.wfield + i);
      if (a.in_bits && !(__ldg(a.flags + i) & a.in_bits)) v = (T)0;
      g[e] = v;
      C[e] = cl;
      reg = cl == 0 && reg;
    }
    if (__syncthreads_and(reg)) {
      [[maybe_unused]] T *G2 = G + nG, *F2 = F + nF;  // (F takes the place of y, which the y sums no longer read)
      for (int e = threadIdx.x; e < nG; e += kBlockThreads) {
        const T c = even_conv<T, R>(0, g + e, wxy, a.tab);
        if constexpr (S == 10) {
          G[e] = a.b0reg[0] * c + a.b0reg[9] * even_conv<T, R>(2, g + e, wxy, a.tab);
          G2[e] = c;
        } else {
          G[e] = a.b0reg[0] * c;
        }
      }
      __syncthreads();
      for (int e = threadIdx.x; e < nF; e += kBlockThreads) {
        const int t = box_div(e, rwx), x = e - t * wx, z = box_div(t, rny), y = t - z * ny;
        const int o = x + wx * (y + wy * z);
        T f = even_conv<T, R>(0, G + o, wx, a.tab);
        if constexpr (S == 10) {
          f += a.b0reg[7] * even_conv<T, R>(2, G2 + o, wx, a.tab);
          F2[e] = a.b0reg[4] * even_conv<T, R>(0, G2 + o, wx, a.tab);
        }
        F[e] = f;
      }
      __syncthreads();
      for (int e = threadIdx.x; e < nx * ny * nz; e += kBlockThreads) {
        const int t = box_div(e, rnx), x = e - t * nx;
        const long long i = node(e);
        T w = even_conv<T, R>(0, F + x + wx * t, 1, a.tab);
        if constexpr (S == 10) w += even_conv<T, R>(2, F2 + x + wx * t, 1, a.tab);
        a.out[i] = __ldg(a.flags + i) & a.out_bits ? w : (T)0;
      }
      return;
    }
    for (int e = threadIdx.x; e < wn; e += kBlockThreads) {
      const int t = box_div(e, rwx), x = e - t * wx, z = box_div(t, rwy), y = t - z * wy;
      const long long i = ox[x] + oy[y] + oz[z];
      const int cl = C[e];
      const T v = g[e];
#pragma unroll
      for (int p = 0; p < S; ++p) {
        const T b0 = cl > 0 ? __ldg(a.b0 + p * a.nbox + i) : (cl == 0 ? a.b0reg[p] : (p == 0 ? (T)1 : (T)0));
        g[p * wn + e] = cl == 0 && a.diag0 && !even_p<S>(p) ? (T)0 : b0 * v;
      }
    }
  }
  __syncthreads();
  // z: G(z) += T(o) g(z + o)
  for (int e = threadIdx.x; e < nG; e += kBlockThreads) {
    T s[B::NG];
#pragma unroll
    for (int p = 0; p < S; ++p) {
      T v[2 * R + 1];
#pragma unroll
      for (int j = 0; j <= 2 * R; ++j) v[j] = g[p * wn + e + j * wxy];
      const T w = conv1_m<R, -1>(B::az(p), v, R, a.tab);
      s[B::grp(p)] = B::az(p) == 0 ? w : s[B::grp(p)] + w;  // (m_x, m_y, 0) comes first
    }
#pragma unroll
    for (int k = 0; k < B::NG; ++k) G[k * nG + e] = s[k];
  }
  __syncthreads();
  for (int e = threadIdx.x; e < nF; e += kBlockThreads) {
    const int t = box_div(e, rwx), x = e - t * wx, z = box_div(t, rny), y = t - z * ny;
    T acc[B::NX];
#pragma unroll
    for (int k = 0; k < B::NG; ++k) {
      T v[2 * R + 1];
#pragma unroll
      for (int j = 0; j <= 2 * R; ++j) v[j] = G[k * nG + x + wx * (y + j + wy * z)];
      const T w = conv1_m<R, -1>(B::gmy(k), v, R, a.tab);
      acc[B::gmx(k)] = B::gmy(k) == 0 ? w : acc[B::gmx(k)] + w;
    }
#pragma unroll
    for (int m = 0; m < B::NX; ++m) F[m * nF + e] = acc[m];
  }
  __syncthreads();
  [[maybe_unused]] DotAccPair<T> dot;
  [[maybe_unused]] const T* p = nullptr;
  if constexpr (CG) p = a.cg->par ? a.p0 : a.p1;
  for (int e = threadIdx.x; e < nx * ny * nz; e += kBlockThreads) {
    const int t = box_div(e, rnx), x = e - t * nx;
    const long long i = node(e);
    T acc = (T)0;
    if (__ldg(a.flags + i) & a.out_bits) {
#pragma unroll
      for (int m = 0; m < B::NX; ++m) {
        T v[2 * R + 1];
#pragma unroll
        for (int j = 0; j <= 2 * R; ++j) v[j] = F[m * nF + x + j + wx * t];
        const T w = conv1_m<R, -1>(m, v, R, a.tab);
        acc = m == 0 ? w : acc + w;
      }
    }
    a.out[i] = acc;
    if constexpr (CG) dot.add(cmk(p[i], (T)0), cmk(acc, (T)0));
  }
  if constexpr (CG) direct_pap_reduce<kBlockThreads>(dot, a);
}

}  // namespace rk
