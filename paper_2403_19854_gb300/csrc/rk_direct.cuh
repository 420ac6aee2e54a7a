// rk_direct.cuh -- the operators of Alg. 2-4 by direct sums, for supports of at most
// kDirectMaxReach nodes: k_direct (below), the regular stencil with its corrections
// (k_regular, k_delta, k_correct; further down) and, in rk_cells.cuh, blocks of nodes.
// rk_direct_launch.cuh chooses.
//
// Along an axis the tables T_m(o) = (o/a~)^m phi(|o|/a~) (Eq. 6-7, 44, 77) have 2r + 1
// terms, r <= 4.  Summed directly, a 1D circular convolution (Eq. 34) costs about
// 2r + 1 multiply-adds per node; a forward and an inverse transform of a 256-node line
// cost about 40, and in FP64, which issues at 1/64 of the FP32 rate on this GPU, that
// is what bounded the transform passes (9.30 ms per K.u at 256^3, 0.44 ms of HBM
// traffic at the copy bandwidth).  Direct sums also need only neighbours, so an operator
// fits in one kernel and its intermediate fields (90 bytes per node in FP32 through HBM
// before) stay in registers and shared memory.
//
// k_direct: every node on its own, on 2D boxes and on large 3D ones without regular nodes
// (K at 256^2 in FP64, r = 1: 282 us by transform passes, 16 us).  A block owns TX x TY columns of the box and walks along z, one plane per step.  The
// chain of a step, each stage working on the plane the stage before it finished in the
// step before (double buffers, so one barrier per step):
//   load   d of the next plane, with its halo, masked (Eq. 91), or r + beta p (CG)
//   x fwd  a_m = T_m (*)_x d                                    shared -> shared
//   y, z   E_(mx,my) = T_my (*)_y a_mx; the last 2r + 1 planes of E stay in registers;
//          D_p = T_mz (*)_z E (Eq. 86); g_p from D (Eq. 90-91); the reflected sums
//          G_(mx,my) += Tbar_mz (*)_z g_p of the next 2r + 1 planes in registers
//   y refl F_mx = sum_my Tbar_my (*)_y G                         shared -> shared
//   x refl f = sum_mx Tbar_mx (*)_x F, masked                    shared -> HBM
// A thread of the y, z stage holds NR rows of one x, so that a shared-memory value of
// the y sums serves up to NR of them (the shared-memory reads bound FP32 otherwise) and
// the z sums run on row pairs in the packed two-lane FP32 instructions.
// The halo is computed twice by neighbouring blocks; the tile sizes below weigh that
// against the registers the z window takes (2 n_Y (2r + 1) values per column).
#pragma once

#include "rk_common.cuh"
#include "rk_passes.cuh"
#include "rk_pointwise.cuh"

namespace rk {

constexpr int kDirectMaxReach = 4;  // supports up to a = 5h

// DM_MASS_STIFF: M + dt K of a CG step, by blocks of nodes in FP64
enum DirectMode { DM_STIFF = 0, DM_EVAL_U = 1, DM_TRANSPOSE_U = 2, DM_MASS_STIFF = 3 };

// per-node flag byte
constexpr int kRowPad = 8;      // nodes a padded row of flags starts before x = 0
constexpr int kRowTile = 32;    // and it ends kRowPad after the next multiple of this
constexpr unsigned kNodeChi = 1, kNodeOmega = 2, kNodeGamma = 4;

// Classes of the cells (kCell^3 nodes) of the box: without chi nodes; inner (every node
// within twice the reach lies in chi and none of the cell's in chi_gamma: no mask changes
// an input or an output of the cell); any other.
constexpr int kCell = 8;
constexpr int kCellZero = 0, kCellInner = 1, kCellMixed = 2;

// A cell of the corrections, and its bounding box (offsets in the cell, lo <= . < hi) of
// the nodes concerned.
struct CorrCell {
  short c[3];
  unsigned char lo[3], hi[3];
};

// The separable structure of a basis: basis function p is x^mx y^my z^mz with
// (mx, my) = its group; groups in order of first appearance.
template <int S>
struct DBasis;
template <>
struct DBasis<4> {  // 3D, [1, x, y, z]
  static constexpr int DIM = 3, NX = 2, NG = 3;
  static constexpr RK_HD int gmx(int g) { return g == 1 ? 1 : 0; }
  static constexpr RK_HD int gmy(int g) { return g == 2 ? 1 : 0; }
  static constexpr RK_HD int grp(int p) { return p == 3 ? 0 : p; }
  static constexpr RK_HD int az(int p) { return p == 3 ? 1 : 0; }
};
template <>
struct DBasis<10> {  // 3D, [1, x, y, z, x^2, xy, xz, y^2, yz, z^2]
  static constexpr int DIM = 3, NX = 3, NG = 6;
  static constexpr RK_HD int gmx(int g) { return g == 1 || g == 4 ? 1 : (g == 3 ? 2 : 0); }
  static constexpr RK_HD int gmy(int g) { return g == 2 || g == 4 ? 1 : (g == 5 ? 2 : 0); }
  static constexpr RK_HD int grp(int p) {
    return p == 0 || p == 3 || p == 9 ? 0 : (p == 1 || p == 6 ? 1 : (p == 2 || p == 8 ? 2 : (p == 4 ? 3 : (p == 5 ? 4 : 5))));
  }
  static constexpr RK_HD int az(int p) { return p == 9 ? 2 : (p == 3 || p == 6 || p == 8 ? 1 : 0); }
};
template <>
struct DBasis<3> {  // 2D, [1, x, y]
  static constexpr int DIM = 2, NX = 2, NG = 3;
  static constexpr RK_HD int gmx(int g) { return g == 1 ? 1 : 0; }
  static constexpr RK_HD int gmy(int g) { return g == 2 ? 1 : 0; }
  static constexpr RK_HD int grp(int p) { return p; }
  static constexpr RK_HD int az(int) { return 0; }
};
template <>
struct DBasis<6> {  // 2D, [1, x, y, x^2, xy, y^2]
  static constexpr int DIM = 2, NX = 3, NG = 6;
  static constexpr RK_HD int gmx(int g) { return g == 1 || g == 4 ? 1 : (g == 3 ? 2 : 0); }
  static constexpr RK_HD int gmy(int g) { return g == 2 || g == 4 ? 1 : (g == 5 ? 2 : 0); }
  static constexpr RK_HD int grp(int p) { return p; }
  static constexpr RK_HD int az(int) { return 0; }
};
// basis functions even in every coordinate: the only ones whose b^0 is not zero at a
// node with a symmetric support
template <int S>
constexpr RK_HD bool even_p(int p) {
  return S == 10 ? (p == 0 || p == 4 || p == 7 || p == 9) : (S == 6 ? (p == 0 || p == 3 || p == 5) : p == 0);
}

// What a launch would do: the partials p . Ap it writes, whether K takes the way through the
// fields g_p (on entry: whether the handle has or could have them), and the time it takes on a
// box with that share of its cells active (not empty of chi nodes; 0: not estimated, a way
// that the transform passes do not beat).
struct DirectQuery {
  long long blocks = 0;
  bool fields = false;
  bool cg = true;
  double active = 1.0;
  double us = 0.0;
};

template <typename T>
struct DirectArgs {
  const T* in;
  T* out;
  const uint8_t* flags;  // per node: kNodeChi | kNodeOmega | kNodeGamma
  unsigned in_bits;      // inputs count where flags & in_bits (0: everywhere)
  unsigned out_bits;     // outputs are 0 where !(flags & out_bits)
  const uint8_t* cls;    // per cell: its class
  const uint8_t* prow;   // the flags with every row continued periodically: row (y, z) at
  int ppitch;            // ppitch (y + ny z), its node x at byte kRowPad + x
  const int* cidx;       // per node: -1 outside chi, 0 regular, 1 + row of ctab
  const T* ctab;         // rows of the irregular nodes, pitch ctab_pitch<T>(S)
  T breg[31];            // b^x_p, b^y_p, b^z_p, chi V of a regular node
  int diag;              // b^k of a regular node is diagonal (g_{1+k} = creg[k] D_{1+k})
  T creg[3];
  const T* b0;           // b^0_p fields, [S][nbox]
  int diag0;             // b^0 of a regular node is zero but for the even p
  T b0reg[10];
  T vreg;                // chi V of a regular node
  T dt;                  // MASS_STIFF
  const T* wfield;       // TRANSPOSE_U: weight of the input (may be null)
  T tab[3][kDirectMaxReach + 1];  // T_m(o), m = 0 .. 2, o = 0 .. r
  int nx, ny, nz;
  long long nbox;
  T w0[2 * kDirectMaxReach + 1];     // regular stencil: sum_o T_0(o) T_0(o + k), k = 0 .. 2r
  T w1[3][2 * kDirectMaxReach + 1];  // c_k times that of T_1, per axis
  int tiles_x, tiles_y, zc;  // block b: tile (b % tiles_x, b / tiles_x % tiles_y), planes zc (b / (tiles_x tiles_y)) ...
  // corrections of the regular stencil: cells with nodes where delta may not vanish, and
  // with outputs that see one; slot of a cell in delta (-1: none), [slot][p][kCell^3]
  const CorrCell *ncell, *ocell;
  const int* slot;
  T* delta;
  int corrected;  // the box has these lists
  int ncells, ocells;
  // the operators by blocks of nodes: the extents of a block, and the fields g_p [S][nbox]
  // (zero in the cells without chi nodes)
  int bx, by, bz;
  T* gall;
  int after;  // the launches may overlap the ends of those before them (launch_after)
  // CG: in = r (or z), p of the last step in p[par], that of this step to p[par ^ 1]
  T* p0;
  T* p1;
  CGState* cg;
  double* partials;      // one p.Ap per block of the step's launches
  unsigned* counter;
  unsigned part0, parts; // this launch's first partial, and how many all launches write
};

// ------------------------------------------------------------- row vectors
template <typename T, int N>
struct RowVec {
  T v[N];
};
template <typename T, int N>
constexpr bool rv_packed() {
#if defined(RK_PACKED_F32)
  return std::is_same<T, float>::value && N % 2 == 0;
#else
  return false;
#endif
}
template <typename T, int N>
RK_DEV void rv_fma(RowVec<T, N>& acc, T c, const RowVec<T, N>& a) {
  if constexpr (rv_packed<T, N>()) {
#pragma unroll
    for (int i = 0; i < N; i += 2) {
      const cpx<T> r = pfma(cmk(a.v[i], a.v[i + 1]), cmk(c, c), cmk(acc.v[i], acc.v[i + 1]));
      acc.v[i] = r.x;
      acc.v[i + 1] = r.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) acc.v[i] = c * a.v[i] + acc.v[i];
  }
}
template <typename T, int N>
RK_DEV RowVec<T, N> rv_mul(T c, const RowVec<T, N>& a) {
  RowVec<T, N> r;
  if constexpr (rv_packed<T, N>()) {
#pragma unroll
    for (int i = 0; i < N; i += 2) {
      const cpx<T> q = cscale(cmk(a.v[i], a.v[i + 1]), c);
      r.v[i] = q.x;
      r.v[i + 1] = q.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) r.v[i] = c * a.v[i];
  }
  return r;
}
// a + b or a - b
template <int SGN, typename T, int N>
RK_DEV RowVec<T, N> rv_add(const RowVec<T, N>& a, const RowVec<T, N>& b) {
  RowVec<T, N> r;
  if constexpr (rv_packed<T, N>()) {
#pragma unroll
    for (int i = 0; i < N; i += 2) {
      const cpx<T> x = cmk(a.v[i], a.v[i + 1]), y = cmk(b.v[i], b.v[i + 1]);
      const cpx<T> q = SGN > 0 ? x + y : x - y;
      r.v[i] = q.x;
      r.v[i + 1] = q.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) r.v[i] = SGN > 0 ? a.v[i] + b.v[i] : a.v[i] - b.v[i];
  }
  return r;
}

// A coefficient of row vectors.  In the packed FP32 form it takes a register pair holding it
// twice; pinned there, since the compiler otherwise builds the pair anew from the kernel's
// parameters at every use (more instructions than the sums themselves).
template <typename T, int N>
struct RowCoef {
  RowVec<T, rv_packed<T, N>() ? 2 : 1> p;
  RK_DEV void set(T c) {
    p.v[0] = c;
    if constexpr (rv_packed<T, N>()) {
      p.v[1] = c;
      asm volatile("" : "+f"(p.v[0]), "+f"(p.v[1]));
    }
  }
};
template <typename T, int N>
RK_DEV void rv_fma(RowVec<T, N>& acc, const RowCoef<T, N>& c, const RowVec<T, N>& a) {
  if constexpr (rv_packed<T, N>()) {
#pragma unroll
    for (int i = 0; i < N; i += 2) {
      const cpx<T> r = pfma(cmk(a.v[i], a.v[i + 1]), cmk(c.p.v[0], c.p.v[1]), cmk(acc.v[i], acc.v[i + 1]));
      acc.v[i] = r.x;
      acc.v[i + 1] = r.y;
    }
  } else {
    rv_fma(acc, c.p.v[0], a);
  }
}
template <typename T, int N>
RK_DEV RowVec<T, N> rv_mul(const RowCoef<T, N>& c, const RowVec<T, N>& a) {
  if constexpr (rv_packed<T, N>()) {
    RowVec<T, N> r;
#pragma unroll
    for (int i = 0; i < N; i += 2) {
      const cpx<T> q = pmul(cmk(a.v[i], a.v[i + 1]), cmk(c.p.v[0], c.p.v[1]));
      r.v[i] = q.x;
      r.v[i + 1] = q.y;
    }
    return r;
  } else {
    return rv_mul(c.p.v[0], a);
  }
}

// One output of a 1D sum at position c of `in` (spacing 1): sum_o T_m(o) in(c - DIR o);
// T_m is even for even m and odd for odd m, T_1(0) = T_2(0) = 0.
template <int M, int R, int DIR, typename T>
RK_DEV T conv1(const T* in, int c, const T (*tab)[kDirectMaxReach + 1]) {
  T acc = M == 0 ? tab[0][0] * in[c] : (T)0;
#pragma unroll
  for (int o = 1; o <= R; ++o) {
    const T s = M == 1 ? (DIR > 0 ? in[c - o] - in[c + o] : in[c + o] - in[c - o]) : in[c - o] + in[c + o];
    acc = (M != 0 && o == 1) ? tab[M][1] * s : tab[M][o] * s + acc;
  }
  return acc;
}
template <int R, int DIR, typename T>
RK_DEV T conv1_m(int m, const T* in, int c, const T (*tab)[kDirectMaxReach + 1]) {
  return m == 0 ? conv1<0, R, DIR>(in, c, tab) : (m == 1 ? conv1<1, R, DIR>(in, c, tab) : conv1<2, R, DIR>(in, c, tab));
}

// N consecutive shared-memory values from a 16-byte boundary (N even)
template <int N, typename T>
RK_DEV void smem_row(const T* p, T* v) {
  constexpr int W = 16 / (int)sizeof(T);
  constexpr int NV = N / W;
  using V16 = Vec16<T>;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const V16 q = *reinterpret_cast<const V16*>(p + k * W);
    memcpy(v + k * W, &q, 16);
  }
  if constexpr (N % W != 0) {
    const float2 q = *reinterpret_cast<const float2*>(p + NV * W);  // FP32, two values left
    v[N - 2] = q.x;
    v[N - 1] = q.y;
  }
}
template <int N, typename T>
RK_DEV void smem_row_put(T* p, const T* v) {
  constexpr int W = 16 / (int)sizeof(T);
#pragma unroll
  for (int k = 0; k < N / W; ++k) {
    Vec16<T> q;
    memcpy(&q, v + k * W, 16);
    reinterpret_cast<Vec16<T>*>(p)[k] = q;
  }
}

// one value from global to shared memory, asynchronously
template <typename T>
RK_DEV void cp_async_value(T* smem, const T* gmem) {
  if constexpr (sizeof(T) == 4)
    cp_async4(smem, gmem, 4);
  else
    cp_async8(smem, gmem, 8);
}
template <int N>
RK_DEV void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// planes of the input in shared memory: one in use and three on their way (a load from
// HBM takes longer than a step)
constexpr int kStages = 4;

// Tile of a block: TX x TY columns, NR rows per thread of the y, z stage; the small
// tile spreads small boxes over the chip.
template <typename T, int S, int R, int MODE, bool SMALL>
struct DTile {
  using B = DBasis<S>;
  static constexpr bool FWD = MODE != DM_TRANSPOSE_U, REFL = MODE != DM_EVAL_U;
  static constexpr int RF = FWD ? R : 0, RO = REFL ? R : 0;
  static constexpr int ZF = B::DIM == 3 ? RF : 0, ZO = B::DIM == 3 ? RO : 0;
  static constexpr int NE = 2 * ZF + 1, NGR = 2 * ZO + 1;  // planes of the z windows
  static constexpr int PERIOD = B::DIM == 3 ? 2 * R + 1 : 1;
  // registers of the windows per column, in 4-byte units
  static constexpr int WIN = ((FWD ? NE : 0) + (REFL ? NGR : 0)) * B::NG * (int)sizeof(T) / 4;
  static constexpr int NR = WIN <= 42 ? 2 : 1;
  static constexpr int TX = SMALL ? 8 : 16, TY = 8;
  // coefficients of an irregular node, and whether those of the next plane are loaded
  // a step ahead (else where they are used, for want of registers)
  static constexpr int NCO = MODE == DM_STIFF ? ctab_pitch<T>(S) : S;
  static constexpr bool AHEAD = WIN * NR + NCO * NR * (int)sizeof(T) / 4 <= 140;
  // outputs per item of the x stages, rows per item of the reflected y stage: FP64
  // stages are cut finer (their time is issue time, which the warps should share evenly)
  static constexpr int XW = sizeof(T) == 8 ? 2 : 4, NRO = 2;
  static constexpr int GX = TX + 2 * RO, GY = TY + 2 * RO;   // columns of g
  static constexpr int NGY = (GY + NR - 1) / NR, GYP = NGY * NR;
  static constexpr int YZ = GX * NGY;                        // threads of the y, z stage
  static constexpr int THREADS = (YZ + 31) / 32 * 32;
  static constexpr int LX = GX + 2 * RF, LY = GY + 2 * RF;   // values of d
  static constexpr int XQ = (GX + XW - 1) / XW;
  static constexpr int AP = (GX + 3) / 4 * 4;                // pitch of a, G, F
  static constexpr int NXI = FWD ? (LY * XQ + THREADS - 1) / THREADS : 0;
  static constexpr int DP = (AP + 2 * RF + 3) / 4 * 4;       // pitch of d
  static constexpr int DR = GYP + 2 * RF;                    // rows of d and a (padded)
  static constexpr int NLD = FWD ? (LX * LY + THREADS - 1) / THREADS : 0;
  static constexpr int FW = LX / 4 + 2;                      // 4-byte words of flags per row
  static constexpr int ND = FWD ? DR * DP : 0, NA = FWD ? B::NX * DR * AP : 0;
  static constexpr int NGB = REFL ? B::NG * GY * AP : 0, NF = REFL ? B::NX * TY * AP : 0;
  static constexpr size_t smem(bool cg) {
    return sizeof(T) * ((size_t)kStages * ND * (cg ? 2 : 1) + 2 * (size_t)(NA + NGB + NF)) +
           (FWD && !cg ? (size_t)kStages * LY * FW * 4 : 0);
  }
  // blocks an SM should hold: as many as the windows and the working set of the
  // y, z stage leave registers for
  static constexpr int REGS = WIN * NR + (AHEAD ? NCO * NR * (int)sizeof(T) / 4 : 0) + (sizeof(T) == 8 ? 80 : 56) + (S > 4 ? 24 : 0);
  static constexpr int FIT = 65536 / (THREADS * (REGS < 248 ? (REGS + 7) / 8 * 8 : 248));
  static constexpr int MINB = FIT < 1 ? 1 : (FIT > 8 ? 8 : FIT);
};

// p . Ap of the CG step: as cg_pap_reduce_warps, over the blocks of all the launches of
// the step (the last of them to finish sums the partials in order)
template <int THREADS, typename T>
RK_DEV void direct_pap_reduce(const DotAccPair<T>& dot, const DirectArgs<T>& a) {
  constexpr int W = THREADS / 32;
  __shared__ double wsum[W];
  __shared__ bool last;
  const double v = dot.warp_value();
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < W; ++w) s += wsum[w];
    a.partials[a.part0 + blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z)] = s;
    __threadfence();
    last = atomicAdd(a.counter, 1u) == a.parts - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  // (the scalars are on their way with the partials: this block's chain ends the step)
  CGState* st = a.cg;
  const double rz = st->rz, rr = st->rr, stop = st->stop;
  double s = partial_sums<THREADS>(a.partials, a.parts);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double pap = 0.0;
    for (int w = 0; w < W; ++w) pap += wsum[w];
    st->pAp = pap;
    double al = 0.0;
    bool done = false;  // past the caller's bound (CGState::stop) a step changes nothing
    if (stop >= 0.0) {
      done = !(sqrt(rr) > stop);
      if (!done) {
        ++st->steps;
        if (!(pap > 0.0) || !isfinite(pap)) st->flag = 1;
      }
    }
    if (!done && rz > 0.0) {
      if (pap > 0.0 && isfinite(pap))
        al = rz / pap;
      else
        st->flag = 1;
    }
    st->alpha = al;
    *a.counter = 0u;
  }
}

RK_DEV int wrap_idx(int v, int n) {
  v %= n;
  return v < 0 ? v + n : v;
}
// of an index at most one period away
RK_DEV int wrap_once(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// classes of the cells of a block's column of cells, in shared memory
template <int CX, int CY>
struct CellMap {
  static constexpr int MAXZ = 256 / kCell;
  uint8_t c[MAXZ * CY * CX];
  RK_DEV int at(int x, int y, int z) const {  // offsets in the block, none negative
    return c[((unsigned)z / kCell * CY + (unsigned)y / kCell) * CX + (unsigned)x / kCell];
  }
};
// loads the map and returns the z-cells holding a cell that `mine` accepts, a bit each;
// zinner: the z-cells whose cells are all inner
template <int CX, int CY, int THREADS, typename T, class F>
RK_DEV unsigned cell_map(CellMap<CX, CY>& m, unsigned& zmask, unsigned& zinner, const DirectArgs<T>& a, int x0, int y0,
                         int z0, int zn, F mine) {
  const int cnx = (a.nx + kCell - 1) / kCell, cny = (a.ny + kCell - 1) / kCell;
  if (threadIdx.x == 0) {
    zmask = 0u;
    zinner = ~0u;
  }
  __syncthreads();
  const int n = CX * CY * ((zn + kCell - 1) / kCell);
  for (int e = threadIdx.x; e < n; e += THREADS) {
    const int x = x0 + e % CX * kCell, y = y0 + e / CX % CY * kCell, zc = e / (CX * CY);
    int c = -1;
    if (x < a.nx && y < a.ny) {
      c = a.cls[x / kCell + cnx * (y / kCell + (long long)cny * ((z0 + zc * kCell) / kCell))];
      if (mine(c)) atomicOr(&zmask, 1u << zc);
      if (c != kCellInner) atomicAnd(&zinner, ~(1u << zc));
    }
    m.c[e] = (uint8_t)c;
  }
  __syncthreads();
  return zmask;
}

template <typename T, int S, int R, int MODE, bool SMALL, bool CG>
__global__ void __launch_bounds__(DTile<T, S, R, MODE, SMALL>::THREADS, DTile<T, S, R, MODE, SMALL>::MINB)
    k_direct(const __grid_constant__ DirectArgs<T> a) {
  using D = DTile<T, S, R, MODE, SMALL>;
  using B = DBasis<S>;
  using RV = RowVec<T, D::NR>;
  constexpr int NR = D::NR, NE = D::NE, NGR = D::NGR, PERIOD = D::PERIOD, XW = D::XW;
  RK_DYN_SMEM(T, sm);
  T* dbuf = sm;                                     // [kStages][DR][DP]
  T* pbuf = dbuf + kStages * D::ND;                 // CG: the last p
  T* abuf = pbuf + (CG ? kStages * D::ND : 0);      // [2][NX][DR][AP], the first two m interleaved
  T* gbuf = abuf + 2 * D::NA;                       // [2][NG][GY][AP]
  T* fbuf = gbuf + 2 * D::NGB;                      // [2][NX][TY][AP]
  uint8_t* mbuf = reinterpret_cast<uint8_t*>(fbuf + 2 * D::NF);  // [kStages][LY][4 FW] flags of the d tile
  const int tid = threadIdx.x;
  const int x0 = blockIdx.x % a.tiles_x * D::TX, y0 = blockIdx.x / a.tiles_x % a.tiles_y * D::TY;
  int z0 = blockIdx.x / (a.tiles_x * a.tiles_y) * a.zc;
  int zn = min(a.zc, a.nz - z0);  // output planes
  const long long ps = (long long)a.nx * a.ny;
  const T* p_old = nullptr;
  T* p_new = nullptr;
  T beta = (T)0;
  if constexpr (CG) {
    const int par = a.cg->par;
    p_old = par ? a.p1 : a.p0;
    p_new = par ? a.p0 : a.p1;
    beta = (T)a.cg->beta;
  }

  // the cells of the block: zeros where there is no node of chi, and the planes between
  // the first and the last cell that this kernel computes
  auto mine = [](int c) { return c == kCellMixed || c == kCellInner; };
  __shared__ CellMap<D::TX / kCell, 1> map;
  __shared__ unsigned zmask, zinner;
  int zfirst = 0;
  {
    constexpr int CX = D::TX / kCell;
    const unsigned m = cell_map<CX, 1, D::THREADS>(map, zmask, zinner, a, x0, y0, z0, zn, mine);
    for (int c = 0; c < CX * ((zn + kCell - 1) / kCell); ++c) {
      if (map.c[c] != kCellZero) continue;
      const int xc = x0 + c % CX * kCell, zc = z0 + c / CX * kCell;
      const int nzero = min(kCell, z0 + zn - zc);
      for (int e = tid; e < kCell * kCell * nzero; e += D::THREADS) {
        const int x = xc + e % kCell, y = y0 + e / kCell % kCell;
        if (x < a.nx && y < a.ny) {
          const long long i = x + (long long)a.nx * y + ps * (zc + e / (kCell * kCell));
          a.out[i] = (T)0;
          if constexpr (CG) p_new[i] = (T)0;
        }
      }
    }
    if (m == 0u) {
      if constexpr (CG) direct_pap_reduce<D::THREADS>(DotAccPair<T>(), a);
      return;
    }
    zfirst = (__ffs(m) - 1) * kCell;
    zn = min(zn, (32 - __clz(m)) * kCell) - zfirst;
    z0 += zfirst;
  }
  // class of the cell of the block's column (x, y) in output plane j
  auto mine_at = [&](int x, int y, int j) { return mine(map.at(x, y, zfirst + j)); };

  // loader items: one value of the d tile each, at the same place of every plane
  constexpr int NL = D::NLD > 0 ? D::NLD : 1;
  int goff[NL];
  bool inner[CG ? NL : 1];
  if constexpr (D::FWD) {
#pragma unroll
    for (int i = 0; i < D::NLD; ++i) {
      const int e = tid + i * D::THREADS;
      const int rr = e / D::LX - D::RO - D::RF, cc = e % D::LX - D::RO - D::RF;
      goff[i] = e < D::LX * D::LY ? wrap_idx(x0 + cc, a.nx) + a.nx * wrap_idx(y0 + rr, a.ny) : -1;
      if constexpr (CG) inner[i] = rr >= 0 && rr < D::TY && cc >= 0 && cc < D::TX && y0 + rr < a.ny && x0 + cc < a.nx;
    }
  }
  // flags of the d tile: 4-byte words where rows are whole words, else single bytes
  const bool masked = D::FWD && !CG && a.in_bits;
  const bool words = a.nx % 4 == 0;
  const int xw0 = wrap_idx(x0 - D::RO - D::RF, a.nx);  // x of the tile's first column
  const int mshift = words ? xw0 & 3 : 0;              // its byte in the row of flags
  // items of the x stage: offsets in d and a
  constexpr int NXI = D::NXI > 0 ? D::NXI : 1;
  int xs[NXI], xd[NXI];
#pragma unroll
  for (int i = 0; i < D::NXI; ++i) {
    const int e = tid + i * D::THREADS;
    xs[i] = e < D::LY * D::XQ ? e / D::XQ * D::DP + e % D::XQ * XW : -1;
    xd[i] = e / D::XQ * D::AP + e % D::XQ * XW;
  }
  // the columns of the y, z stage
  const int gx = tid % D::GX, gy = tid / D::GX * NR;
  const bool yz_on = tid < D::YZ;
  const unsigned yz_mask = __ballot_sync(0xffffffffu, yz_on);
  int noff[NR];
#pragma unroll
  for (int r = 0; r < NR; ++r) noff[r] = wrap_idx(x0 - D::RO + gx, a.nx) + a.nx * wrap_idx(y0 - D::RO + gy + r, a.ny);

  const int K = zn + 2 * D::ZF + 2 * D::ZO;     // planes of the input
  int zl = wrap_idx(z0 - D::ZF - D::ZO, a.nz);  // z of the plane loaded next
  int zg = wrap_idx(z0 - D::ZO, a.nz);          // z of the plane of g whose class is loaded next
  RV E[D::FWD ? NE : 1][B::NG], G[D::REFL ? NGR : 1][B::NG];
#pragma unroll
  for (int g = 0; g < B::NG; ++g) {
#pragma unroll
    for (int j = 0; j < NGR; ++j)
#pragma unroll
      for (int r = 0; r < NR; ++r) G[D::REFL ? j : 0][g].v[r] = (T)0;
#pragma unroll
    for (int j = 0; j < NE; ++j)
#pragma unroll
      for (int r = 0; r < NR; ++r) E[D::FWD ? j : 0][g].v[r] = (T)0;
  }
  // copies of plane k of the input (and of p, of the flags) on their way
  auto issue = [&](int k) {
    if constexpr (D::FWD) {
      if (k < K) {
        const long long pz = ps * zl;
        const int st = k % kStages;
#pragma unroll
        for (int i = 0; i < D::NLD; ++i)
          if (goff[i] >= 0) {
            const int e = tid + i * D::THREADS;
            const int o = st * D::ND + e / D::LX * D::DP + e % D::LX;
            cp_async_value(dbuf + o, a.in + pz + goff[i]);
            if constexpr (CG) cp_async_value(pbuf + o, p_old + pz + goff[i]);
          }
        if (masked) {
          if (words) {
            for (int e = tid; e < D::LY * D::FW; e += D::THREADS) {
              const int x = wrap_idx(xw0 - mshift + 4 * (e % D::FW), a.nx);
              const int y = wrap_idx(y0 - D::RO - D::RF + e / D::FW, a.ny);
              cp_async4(mbuf + (st * D::LY * D::FW + e) * 4, a.flags + pz + x + (long long)a.nx * y, 4);
            }
          } else {
#pragma unroll
            for (int i = 0; i < D::NLD; ++i)
              if (goff[i] >= 0) {
                const int e = tid + i * D::THREADS;
                mbuf[(st * D::LY + e / D::LX) * D::FW * 4 + e % D::LX] = __ldg(a.flags + pz + goff[i]);
              }
          }
        }
        zl = zl + 1 == a.nz ? 0 : zl + 1;
      }
      cp_async_commit();
    }
  };
  // plane k has landed: mask it, or form p
  auto finish = [&](int k) {
    if constexpr (D::FWD) {
      const int st = k % kStages;
      if constexpr (CG) {
        const bool own = k >= D::ZF + D::ZO && k < D::ZF + D::ZO + zn;
        const long long pz = ps * (z0 + k - D::ZF - D::ZO);
#pragma unroll
        for (int i = 0; i < D::NLD; ++i)
          if (goff[i] >= 0) {
            const int e = tid + i * D::THREADS;
            const int o = st * D::ND + e / D::LX * D::DP + e % D::LX;
            const T v = dbuf[o] + beta * pbuf[o];
            dbuf[o] = v;
            if (own && inner[i] && mine_at(e % D::LX - D::RO - D::RF, 0, k - D::ZF - D::ZO)) p_new[pz + goff[i]] = v;
          }
      } else if (masked) {
        // (flags may have been copied by another thread)
        __syncthreads();
#pragma unroll
        for (int i = 0; i < D::NLD; ++i)
          if (goff[i] >= 0) {
            const int e = tid + i * D::THREADS;
            if (!(mbuf[(st * D::LY + e / D::LX) * D::FW * 4 + mshift + e % D::LX] & a.in_bits))
              dbuf[st * D::ND + e / D::LX * D::DP + e % D::LX] = (T)0;
          }
      }
    }
  };
  // node classes, their coefficients (and the inputs of TRANSPOSE_U) of the coming planes of g
  int cnow[NR], cnext[NR];
  T co[D::AHEAD ? NR : 1][D::NCO];
  RV yin, win;
  uint8_t fin[NR];
  auto load_class = [&]() {
    const long long pz = ps * zg;
    zg = zg + 1 == a.nz ? 0 : zg + 1;
#pragma unroll
    for (int r = 0; r < NR; ++r) cnext[r] = __ldg(a.cidx + pz + noff[r]);
  };
  auto load_coefs = [&](T* c, int idx, long long i) {
    if constexpr (MODE == DM_STIFF) {
      const Vec16<T>* src = reinterpret_cast<const Vec16<T>*>(a.ctab + (long long)(idx - 1) * D::NCO);
#pragma unroll
      for (int t = 0; t < D::NCO / (16 / (int)sizeof(T)); ++t) {
        const Vec16<T> raw = __ldg(src + t);
        memcpy(c + t * (16 / (int)sizeof(T)), &raw, 16);
      }
    } else {
#pragma unroll
      for (int p = 0; p < S; ++p) c[p] = __ldg(a.b0 + (long long)p * a.nbox + i);
    }
  };
  auto load_node = [&](long long pz) {  // of the plane at pz, class cnow
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      if constexpr (D::AHEAD) {
        if (cnow[r] > 0) load_coefs(co[r], cnow[r], pz + noff[r]);
      }
      if constexpr (MODE == DM_TRANSPOSE_U) {
        yin.v[r] = __ldg(a.in + pz + noff[r]);
        if (a.wfield) win.v[r] = __ldg(a.wfield + pz + noff[r]);
        if (a.in_bits) fin[r] = __ldg(a.flags + pz + noff[r]);
      }
    }
  };
  // the item of the reflected x stage: XW outputs of a row, and their masks (and p) one
  // step ahead
  constexpr int NXR = D::REFL ? (D::TY * (D::TX / XW) + D::THREADS - 1) / D::THREADS : 1;
  int fo[NXR][XW];
  T pv[NXR][CG ? XW : 1];
  auto xr_item = [&](int i, int& row, int& c) {
    const int e = D::THREADS - 1 - tid + i * D::THREADS;
    row = e / (D::TX / XW);
    c = e % (D::TX / XW) * XW;
    return e < D::TY * (D::TX / XW) && y0 + row < a.ny && x0 + c < a.nx;
  };
  auto load_out = [&](int j) {  // of output plane j
#pragma unroll
    for (int i = 0; i < NXR; ++i) {
      int row, c;
      if (!xr_item(i, row, c)) continue;
      const long long o = ps * (z0 + j) + (long long)(y0 + row) * a.nx + x0 + c;
#pragma unroll
      for (int w = 0; w < XW; ++w)
        if (x0 + c + w < a.nx) {
          fo[i][w] = __ldg(a.flags + o + w);
          if constexpr (CG) pv[i][w] = __ldcg(p_new + o + w);
        }
    }
  };

  DotAccPair<T> dot;
  constexpr int LAG = D::FWD ? 1 : 0;
  int zgc = zg;  // z of the plane of g formed next
  if (yz_on) {
    load_class();
#pragma unroll
    for (int r = 0; r < NR; ++r) cnow[r] = cnext[r];
    load_node(ps * zgc);
    load_class();
  }
  if constexpr (D::FWD) {
#pragma unroll
    for (int k = 0; k < kStages - 1; ++k) issue(k);
    cp_async_wait<kStages - 2>();
    finish(0);
  }
  __syncthreads();

  // steps: the y, z stage of step k handles plane k - 1 (TRANSPOSE_U: k), the y sums
  // the plane the y, z stage finished in step k - 1, the x sums the one after
  const int steps = D::REFL ? K + LAG + 2 : K + LAG;
  for (int kk = 0; kk < steps; kk += PERIOD) {
#pragma unroll
    for (int ph = 0; ph < PERIOD; ++ph) {
      const int k = kk + ph;
      if (k >= steps) break;
      issue(k + kStages - 1);
      if constexpr (D::FWD) {
        // ---- x forward: plane k
        if (k < K) {
          const T* d = dbuf + k % kStages * D::ND;
          T* o = abuf + (k & 1) * D::NA;
#pragma unroll
          for (int i = 0; i < D::NXI; ++i)
            if (xs[i] >= 0) {
              T v[XW + 2 * R];
              smem_row<XW + 2 * R>(d + xs[i], v);
              T w[2 * XW];
#pragma unroll
              for (int j = 0; j < XW; ++j) {
                w[2 * j] = conv1<0, R, 1>(v, j + R, a.tab);
                w[2 * j + 1] = conv1<1, R, 1>(v, j + R, a.tab);
              }
              smem_row_put<2 * XW>(o + 2 * xd[i], w);
              if constexpr (B::NX == 3) {
#pragma unroll
                for (int j = 0; j < XW; ++j) w[j] = conv1<2, R, 1>(v, j + R, a.tab);
                smem_row_put<XW>(o + 2 * D::DR * D::AP + xd[i], w);
              }
            }
        }
      }
      // ---- y forward, z, pointwise, z reflected: plane q
      const int q = k - LAG;
      if (q >= 0 && q < K && yz_on) {
        constexpr int L = PERIOD;
        // slots: plane q of E at (ph - LAG) mod L; the plane of g is q - ZF
        const int se = ((ph - LAG) % L + L) % L;
        RV Dp[S];
        if constexpr (D::FWD) {
          const T* av = abuf + (q & 1) * D::NA;
          {
            const cpx<T>* ap = reinterpret_cast<const cpx<T>*>(av) + gy * D::AP + gx;
            cpx<T> v[NR + 2 * R];
#pragma unroll
            for (int j = 0; j < NR + 2 * R; ++j) v[j] = ap[j * D::AP];
#pragma unroll
            for (int r = 0; r < NR; ++r) {
              // groups (0, 0), (1, 0): T_0 of both; (0, 1), (1, 1): T_1; (0, 2): T_2 of a_0
              cpx<T> e0 = cscale(v[r + R], a.tab[0][0]), e1 = cmk((T)0, (T)0);
              T e1x = (T)0, e2 = (T)0;
#pragma unroll
              for (int o = 1; o <= R; ++o) {
                const cpx<T> sm2 = v[r + R - o] + v[r + R + o];
                e0 = pfma(sm2, cmk(a.tab[0][o], a.tab[0][o]), e0);
                if constexpr (B::NX == 3) {
                  const cpx<T> df = v[r + R - o] - v[r + R + o];
                  e1 = o == 1 ? cscale(df, a.tab[1][o]) : pfma(df, cmk(a.tab[1][o], a.tab[1][o]), e1);
                  e2 = o == 1 ? a.tab[2][o] * sm2.x : a.tab[2][o] * sm2.x + e2;
                } else {
                  const T df = v[r + R - o].x - v[r + R + o].x;
                  e1x = o == 1 ? a.tab[1][o] * df : a.tab[1][o] * df + e1x;
                }
              }
              E[se][0].v[r] = e0.x;
              E[se][1].v[r] = e0.y;
              if constexpr (B::NX == 3) {
                E[se][2].v[r] = e1.x;
                E[se][4 % B::NG].v[r] = e1.y;
                E[se][5 % B::NG].v[r] = e2;
              } else {
                E[se][2].v[r] = e1x;
              }
            }
          }
          if constexpr (B::NX == 3) {  // group (2, 0): T_0 of a_2
            const T* ap = av + 2 * D::DR * D::AP + gy * D::AP + gx;
            T v[NR + 2 * R];
#pragma unroll
            for (int j = 0; j < NR + 2 * R; ++j) v[j] = ap[j * D::AP];
#pragma unroll
            for (int r = 0; r < NR; ++r) E[se][3 % B::NG].v[r] = conv1<0, R, 1>(v, r + R, a.tab);
          }
        }
        if (q >= 2 * D::ZF) {
          // D_p of plane q - ZF: sum_o T_mz(o) E(z - o)
          auto form_D = [&](int p) {
            const int g = B::grp(p);
            if constexpr (D::ZF == 0) {
              Dp[p] = E[D::FWD ? se : 0][g];
            } else {
              constexpr int ZF = D::ZF;
              const int m = B::az(p);
              auto slot = [&](int o) { return ((se - ZF - o) % L + 2 * L) % L; };  // plane q - ZF - o
              RV acc;
              if (m == 0) acc = rv_mul(a.tab[0][0], E[slot(0)][g]);
#pragma unroll
              for (int o = 1; o <= ZF; ++o) {
                const RV sd = m == 1 ? rv_add<-1>(E[slot(o)][g], E[slot(-o)][g]) : rv_add<1>(E[slot(o)][g], E[slot(-o)][g]);
                if (m != 0 && o == 1)
                  acc = rv_mul(a.tab[m][1], sd);
                else
                  rv_fma(acc, a.tab[m][o], sd);
              }
              Dp[p] = acc;
            }
          };
          // G(z) += T_mz(o) g_p(z + o): the plane of g adds to the planes z - o
          const int sg = ((ph - LAG - D::ZF) % L + 2 * L) % L;  // slot of the plane of g
          auto scatter = [&](int p, const RV& gp) {
            const int g = B::grp(p);
            if constexpr (D::ZO == 0) {
              G[0][g] = gp;  // one basis function per group
            } else {
              const int m = B::az(p);
              if (m == 0) rv_fma(G[sg][g], a.tab[0][0], gp);
#pragma unroll
              for (int o = 1; o <= D::ZO; ++o) {
                rv_fma(G[((sg - o) % L + L) % L][g], a.tab[m][o], gp);
                rv_fma(G[(sg + o) % L][g], m == 1 ? -a.tab[m][o] : a.tab[m][o], gp);
              }
            }
          };
          bool irr = false;
#pragma unroll
          for (int r = 0; r < NR; ++r) irr |= cnow[r] > 0;
          const long long pz = ps * zgc;
          zgc = zgc + 1 == a.nz ? 0 : zgc + 1;
          if constexpr (MODE == DM_STIFF) {
            if (a.diag && !__any_sync(yz_mask, irr)) {
              // regular nodes and nodes outside chi only: g_{1+k} = c_k D_{1+k} or 0
#pragma unroll
              for (int kx = 0; kx < B::DIM; ++kx) {
                form_D(1 + kx);
                RV gp;
#pragma unroll
                for (int r = 0; r < NR; ++r) gp.v[r] = cnow[r] == 0 ? a.creg[kx] * Dp[1 + kx].v[r] : (T)0;
                scatter(1 + kx, gp);
              }
            } else {
#pragma unroll
              for (int p = 0; p < S; ++p) form_D(p);
#pragma unroll
              for (int r = 0; r < NR; ++r) {
                T cl[D::NCO];
                if (cnow[r] > 0) {
                  if constexpr (D::AHEAD) {
#pragma unroll
                    for (int t = 0; t < 3 * S + 1; ++t) cl[t] = co[r][t];
                  } else {
                    load_coefs(cl, cnow[r], 0);
                  }
                } else {
#pragma unroll
                  for (int t = 0; t < 3 * S + 1; ++t) cl[t] = a.breg[t];
                }
                T dd[S], gg[S];
#pragma unroll
                for (int p = 0; p < S; ++p) dd[p] = Dp[p].v[r];
                pointwise_node<T, S>(cl, cnow[r], dd, gg);
#pragma unroll
                for (int p = 0; p < S; ++p) Dp[p].v[r] = gg[p];
              }
#pragma unroll
              for (int p = 0; p < S; ++p) scatter(p, Dp[p]);
            }
          } else {
            // Alg. 3: u = sum_p b0_p D_p; Alg. 4: g_p = b0_p y.  Outside chi M is the
            // identity: b0 = (1, 0, ...).
            RV y;
            if constexpr (MODE == DM_TRANSPOSE_U) {
#pragma unroll
              for (int r = 0; r < NR; ++r) {
                y.v[r] = a.wfield ? yin.v[r] * win.v[r] : yin.v[r];
                if (a.in_bits && !(fin[r] & a.in_bits)) y.v[r] = (T)0;
              }
            }
            if (a.diag0 && !__any_sync(yz_mask, irr)) {
#pragma unroll
              for (int p = 0; p < S; ++p)
                if (even_p<S>(p)) {
                  if constexpr (D::FWD) {
                    form_D(p);
                    if (p == 0)
                      y = rv_mul(a.b0reg[0], Dp[0]);
                    else
                      rv_fma(y, a.b0reg[p], Dp[p]);
                  } else {
                    RV gp;
#pragma unroll
                    for (int r = 0; r < NR; ++r) gp.v[r] = (cnow[r] == 0 ? a.b0reg[p] : (p == 0 ? (T)1 : (T)0)) * y.v[r];
                    scatter(p, gp);
                  }
                }
            } else {
              if constexpr (D::FWD) {
#pragma unroll
                for (int p = 0; p < S; ++p) form_D(p);
              }
#pragma unroll
              for (int r = 0; r < NR; ++r) {
                T b0[S];
                if (cnow[r] > 0) {
                  if constexpr (D::AHEAD) {
#pragma unroll
                    for (int p = 0; p < S; ++p) b0[p] = co[r][p];
                  } else {
                    load_coefs(b0, cnow[r], pz + noff[r]);
                  }
                } else {
#pragma unroll
                  for (int p = 0; p < S; ++p) b0[p] = cnow[r] == 0 ? a.b0reg[p] : (p == 0 ? (T)1 : (T)0);
                }
                if constexpr (D::FWD) {
                  T s = (T)0;
#pragma unroll
                  for (int p = 0; p < S; ++p) s += b0[p] * Dp[p].v[r];
                  y.v[r] = s;
                } else {
#pragma unroll
                  for (int p = 0; p < S; ++p) Dp[p].v[r] = b0[p] * y.v[r];
                }
              }
              if constexpr (D::REFL) {
#pragma unroll
                for (int p = 0; p < S; ++p) scatter(p, Dp[p]);
              }
            }
            if constexpr (MODE == DM_EVAL_U) {
#pragma unroll
              for (int r = 0; r < NR; ++r)
                if (gy + r < D::TY && x0 + gx < a.nx && y0 + gy + r < a.ny && mine_at(gx, gy + r, q - 2 * D::ZF))
                  a.out[pz + noff[r]] = cnow[r] >= 0 ? y.v[r] : (T)0;
            }
          }
          // coefficients of the next plane, classes of the one after
          if (q + 1 < K) {
#pragma unroll
            for (int r = 0; r < NR; ++r) cnow[r] = cnext[r];
            load_node(ps * zgc);
            if (q + 2 < K) load_class();
          }
          // G of plane q - ZF - ZO is complete
          if constexpr (D::REFL) {
            const int so = D::ZO == 0 ? 0 : ((sg - D::ZO) % L + L) % L;
            if (q >= 2 * D::ZF + 2 * D::ZO) {
              T* dst = gbuf + (k & 1) * D::NGB + gy * D::AP + gx;
#pragma unroll
              for (int g = 0; g < B::NG; ++g)
#pragma unroll
                for (int r = 0; r < NR; ++r)
                  if (gy + r < D::GY) dst[g * (D::GY * D::AP) + r * D::AP] = G[so][g].v[r];
            }
#pragma unroll
            for (int g = 0; g < B::NG; ++g)
#pragma unroll
              for (int r = 0; r < NR; ++r) G[so][g].v[r] = (T)0;
          }
        }
      }
      if constexpr (D::REFL) {
        // ---- y reflected: the plane finished in step k - 1
        const int jy = q - 1 - 2 * D::ZF - 2 * D::ZO;
        if (jy >= 0 && jy < zn) {
          constexpr int NRO = D::NRO;
          const T* gs = gbuf + ((k - 1) & 1) * D::NGB;
          T* fd = fbuf + (k & 1) * D::NF;
          for (int e = tid; e < D::GX * (D::TY / NRO); e += D::THREADS) {
            const int x = e % D::GX, row = e / D::GX * NRO;
            T acc[B::NX][NRO];
#pragma unroll
            for (int g = 0; g < B::NG; ++g) {
              T v[NRO + 2 * R];
#pragma unroll
              for (int j = 0; j < NRO + 2 * R; ++j) v[j] = gs[g * (D::GY * D::AP) + (row + j) * D::AP + x];
#pragma unroll
              for (int r = 0; r < NRO; ++r) {
                const T w = conv1_m<R, -1>(B::gmy(g), v, r + R, a.tab);
                acc[B::gmx(g)][r] = B::gmy(g) == 0 ? w : acc[B::gmx(g)][r] + w;  // (m, 0) comes first
              }
            }
#pragma unroll
            for (int m = 0; m < B::NX; ++m)
#pragma unroll
              for (int r = 0; r < NRO; ++r) fd[m * (D::TY * D::AP) + (row + r) * D::AP + x] = acc[m][r];
          }
        }
        // ---- x reflected: the plane of the y sums of step k - 1
        const int jx = jy - 1;
        if (jx >= 0 && jx < zn) {
          const T* fs = fbuf + ((k - 1) & 1) * D::NF;
#pragma unroll
          for (int i = 0; i < NXR; ++i) {
            int row, c;
            if (!xr_item(i, row, c) || !mine_at(c, row, jx)) continue;
            T acc[XW];
#pragma unroll
            for (int m = 0; m < B::NX; ++m) {
              T v[XW + 2 * R];
              smem_row<XW + 2 * R>(fs + m * (D::TY * D::AP) + row * D::AP + c, v);
#pragma unroll
              for (int j = 0; j < XW; ++j) {
                const T w = conv1_m<R, -1>(m, v, j + R, a.tab);
                acc[j] = m == 0 ? w : acc[j] + w;
              }
            }
            T* out = a.out + ps * (z0 + jx) + (long long)(y0 + row) * a.nx + x0 + c;
#pragma unroll
            for (int j = 0; j < XW; ++j)
              if (x0 + c + j < a.nx) {
                if (!(fo[i][j] & (int)a.out_bits)) acc[j] = (T)0;
                out[j] = acc[j];
                if constexpr (CG) dot.add(cmk(pv[i][j], (T)0), cmk(acc[j], (T)0));
              }
          }
        }
        if (jx + 1 >= 0 && jx + 1 < zn) load_out(jx + 1);
      }
      if constexpr (D::FWD) {
        cp_async_wait<kStages - 2>();
        if (k + 1 < K) finish(k + 1);
      }
      __syncthreads();
    }
  }
  if constexpr (CG) direct_pap_reduce<D::THREADS>(dot, a);
}

// --------------------------------------------- the regular stencil and its corrections
// At a regular node (its whole support in chi, interior V) g_{1+k} = c_k D_{1+k} and the
// other g_p vanish (Eq. 90-91 with the symmetric support).  Writing g_p = c_p D_p + delta_p
// at every node, the part c_p D_p is a plain stencil: the forward and the reflected sums of
// a table along an axis merge into one sum with its autocorrelation (w0 of T_0, w1 of T_1;
// 4r + 1 terms, even),
//   f = c_x w1 x w0 y w0 z d + c_y w0 x w1 y w0 z d + c_z w0 x w0 y w1 z d  (+ corrections),
// about 55 multiply-adds per node for the linear basis's r = 2 against about 70 with every
// sum on its own, and one window of 4r + 1 planes instead of two per group.  delta_p is zero
// at regular nodes and farther than the support from chi, so its reflected sums are added
// by k_delta and k_correct on the cells at the boundary only.
//
// k_regular: a block owns TX x TY columns and walks along z, one barrier per plane.  Its
// warps share the stages, so that a step takes the longer of the two chains, not their sum:
//   x warps     start the copy of a plane three steps ahead; a = w0 (*)_x d and
//               b = c_x w1 (*)_x d of one plane (shared -> shared); mask or form p of the next
//   y, z warps  Q = w0 (*)_y a, P = w0 (*)_y b + c_y w1 (*)_y a of the plane before; the
//               4r + 1 planes of f within reach add w0 P + c_z w1 Q, held in registers, the
//               finished one is stored
// In FP32 a thread of the y, z stage holds column pairs and the x stage takes output pairs:
// the packed two-lane FP32 instructions then do two outputs each.
//
// Bounded by instruction issue in FP32 (of 132 instructions per 32 nodes about 40 are the
// sums; without the roles, the pairs and the pointers that step from plane to plane they were
// over 170) and by the FP64 pipe in FP64 (58 multiply-adds per node with the halo of the tile,
// 2 per cycle and SM).  r = 2, the roles against one chain of stages per thread: FP32 128^3
// 30.4 -> 21.7 us, 96^3 19 -> 15.2 us, spheres in 256^3 173 -> 112 us, a full cube in 256^3
// 125 us both ways; r = 3, 162 x 100 x 72: 43 -> 36 us; FP64 256^3 2.50 -> 2.41 ms.
template <typename T, int R, bool SMALL>
struct RTile {
  static constexpr bool F32 = sizeof(T) == 4;
  static constexpr int XC = F32 ? 2 : 1;                                       // columns per thread
  static constexpr int NR = F32 ? 2 : (SMALL ? 1 : 4);                         // and rows
  static constexpr bool WIDE = F32 && R >= 4;                                  // taller tiles: the halo is 4 r rows
  static constexpr int TX = 32, TY = SMALL ? (WIDE ? 16 : 8) : (F32 && !WIDE ? 16 : 32);
  static constexpr int H = 2 * R, L = 2 * H + 1;
  static constexpr int VL = 16 / (int)sizeof(T);                 // values per 16-byte copy
  static constexpr int HP = (H + VL - 1) / VL * VL;              // halo of the tile along x
  static constexpr int LX = TX + 2 * HP, LY = TY + 2 * H, QX = LX / VL;
  static constexpr int XW = F32 ? 4 : 2, XQ = TX / XW;           // outputs per item of the x stage
  static constexpr int YZT = TX / XC * (TY / NR);                // y, z threads
  static constexpr int XT = WIDE && !SMALL ? 256 : 128;           // x threads
  static constexpr int THREADS = YZT + XT;
  static constexpr int NXI = (LY * XQ + XT - 1) / XT;
  static constexpr int NLD = (QX * LY + XT - 1) / XT;            // copies per x thread
  static constexpr int ND = LY * LX, NA = LY * TX * 2;
  static constexpr size_t smem(bool cg) {
    return sizeof(T) * ((size_t)kStages * ND * (cg ? 2 : 1) + 2 * (size_t)NA) + (cg ? 0 : (size_t)kStages * QX * LY * 4);
  }
  static constexpr int REGS = L * NR * XC * (int)sizeof(T) / 4 + (F32 ? 56 : 90);
  static constexpr int FIT = 65536 / (THREADS * (REGS < 248 ? (REGS + 7) / 8 * 8 : 248));
  static constexpr int MINB = FIT < 1 ? 1 : (FIT > 6 ? 6 : FIT);
};

template <typename T, int R, bool SMALL, bool CG>
__global__ void __launch_bounds__(RTile<T, R, SMALL>::THREADS, RTile<T, R, SMALL>::MINB)
    k_regular(const __grid_constant__ DirectArgs<T> a) {
  using D = RTile<T, R, SMALL>;
  constexpr int H = D::H, L = D::L, NR = D::NR, XW = D::XW, VL = D::VL, XC = D::XC, HP = D::HP;
  using RV = RowVec<T, XC>;
  RK_DYN_SMEM(T, sm);
  T* dbuf = sm;                                 // [kStages][LY][LX]
  T* pbuf = dbuf + kStages * D::ND;             // CG: the last p
  T* abuf = pbuf + (CG ? kStages * D::ND : 0);  // [2][a, b][LY][TX]
  unsigned* mbuf = reinterpret_cast<unsigned*>(abuf + 2 * D::NA);  // [kStages][LY QX] flags of each 16-byte unit
  const int x0 = blockIdx.x % a.tiles_x * D::TX, y0 = blockIdx.x / a.tiles_x % a.tiles_y * D::TY;
  int z0 = blockIdx.x / (a.tiles_x * a.tiles_y) * a.zc;
  int zn = min(a.zc, a.nz - z0);
  const long long ps = (long long)a.nx * a.ny;
  const T* p_old = nullptr;
  T* p_new = nullptr;
  T beta = (T)0;
  // cells without chi nodes: zeros; the planes from the first to the last other cell
  constexpr int CX = D::TX / kCell, CY = D::TY / kCell;
  __shared__ CellMap<CX, CY> map;
  __shared__ unsigned zmask, zinner;
  auto mine = [](int c) { return c == kCellMixed || c == kCellInner; };
  const unsigned zm = cell_map<CX, CY, D::THREADS>(map, zmask, zinner, a, x0, y0, z0, zn, mine);
  grid_wait();
  grid_trigger();  // (after the wait: k_delta relies on it)
  if constexpr (CG) {
    const int par = a.cg->par;
    p_old = par ? a.p1 : a.p0;
    p_new = par ? a.p0 : a.p1;
    beta = (T)a.cg->beta;
  }
  for (int c = 0; c < CX * CY * ((zn + kCell - 1) / kCell); ++c) {
    if (map.c[c] != kCellZero) continue;
    const int xc = x0 + c % CX * kCell, yc = y0 + c / CX % CY * kCell, zc = z0 + c / (CX * CY) * kCell;
    const int nzero = min(kCell, z0 + zn - zc);
    for (int e = threadIdx.x; e < kCell * kCell * nzero; e += D::THREADS) {
      const int x = xc + e % kCell, y = yc + e / kCell % kCell;
      if (x < a.nx && y < a.ny) {
        const long long i = x + (long long)a.nx * y + ps * (zc + e / (kCell * kCell));
        a.out[i] = (T)0;
        if constexpr (CG) p_new[i] = (T)0;
      }
    }
  }
  if (zm == 0u) {
    if constexpr (CG) direct_pap_reduce<D::THREADS>(DotAccPair<T>(), a);
    return;
  }
  const int zfirst = (__ffs(zm) - 1) * kCell;
  zn = min(zn, (32 - __clz(zm)) * kCell) - zfirst;
  z0 += zfirst;
  const int K = zn + 2 * H;
  DotAccPair<T> dot;

  // the warps of the two roles, in turn from block to block so that the SM's schedulers
  // get as many of either
  static_assert(D::YZT % 32 == 0 && D::XT % 32 == 0, "whole warps per role");
  const int rtid = (int)((threadIdx.x + (blockIdx.x & 1) * (D::THREADS / 64 * 32)) % D::THREADS);
  if (rtid >= D::YZT) {
    // ------------------------------------------------------------ x warps
    // Address and predicate instructions outnumber the sums here if they are left to the
    // inner loop: copies run through pointers that step from plane to plane, a thread
    // without an item of its own repeats the last one (the same values to the same place),
    // and 16-byte copies and single ones are two loops.  A CG step copies every unit once:
    // its owner forms p in place as soon as its own copies have landed, and a second copy of
    // the unit could land after that and leave r where p belongs.
    const int tid = rtid - D::YZT;
    static_assert(HP <= kRowPad && D::TX <= kRowTile, "padded rows of flags");
    static_assert((kStages & (kStages - 1)) == 0, "stages by masking");
    constexpr int UNITS = D::QX * D::LY, ITEMS = D::LY * D::XQ;
    int xs[D::NXI], xd[D::NXI];
#pragma unroll
    for (int i = 0; i < D::NXI; ++i) {
      const int e = min(tid + i * D::XT, ITEMS - 1);
      xs[i] = e / D::XQ * D::LX + e % D::XQ * XW;
      xd[i] = e / D::XQ * D::TX + e % D::XQ * XW;
    }
    RowCoef<T, 2> w0[H + 1], w1[H + 1];
#pragma unroll
    for (int u = 0; u <= H; ++u) {
      w0[u].set(a.w0[u]);
      w1[u].set(a.w1[0][u]);
    }
    auto walk = [&](auto vec_) {
      constexpr bool VEC = decltype(vec_)::value;  // rows are whole 16-byte units
      const T* src[D::NLD];                        // the unit in the plane copied next
      const uint8_t* msk[D::NLD];                  // the word that holds its flags
      int unit[D::NLD];
      [[maybe_unused]] int wr[CG ? D::NLD : 1];                     // CG: its place in the tile where p is written here, else -1
      const int zs = wrap_idx(z0 - H, a.nz);
      unsigned left = (unsigned)(a.nz - zs);       // planes to the end of the box
      const long long back = ps * a.nz;
      const long long mplane = (long long)a.ppitch * a.ny, mback = mplane * a.nz;
#pragma unroll
      for (int i = 0; i < D::NLD; ++i) {
        const int e = min(tid + i * D::XT, UNITS - 1);
        unit[i] = e;
        const int rr = e / D::QX - H, cc = e % D::QX * VL - HP;
        const int y = wrap_idx(y0 + rr, a.ny);
        src[i] = a.in + ps * zs + (long long)a.nx * y + (VEC ? wrap_idx(x0 + cc, a.nx) : 0);
        msk[i] = a.prow + mplane * zs + (long long)a.ppitch * y + ((x0 + kRowPad + cc) & ~3);
        if constexpr (CG)
          wr[i] = tid + i * D::XT < UNITS && rr >= 0 && rr < D::TY && cc >= 0 && cc < D::TX && y0 + rr < a.ny && x0 + cc < a.nx
                      ? rr * D::TX + cc : -1;
      }
      [[maybe_unused]] const long long pdiff = CG ? p_old - a.in : 0;
      // the planes whose tile is not inner (bit: z-cell of the nearest output plane)
      auto masked = [&](unsigned k) {
        const unsigned j = k < (unsigned)H ? 0u : min(k - H, (unsigned)zn - 1u);
        return !(zinner >> (((unsigned)zfirst + j) / kCell) & 1u);
      };
      const bool masking = !CG && a.in_bits != 0;
      auto issue = [&](unsigned k) {
        if (k < (unsigned)K) {
          T* to = dbuf + (k & (kStages - 1)) * D::ND;
#pragma unroll
          for (int i = 0; i < D::NLD; ++i) {
            if constexpr (CG) {
              if (D::XT * (i + 1) > UNITS && tid + i * D::XT >= UNITS) continue;
            }
            if constexpr (VEC) {
              cp_async16(to + unit[i] * VL, src[i], 16);
              if constexpr (CG) cp_async16(to + kStages * D::ND + unit[i] * VL, src[i] + pdiff, 16);
            } else {
#pragma unroll
              for (int w = 0; w < VL; ++w) {
                const int x = wrap_idx(x0 - HP + unit[i] % D::QX * VL + w, a.nx);
                cp_async_value(to + unit[i] * VL + w, src[i] + x);
                if constexpr (CG) cp_async_value(to + kStages * D::ND + unit[i] * VL + w, src[i] + pdiff + x);
              }
            }
            src[i] += ps;
          }
          if (masking) {
            if (masked(k)) {
#pragma unroll
              for (int i = 0; i < D::NLD; ++i) cp_async4(mbuf + (k & (kStages - 1)) * UNITS + unit[i], msk[i], 4);
            }
#pragma unroll
            for (int i = 0; i < D::NLD; ++i) msk[i] += mplane;
          }
          if (--left == 0) {
            left = (unsigned)a.nz;
#pragma unroll
            for (int i = 0; i < D::NLD; ++i) {
              src[i] -= back;
              msk[i] -= mback;
            }
          }
        }
        cp_async_commit();
      };
      // plane k has landed: form p, or mask d; a thread works on the units it copied
      [[maybe_unused]] T* pn = CG ? p_new + ps * z0 + (long long)a.nx * y0 + x0 : nullptr;
      auto finish = [&](unsigned k) {
        const unsigned st = k & (kStages - 1);
        if constexpr (CG) {
          const bool own = k >= (unsigned)H && k < (unsigned)(H + zn);
#pragma unroll
          for (int i = 0; i < D::NLD; ++i) {
            if (D::XT * (i + 1) > UNITS && tid + i * D::XT >= UNITS) continue;
            T* o = dbuf + st * D::ND + unit[i] * VL;
            T v[VL], w[VL];
            smem_row<VL>(o, v);
            smem_row<VL>(o + kStages * D::ND, w);
#pragma unroll
            for (int t = 0; t < VL; ++t) v[t] += beta * w[t];
            smem_row_put<VL>(o, v);
            // a unit lies in one cell, whose class says whether p is written here
            if (own && wr[i] >= 0) {
              const int c = wr[i] % D::TX, r = wr[i] / D::TX;
              if (mine(map.at(c, r, zfirst + (int)k - H))) {
                T* q = pn + (long long)a.nx * r + c;
                if constexpr (VEC) {
                  smem_row_put<VL>(q, v);
                } else {
#pragma unroll
                  for (int t = 0; t < VL; ++t)
                    if (x0 + c + t < a.nx) q[t] = v[t];
                }
              }
            }
          }
          if (own) pn += ps;
        } else if (masking && masked(k)) {
          const unsigned want = a.in_bits * (VL == 4 ? 0x01010101u : 0x0101u);
#pragma unroll
          for (int i = 0; i < D::NLD; ++i) {
            const int e = unit[i];
            const unsigned m = mbuf[st * UNITS + e] >> (VL == 4 ? 0 : 8 * ((e % D::QX * VL + kRowPad - HP) & 2));
            if ((m & want) != want) {
#pragma unroll
              for (int t = 0; t < VL; ++t)
                if (!(m >> (8 * t) & a.in_bits)) dbuf[st * D::ND + e * VL + t] = (T)0;
            }
          }
        }
      };
#pragma unroll
      for (int k = 0; k < kStages - 1; ++k) issue(k);
      cp_async_wait<kStages - 2>();
      finish(0);
      __syncthreads();
      for (unsigned k = 0; k <= (unsigned)K; ++k) {
        issue(k + kStages - 1);
        if (k < (unsigned)K) {
          const T* d = dbuf + (k & (kStages - 1)) * D::ND;
          T* o = abuf + (k & 1) * D::NA;
#pragma unroll
          for (int i = 0; i < D::NXI; ++i) {
            T v[XW + 2 * HP];
            smem_row<XW + 2 * HP>(d + xs[i], v);
            T wa[XW], wb[XW];
#pragma unroll
            for (int j = 0; j < XW; j += 2) {
              RowVec<T, 2> c{{v[j + HP], v[j + HP + 1]}};
              RowVec<T, 2> s0 = rv_mul(w0[0], c), s1 = rv_mul(w1[0], c);
#pragma unroll
              for (int t = 1; t <= H; ++t) {
                // (pairs at an even distance are aligned in registers: one packed sum)
                const RowVec<T, 2> l{{v[j + HP - t], v[j + HP + 1 - t]}}, r{{v[j + HP + t], v[j + HP + 1 + t]}};
                RowVec<T, 2> q;
                if (t % 2 == 0)
                  q = rv_add<1>(l, r);
                else
                  q = RowVec<T, 2>{{l.v[0] + r.v[0], l.v[1] + r.v[1]}};
                rv_fma(s0, w0[t], q);
                rv_fma(s1, w1[t], q);
              }
              wa[j] = s0.v[0];
              wa[j + 1] = s0.v[1];
              wb[j] = s1.v[0];
              wb[j + 1] = s1.v[1];
            }
            smem_row_put<XW>(o + xd[i], wa);
            smem_row_put<XW>(o + D::LY * D::TX + xd[i], wb);
          }
        }
        cp_async_wait<kStages - 2>();
        if (k + 1 < (unsigned)K) finish(k + 1);
        __syncthreads();
      }
    };
    if (a.nx % VL == 0)
      walk(std::true_type{});
    else
      walk(std::false_type{});
  } else {
    // ------------------------------------------------------------ y, z warps
    const int cx = rtid % (D::TX / XC) * XC, cy = rtid / (D::TX / XC) * NR;
    // rows of the thread inside the box (n_x is even: a column pair is in or out)
    const int nvr = x0 + cx < a.nx ? min(max(a.ny - y0 - cy, 0), NR) : 0;
    const T* const av = abuf + cy * D::TX + cx;
    // f of the planes q - 2r .. q + 2r; the window moves by writing each sum one place down
    RV acc[L][NR];
#pragma unroll
    for (int j = 0; j < L; ++j)
#pragma unroll
      for (int r = 0; r < NR; ++r)
#pragma unroll
        for (int c = 0; c < XC; ++c) acc[j][r].v[c] = (T)0;
    RowCoef<T, XC> w0[H + 1], wy[H + 1], wz[H + 1];
#pragma unroll
    for (int u = 0; u <= H; ++u) {
      w0[u].set(a.w0[u]);
      wy[u].set(a.w1[1][u]);
      wz[u].set(a.w1[2][u]);
    }
    T pv[CG ? NR * XC : 1];  // p and the flags of the output plane, a step ahead
    unsigned fo[NR];
    int cl = 0;              // class of the thread's cell there
    const bool keep = (a.out_bits & (kNodeChi | kNodeOmega)) != 0;
    long long oi = x0 + cx + (long long)a.nx * (y0 + cy) + ps * z0;  // the output plane loaded for next
    T* out = a.out + oi;                                             // and the one stored next
    auto ahead = [&](int j) {  // class, flags and p of output plane j
      if (j == 0 || ((zfirst + j) & (kCell - 1)) == 0) cl = nvr > 0 ? map.at(cx, cy, zfirst + j) : 0xff;
      if (cl == kCellMixed || CG) {
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          if (r >= nvr) continue;
          if (cl == kCellMixed) {
            if constexpr (XC == 2)
              fo[r] = __ldg(reinterpret_cast<const uint16_t*>(a.flags + oi + r * a.nx));
            else
              fo[r] = __ldg(a.flags + oi + r * a.nx);
          }
          if constexpr (CG) {
            if constexpr (XC == 2) {
              const float2 w = __ldcg(reinterpret_cast<const float2*>(p_new + oi + r * a.nx));
              pv[2 * r] = w.x;
              pv[2 * r + 1] = w.y;
            } else {
              pv[r] = __ldcg(p_new + oi + r * a.nx);
            }
          }
        }
      }
      oi += ps;
    };
    __syncthreads();
    __syncthreads();  // (step 0: the x warps' alone)
    for (int q = 0; q < K; ++q) {
      const T* ap = av + (q & 1) * D::NA;
      RV v[NR + 2 * H], P[NR], Q[NR];
      auto read = [&](const T* from) {
#pragma unroll
        for (int j = 0; j < NR + 2 * H; ++j) {
          if constexpr (XC == 2) {
            const float2 w = *reinterpret_cast<const float2*>(from + j * D::TX);
            v[j].v[0] = w.x;
            v[j].v[1] = w.y;
          } else {
            v[j].v[0] = from[j * D::TX];
          }
        }
      };
      read(ap);
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        Q[r] = rv_mul(w0[0], v[r + H]);
        P[r] = rv_mul(wy[0], v[r + H]);
#pragma unroll
        for (int t = 1; t <= H; ++t) {
          const RV w = rv_add<1>(v[r + H - t], v[r + H + t]);
          rv_fma(Q[r], w0[t], w);
          rv_fma(P[r], wy[t], w);
        }
      }
      read(ap + D::LY * D::TX);
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        rv_fma(P[r], w0[0], v[r + H]);
#pragma unroll
        for (int t = 1; t <= H; ++t) rv_fma(P[r], w0[t], rv_add<1>(v[r + H - t], v[r + H + t]));
      }
#pragma unroll
      for (int t = 0; t < L; ++t) {
        const int u = t < H ? H - t : t - H;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          if (t == L - 1) {  // a new plane
            acc[t][r] = rv_mul(w0[u], P[r]);
          } else {
            acc[t][r] = acc[t + 1][r];
            rv_fma(acc[t][r], w0[u], P[r]);
          }
          rv_fma(acc[t][r], wz[u], Q[r]);
        }
      }
      const int j = q - 2 * H;  // the finished output plane
      if (j >= 0) {
        auto put = [&](int r, const RV& f) {
          if constexpr (XC == 2)
            *reinterpret_cast<float2*>(out + r * a.nx) = make_float2(f.v[0], f.v[1]);
          else
            out[r * a.nx] = f.v[0];
          if constexpr (CG) {
            if constexpr (XC == 2)
              dot.add(cmk(pv[2 * r], pv[2 * r + 1]), cmk(f.v[0], f.v[1]));
            else
              dot.add(cmk(pv[r], (T)0), cmk(f.v[0], (T)0));
          }
        };
        if (cl == kCellInner && keep) {
#pragma unroll
          for (int r = 0; r < NR; ++r)
            if (r < nvr) put(r, acc[0][r]);
        } else if (mine(cl)) {
#pragma unroll
          for (int r = 0; r < NR; ++r)
            if (r < nvr) {
              RV f = acc[0][r];
#pragma unroll
              for (int c = 0; c < XC; ++c)
                if (cl == kCellInner || !(fo[r] >> (8 * c) & a.out_bits)) f.v[c] = (T)0;
              put(r, f);
            }
        }
        out += ps;
      }
      if (j + 1 >= 0 && j + 1 < zn) ahead(j + 1);
      __syncthreads();
    }
  }
  if constexpr (CG) direct_pap_reduce<D::THREADS>(dot, a);
}

// i / n for i < 4096, n <= 16 as a multiplication: with m = ceil(2^20 / n) the error
// i (m n - 2^20) / (2^20 n) stays under 1 / n, and i m fits 32 bits.  (Conversions to and
// from FP32 run at an eighth of the rate of a multiplication.)
RK_DEV unsigned box_inv(int n) { return ((1u << 20) + (unsigned)n - 1u) / (unsigned)n; }
RK_DEV int box_div(int i, unsigned m) { return (int)(((unsigned)i * m) >> 20); }

// 256 threads against 128: K u on spheres in 256^3, FP32, quadratic basis, k_correct 131
// against 151 us; a cube in 256^3, linear basis, k_delta 40 against 50 us, k_correct 67 / 70.
// Wide supports leave an SM few blocks: r = 4, k_correct 233 us with 512, 254 with 256.
template <int R>
constexpr int corr_threads() {
  return R >= 4 ? 512 : 256;
}

// The sums of a box in shared memory, fields at the given strides; a thread takes two
// neighbouring outputs, which share all but two of their inputs.  For r = 4 alone, where the
// shared-memory reads bound the cells (9 per sum): K u in FP32 on a 256^3 cube, linear basis,
// k_correct 221 against 234 us; at r = 2 the longer chains cost more than the reads.
//   y forward:   a_m [nx wy wz] -> E_g [nx ny wz]
template <typename T, int S, int R, int THREADS>
RK_DEV void box_forward_y(const T* am, int as, T* E, int es, int nx, int ny, int wy, int wz,
                          const T (*tab)[kDirectMaxReach + 1]) {
  using B = DBasis<S>;
  const int nh = (ny + 1) / 2;
  const unsigned rnx = box_inv(nx), rnh = box_inv(nh);
  for (int e = threadIdx.x; e < nx * nh * wz; e += THREADS) {
    const int t = box_div(e, rnx), x = e - t * nx, z = box_div(t, rnh), y = 2 * (t - z * nh);
    const bool two = y + 1 < ny;
#pragma unroll
    for (int m = 0; m < B::NX; ++m) {
      T v[2 * R + 2];
#pragma unroll
      for (int j = 0; j <= 2 * R + 1; ++j)
        v[j] = j <= 2 * R || two ? am[m * as + x + nx * (y + j + wy * z)] : (T)0;
#pragma unroll
      for (int g = 0; g < B::NG; ++g)
        if (B::gmx(g) == m) {
          T* o = E + g * es + x + nx * (y + ny * z);
          o[0] = conv1_m<R, 1>(B::gmy(g), v, R, tab);
          if (two) o[nx] = conv1_m<R, 1>(B::gmy(g), v, R + 1, tab);
        }
    }
  }
}
//   z reflected: g_p [wx wy wz] -> G_g [wx wy nz]
template <typename T, int S, int R, int THREADS>
RK_DEV void box_reflect_z(const T* g, int ps, T* G, int gs, int wx, int wy, int nz, const T (*tab)[kDirectMaxReach + 1]) {
  using B = DBasis<S>;
  const int nh = (nz + 1) / 2, wxy = wx * wy;
  const unsigned rwx = box_inv(wx), rwy = box_inv(wy);
  for (int e = threadIdx.x; e < wxy * nh; e += THREADS) {
    const int zh = box_div(box_div(e, rwx), rwy), i = e + zh * wxy;  // the node of z = 2 zh
    const bool two = 2 * zh + 1 < nz;
    T s[B::NG][2];
#pragma unroll
    for (int p = 0; p < S; ++p) {
      T v[2 * R + 2];
#pragma unroll
      for (int j = 0; j <= 2 * R + 1; ++j) v[j] = j <= 2 * R || two ? g[p * ps + i + j * wxy] : (T)0;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const T w = conv1_m<R, -1>(B::az(p), v, R + k, tab);
        s[B::grp(p)][k] = B::az(p) == 0 ? w : s[B::grp(p)][k] + w;  // (m_x, m_y, 0) comes first
      }
    }
#pragma unroll
    for (int k = 0; k < B::NG; ++k) {
      G[k * gs + i] = s[k][0];
      if (two) G[k * gs + i + wxy] = s[k][1];
    }
  }
}
//   y reflected: G_g [wx wy nz] -> F_m [wx ny nz]
template <typename T, int S, int R, int THREADS>
RK_DEV void box_reflect_y(const T* G, int gs, T* F, int fs, int wx, int wy, int ny, int nz,
                          const T (*tab)[kDirectMaxReach + 1]) {
  using B = DBasis<S>;
  const int nh = (ny + 1) / 2;
  const unsigned rwx = box_inv(wx), rnh = box_inv(nh);
  for (int e = threadIdx.x; e < wx * nh * nz; e += THREADS) {
    const int t = box_div(e, rwx), x = e - t * wx, z = box_div(t, rnh), y = 2 * (t - z * nh);
    const bool two = y + 1 < ny;
    T acc[B::NX][2];
#pragma unroll
    for (int k = 0; k < B::NG; ++k) {
      T v[2 * R + 2];
#pragma unroll
      for (int j = 0; j <= 2 * R + 1; ++j) v[j] = j <= 2 * R || two ? G[k * gs + x + wx * (y + j + wy * z)] : (T)0;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const T w = conv1_m<R, -1>(B::gmy(k), v, R + c, tab);
        acc[B::gmx(k)][c] = B::gmy(k) == 0 ? w : acc[B::gmx(k)][c] + w;
      }
    }
#pragma unroll
    for (int m = 0; m < B::NX; ++m) {
      T* o = F + m * fs + x + wx * (y + ny * z);
      o[0] = acc[m][0];
      if (two) o[wx] = acc[m][1];
    }
  }
}

// delta_p = g_p - c_p D_p on the nodes of a cell's bounding box: the forward sums of
// Eq. 86 along x, y and z in shared memory, then the pointwise stage.  One block per cell.
// Runs beside k_regular, on the issue slots and SMs that one leaves (a CG step: p is formed
// here again): a block of k_regular triggers after its own wait, so all that came before
// k_regular is complete once this kernel starts, and only the end of k_regular is waited for,
// at the end.  K in FP32, 256^3 cube: 239 -> 224 us in all, spheres in 256^3, quadratic basis,
// 336 -> 303 us, 162 x 100 x 72 68 -> 52 us; 128^3 mixed solve 32 -> 25 ms.
template <typename T, int S, int R>
struct DeltaSize {
  using B = DBasis<S>;
  static constexpr int W = kCell + 2 * R;
  static constexpr int ND = W * W * W, NA = B::NX * kCell * W * W, NE = B::NG * kCell * kCell * W;
  static constexpr size_t SMEM = sizeof(T) * (size_t)((ND > NE ? ND : NE) + NA);  // E takes the place of d
};
template <typename T, int S, int R, bool CG>
__global__ void __launch_bounds__(corr_threads<R>()) k_delta(const __grid_constant__ DirectArgs<T> a) {
  using B = DBasis<S>;
  using Z = DeltaSize<T, S, R>;
  RK_DYN_SMEM(T, sm);
  T* d = sm;
  T* E = sm;
  T* am = sm + (Z::ND > Z::NE ? Z::ND : Z::NE);
  const CorrCell c = a.ncell[blockIdx.x];
  const int nx = c.hi[0] - c.lo[0], ny = c.hi[1] - c.lo[1], nz = c.hi[2] - c.lo[2];
  const int wx = nx + 2 * R, wy = ny + 2 * R, wz = nz + 2 * R;
  const int x0 = c.c[0] * kCell + c.lo[0], y0 = c.c[1] * kCell + c.lo[1], z0 = c.c[2] * kCell + c.lo[2];
  const long long ps = (long long)a.nx * a.ny;
  const unsigned rnx = box_inv(nx), rny = box_inv(ny), rwx = box_inv(wx), rwy = box_inv(wy);
  grid_trigger();
  const T *in = a.in, *p_old = nullptr;
  T beta = (T)0;
  if constexpr (CG) {
    p_old = __ldcg(&a.cg->par) ? a.p1 : a.p0;
    beta = (T)__ldcg(&a.cg->beta);
  }
#pragma unroll 4
  for (int e = threadIdx.x; e < wx * wy * wz; e += corr_threads<R>()) {
    const int t = box_div(e, rwx), x = e - t * wx, z = box_div(t, rwy), y = t - z * wy;
    const long long i = wrap_once(x0 - R + x, a.nx) + (long long)a.nx * wrap_once(y0 - R + y, a.ny) + ps * wrap_once(z0 - R + z, a.nz);
    T v = __ldcg(in + i);
    if constexpr (CG) {
      v += beta * __ldcg(p_old + i);
    } else if (a.in_bits) {
      if (!(__ldg(a.flags + i) & a.in_bits)) v = (T)0;
    }
    d[e] = v;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < nx * wy * wz; e += corr_threads<R>()) {
    const int t = box_div(e, rnx), x = e - t * nx;  // t = y + wy z
    T v[2 * R + 1];
#pragma unroll
    for (int j = 0; j <= 2 * R; ++j) v[j] = d[t * wx + x + j];
#pragma unroll
    for (int m = 0; m < B::NX; ++m) am[m * (kCell * Z::W * Z::W) + e] = conv1_m<R, 1>(m, v, R, a.tab);
  }
  __syncthreads();
  const int nxy = nx * ny;
  if constexpr (R >= 4) {
    box_forward_y<T, S, R, corr_threads<R>()>(am, kCell * Z::W * Z::W, E, kCell * kCell * Z::W, nx, ny, wy, wz, a.tab);
  } else {
    for (int e = threadIdx.x; e < nxy * wz; e += corr_threads<R>()) {
      const int t = box_div(e, rnx), x = e - t * nx, z = box_div(t, rny), y = t - z * ny;
#pragma unroll
      for (int m = 0; m < B::NX; ++m) {
        T v[2 * R + 1];
#pragma unroll
        for (int j = 0; j <= 2 * R; ++j) v[j] = am[m * (kCell * Z::W * Z::W) + x + nx * (y + j + wy * z)];
#pragma unroll
        for (int g = 0; g < B::NG; ++g)
          if (B::gmx(g) == m) E[g * (kCell * kCell * Z::W) + e] = conv1_m<R, 1>(B::gmy(g), v, R, a.tab);
      }
    }
  }
  __syncthreads();
  T* out = a.delta + (long long)blockIdx.x * (S * kCell * kCell * kCell);
  for (int e = threadIdx.x; e < nxy * nz; e += corr_threads<R>()) {
    const int t = box_div(e, rnx), x = e - t * nx, z = box_div(t, rny), y = t - z * ny;
    const int cl = __ldg(a.cidx + x0 + x + (long long)a.nx * (y0 + y) + ps * (z0 + z));
    T* o = out + c.lo[0] + x + kCell * (c.lo[1] + y + kCell * (c.lo[2] + z));
    T D[S], g[S];
    if (cl == 0) {
#pragma unroll
      for (int p = 0; p < S; ++p) o[p * (kCell * kCell * kCell)] = (T)0;
      continue;
    }
#pragma unroll
    for (int gr = 0; gr < B::NG; ++gr) {
      T v[2 * R + 1];
#pragma unroll
      for (int j = 0; j <= 2 * R; ++j) v[j] = E[gr * (kCell * kCell * Z::W) + e + j * nxy];
#pragma unroll
      for (int p = 0; p < S; ++p)
        if (B::grp(p) == gr) D[p] = conv1_m<R, 1>(B::az(p), v, R, a.tab);
    }
    if (cl > 0) {
      constexpr int CP = ctab_pitch<T>(S);
      T co[CP];
      const Vec16<T>* src = reinterpret_cast<const Vec16<T>*>(a.ctab + (long long)(cl - 1) * CP);
#pragma unroll
      for (int k = 0; k < CP / (16 / (int)sizeof(T)); ++k) {
        const Vec16<T> raw = __ldg(src + k);
        memcpy(co + k * (16 / (int)sizeof(T)), &raw, 16);
      }
      pointwise_node<T, S>(co, cl, D, g);
    } else {
#pragma unroll
      for (int p = 0; p < S; ++p) g[p] = (T)0;
    }
#pragma unroll
    for (int p = 0; p < S; ++p) o[p * (kCell * kCell * kCell)] = p >= 1 && p <= 3 ? g[p] - a.creg[p - 1] * D[p] : g[p];
  }
  grid_wait();
}

// f += the reflected sums of delta on the outputs of a cell's bounding box, masked; in a CG
// step also p . (the correction).  One block per cell.  delta of the box and its halo is
// copied to shared memory at once (read where it is used, plane by plane, the latency of
// L2 bounded the kernel); the largest bases and reaches take it from L2.
template <typename T, int S, int R>
struct CorrectSize {
  using B = DBasis<S>;
  static constexpr int W = kCell + 2 * R;
  static constexpr int NG = B::NG * W * W * kCell, NF = B::NX * W * kCell * kCell, ND = S * W * W * W;
  static constexpr bool STAGED = sizeof(T) * (size_t)(ND + NG) <= 100 * 1024;
  static constexpr size_t SMEM = sizeof(T) * (size_t)(NG + (STAGED ? (ND > NF ? ND : NF) : NF));  // F takes the place of delta
};
template <typename T, int S, int R, bool CG>
__global__ void __launch_bounds__(corr_threads<R>()) k_correct(const __grid_constant__ DirectArgs<T> a) {
  using B = DBasis<S>;
  using Z = CorrectSize<T, S, R>;
  constexpr int W = Z::W, C3 = kCell * kCell * kCell;
  RK_DYN_SMEM(T, sm);
  T* G = sm;
  T* F = sm + Z::NG;
  T* dl = F;  // [p][wx wy wz]
  // nodes of the box are cut into cells of kCell; the last cell of an axis may be shorter, so
  // a node's cell comes from its wrapped index: per axis the place in the cell and the
  // number of cell borders since the first node of the halo, then the slots of those cells
  __shared__ signed char place[3][W], cellno[3][W];
  constexpr int MC = 5;  // cells a halo of W nodes can touch along an axis (the last one short)
  __shared__ int slots[MC * MC * MC];
  const int n[3] = {a.nx, a.ny, a.nz};
  DotAccPair<T> dot;
  // (a CG step has fewer blocks than cells: every block ends with its turn at the counter)
  for (int cell_no = blockIdx.x; cell_no < a.ocells; cell_no += gridDim.x) {
    const CorrCell c = a.ocell[cell_no];
    const int cn0 = (a.nx + kCell - 1) / kCell, cn1 = (a.ny + kCell - 1) / kCell;
    const int nx = c.hi[0] - c.lo[0], ny = c.hi[1] - c.lo[1], nz = c.hi[2] - c.lo[2];
    const int wx = nx + 2 * R, wy = ny + 2 * R, wz = nz + 2 * R;
    const int x0 = c.c[0] * kCell + c.lo[0], y0 = c.c[1] * kCell + c.lo[1], z0 = c.c[2] * kCell + c.lo[2];
    const long long ps = (long long)a.nx * a.ny;
    const unsigned rnx = box_inv(nx), rny = box_inv(ny), rwx = box_inv(wx), rwy = box_inv(wy);
    for (int e = threadIdx.x; e < 3 * W; e += corr_threads<R>()) {
      const int k = e / W, i = e % W;
      const int first = (k == 0 ? x0 : (k == 1 ? y0 : z0)) - R, len = k == 0 ? n[0] : (k == 1 ? n[1] : n[2]);
      int no = 0, v = wrap_once(first, len);
      for (int t = 0; t < i; ++t) {
        v = v + 1 == len ? 0 : v + 1;
        no += v % kCell == 0 ? 1 : 0;
      }
      place[k][i] = (signed char)(v % kCell);
      cellno[k][i] = (signed char)no;
    }
    __syncthreads();
    const int mx = cellno[0][wx - 1] + 1, my = cellno[1][wy - 1] + 1, mz = cellno[2][wz - 1] + 1;
    for (int e = threadIdx.x; e < mx * my * mz; e += corr_threads<R>()) {
      const int i = e % mx, j = e / mx % my, k = e / (mx * my);
      auto cell = [&](int first, int len, int no) {  // the cell `no` borders after that of the first node
        const int f = wrap_once(first, len) / kCell + no, m = (len + kCell - 1) / kCell;
        return f % m;
      };
      slots[(k * MC + j) * MC + i] =
          __ldg(a.slot + cell(x0 - R, a.nx, i) + cn0 * (cell(y0 - R, a.ny, j) + (long long)cn1 * cell(z0 - R, a.nz, k)));
    }
    __syncthreads();
    auto source = [&](int x, int y, int z) -> const T* {  // delta_0 at a node of the halo (null: zero)
      const int s = slots[(cellno[2][z] * MC + cellno[1][y]) * MC + cellno[0][x]];
      return s < 0 ? nullptr : a.delta + (long long)s * (S * C3) + place[0][x] + kCell * (place[1][y] + kCell * place[2][z]);
    };
    const int wxy = wx * wy, wn = wxy * wz;
    if (cell_no == (int)blockIdx.x) {
      grid_wait();
      grid_trigger();
    }
    if constexpr (Z::STAGED) {
#pragma unroll 2
      for (int e = threadIdx.x; e < wn; e += corr_threads<R>()) {
        const int t = box_div(e, rwx), x = e - t * wx, z = box_div(t, rwy), y = t - z * wy;
        const T* src = source(x, y, z);
#pragma unroll
        for (int p = 0; p < S; ++p) {
          if (src)
            cp_async_value(dl + p * (W * W * W) + e, src + p * C3);
          else
            dl[p * (W * W * W) + e] = (T)0;
        }
      }
      cp_async_commit();
      cp_async_wait<0>();
      __syncthreads();
    }
    // z: G(z) += T(o) delta(z + o)
    if constexpr (R >= 4 && Z::STAGED) {
      box_reflect_z<T, S, R, corr_threads<R>()>(dl, W * W * W, G, W * W * kCell, wx, wy, nz, a.tab);
    } else {
      for (int e = threadIdx.x; e < wxy * nz; e += corr_threads<R>()) {
        T g[B::NG];
#pragma unroll
        for (int k = 0; k < B::NG; ++k) g[k] = (T)0;
        const int t = box_div(e, rwx), x = e - t * wx, z = box_div(t, rwy), y = t - z * wy;
#pragma unroll
        for (int o = -R; o <= R; ++o) {
          const int u = o < 0 ? -o : o;
          T v[S];
          if constexpr (Z::STAGED) {
#pragma unroll
            for (int p = 0; p < S; ++p) v[p] = dl[p * (W * W * W) + e + (o + R) * wxy];
          } else {
            const T* src = source(x, y, z + o + R);
#pragma unroll
            for (int p = 0; p < S; ++p) v[p] = src ? __ldcg(src + p * C3) : (T)0;
          }
#pragma unroll
          for (int p = 0; p < S; ++p) {
            const int m = B::az(p);
            if (m != 0 && o == 0) continue;
            g[B::grp(p)] += (m == 1 && o < 0 ? -a.tab[m][u] : a.tab[m][u]) * v[p];
          }
        }
#pragma unroll
        for (int k = 0; k < B::NG; ++k) G[k * (W * W * kCell) + e] = g[k];
      }
    }
    __syncthreads();
    if constexpr (R >= 4) {
      box_reflect_y<T, S, R, corr_threads<R>()>(G, W * W * kCell, F, W * kCell * kCell, wx, wy, ny, nz, a.tab);
    } else {
      for (int e = threadIdx.x; e < wx * ny * nz; e += corr_threads<R>()) {
        const int t = box_div(e, rwx), x = e - t * wx, z = box_div(t, rny), y = t - z * ny;
        T acc[B::NX];
#pragma unroll
        for (int k = 0; k < B::NG; ++k) {
          T v[2 * R + 1];
#pragma unroll
          for (int j = 0; j <= 2 * R; ++j) v[j] = G[k * (W * W * kCell) + x + wx * (y + j + wy * z)];
          const T w = conv1_m<R, -1>(B::gmy(k), v, R, a.tab);
          acc[B::gmx(k)] = B::gmy(k) == 0 ? w : acc[B::gmx(k)] + w;
        }
#pragma unroll
        for (int m = 0; m < B::NX; ++m) F[m * (W * kCell * kCell) + e] = acc[m];
      }
    }
    __syncthreads();
    const T* p = nullptr;
    if constexpr (CG) p = a.cg->par ? a.p0 : a.p1;
    for (int e = threadIdx.x; e < nx * ny * nz; e += corr_threads<R>()) {
      const int t = box_div(e, rnx), x = e - t * nx, z = box_div(t, rny), y = t - z * ny;
      const long long i = x0 + x + (long long)a.nx * (y0 + y) + ps * (z0 + z);
      if (!(__ldg(a.flags + i) & a.out_bits)) continue;
      const T f = a.out[i];
      T pv = (T)0;
      if constexpr (CG) pv = __ldcg(p + i);
      T acc = (T)0;
#pragma unroll
      for (int m = 0; m < B::NX; ++m) {
        T v[2 * R + 1];
#pragma unroll
        for (int j = 0; j <= 2 * R; ++j) v[j] = F[m * (W * kCell * kCell) + x + j + wx * t];
        const T w = conv1_m<R, -1>(m, v, R, a.tab);
        acc = m == 0 ? w : acc + w;
      }
      a.out[i] = f + acc;
      if constexpr (CG) dot.add(cmk(pv, (T)0), cmk(acc, (T)0));
    }
    __syncthreads();
  }
  if constexpr (CG) direct_pap_reduce<corr_threads<R>()>(dot, a);
}

}  // namespace rk
