// k_push.cu -- the particle step: gather at both bodies, internal
// modified-Coulomb field, relativistic Boris push of both bodies, drift and
// Esirkepov (quadratic shape) current deposit.
//
// Method: arXiv 2208.08038 Sec. 2 (two-body macro-ion, Boris equations,
// modified Coulomb force, body currents q v / dV).  Per step:
//   k_push_quiet  tiles whose neighbourhood never held a field (the field
//                 kernels' tile marks): their co-moving neutral ions only
//                 drift; the other tiles go on a list for the push,
//   k_push_few    2D grids with few ions: the tiles with few, without a box,
//   k_push        persistent blocks walk that list; per tile:
//     1. stage E and B of the tile plus halo in shared memory (FP32, by
//        asynchronous copies issued while the block finishes the previous
//        tile),
//     2. push every particle of the tile (all species), accumulating the
//        current of both bodies in a shared-memory box (tile + halo).  A
//        particle whose bodies keep their nearest nodes deposits three-node
//        windows, the others four-node windows body by body.  The box holds
//          BP_DEPOSIT_SORTED: 64-bit fixed point (integer adds are
//                             associative: the same sums in any order),
//          BP_DEPOSIT_ATOMIC: FP32 shared atomics,
//     3. sorted mode: add every non-zero node of the box to the global 64-bit
//        fixed-point current (and before, when its words may fill); atomic mode: write the box to the tile's slot
//        for the current-sum kernel,
//   k_push_far    sorted mode: the ions k_push left on the far list (a bound
//                 electron a cell or more from its nucleus), pushed with the
//                 global fields and deposited into the global current,
//                 and (tile_active) the tiles the field kernels update this
//                 step: those whose neighbourhood has held a field or holds
//                 moved particles, those next to an antenna plane, every tile
//                 after a far push.
#include <type_traits>

#include "bp_internal.cuh"
#include "bp_particle.cuh"

namespace {

// threads of a push block
__host__ __device__ constexpr int push_threads(int D) { return D == 3 ? 512 : 256; }
// and the blocks per SM its registers are held to (see k_push)
__host__ __device__ constexpr int push_pb(int D, bool free_sp) { return D == 2 ? (free_sp ? 3 : 2) : 1; }

// Where a deposit goes: the tile's box in shared memory, or (tiles with few
// ions in 2D, sorted mode) straight to the global fixed-point current, whose row and
// component strides are the grid's.
template <int D>
struct BoxStride {
  static constexpr int row = Box<D>::J0, comp = Box<D>::JCELLS;
};
struct GridStride {
  int row;
  long long comp;
};
using fx64 = unsigned long long;  // a node of the global fixed-point current

// add v (already in fixed-point units in the sorted mode) to a current node:
// sorted mode, the exact fixed-point add fx_add (low words of the box, high
// words 3 * JCELLS entries later); atomic mode, an FP32 shared atomic.  Zero
// contributions are skipped where SKIP0.
template <int D, bool DET, bool SKIP0 = true, typename JT>
__device__ __forceinline__ void jput(JT *p, float v) {
  if constexpr (std::is_same<JT, fx64>::value) {
    if (fabsf(v) > 0.5f) atomicAdd(p, (fx64)f2ll_rn(v));
  } else if constexpr (DET) {
    if (SKIP0 && fabsf(v) <= 0.5f) return;
    fx_add(p, 3 * Box<D>::JCELLS, v);
  } else {
    if (SKIP0 && v == 0.0f) return;
    atomicAdd(p, v);
  }
}

template <int D, bool DET, typename JT>
__device__ __forceinline__ void jadd(JT *p, float v, float scale) {
  jput<D, DET>(p, DET ? v * scale : v);
}

// jput of a rows x cols block of nodes (the sorted mode's high words under one
// branch)
template <int D, bool DET, int R, int C, typename JT, typename ST>
__device__ __forceinline__ void jput_block(JT *p, const float (*v)[C], const ST &st) {
  if constexpr (std::is_same<JT, fx64>::value) {
#pragma unroll
    for (int j = 0; j < R; ++j)
#pragma unroll
      for (int i = 0; i < C; ++i) jput<D, DET>(p + (long long)st.row * j + i, v[j][i]);
  } else if constexpr (DET) {
    fx_add_block<R, C>(p, Box<D>::J0, 3 * Box<D>::JCELLS, v);
  } else {
#pragma unroll
    for (int j = 0; j < R; ++j)
#pragma unroll
      for (int i = 0; i < C; ++i) atomicAdd(p + Box<D>::J0 * j + i, v[j][i]);
  }
}

// Fast path: all four positions (both bodies, before and after the move)
// share one nearest node per axis, so the window is the three nodes around
// it and S1 - S0 has a closed form in the move d (no cancellation):
//   node n-1: -d (1 - 2 xi - d) / 2,  node n: -d (2 xi + d),  node n+1: d (1 + 2 xi + d) / 2
// with xi = old position - n.  J along a simulated axis then lives on the two
// faces inside the window, with partial sums DS(n-1) and DS(n-1) + DS(n) =
// -DS(n+1).  The Esirkepov factor of the two transverse axes is written
//   S0y S0z + (DSy S0z + S0y DSz)/2 + DSy DSz/3 = Ay Az + DSy DSz/12,
// A = S0 + DS/2 the mid-step shape.  In the sorted mode the charge factors
// carry the fixed-point scale (a power of two, so the products round
// exactly as unscaled ones).  The two bodies' terms are added without FMA
// contraction so that a neutral pair moving together cancels exactly.
template <int D, bool DET, int NB, typename JT, typename ST = BoxStride<D>>
__device__ __forceinline__ void esirkepov3(JT *__restrict__ J, const int n[3], const float (*xi)[3],
                                           const float (*de)[3], const float *qw, const float (*v)[3],
                                           const float dxdt[3], float scale, const ST &st = ST()) {
  constexpr float K12 = 1.0f / 12.0f;
  const float sc = DET ? scale : 1.0f;
  float A[NB][3][3], DS[NB][3][3], DK[NB][3][3], cP[NB][3][2];
#pragma unroll
  for (int b = 0; b < NB; ++b)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if (a < D) {
        const float x = xi[b][a], d = de[b][a];
        float S0[3];
        qweights(x, S0);
        const float d0 = -0.5f * d * (1.0f - 2.0f * x - d);
        const float d1 = -d * (2.0f * x + d);
        const float d2 = 0.5f * d * (1.0f + 2.0f * x + d);
        A[b][a][0] = fmaf(0.5f, d0, S0[0]);
        A[b][a][1] = fmaf(0.5f, d1, S0[1]);
        A[b][a][2] = fmaf(0.5f, d2, S0[2]);
        DS[b][a][0] = d0;
        DS[b][a][1] = d1;
        DS[b][a][2] = d2;
        DK[b][a][0] = K12 * d0;
        DK[b][a][1] = K12 * d1;
        DK[b][a][2] = K12 * d2;
        const float c = -qw[b] * dxdt[a] * sc;
        cP[b][a][0] = c * d0;
        cP[b][a][1] = -c * d2;
      } else {
        A[b][a][0] = A[b][a][2] = 0.0f;
        A[b][a][1] = 1.0f;
        DS[b][a][0] = DS[b][a][1] = DS[b][a][2] = 0.0f;
        DK[b][a][0] = DK[b][a][1] = DK[b][a][2] = 0.0f;
        cP[b][a][0] = cP[b][a][1] = 0.0f;
      }
    }
  JT *Jx = J, *Jy = J + st.comp, *Jz = J + 2 * st.comp;
  const int bx = n[0] - 1, by = n[1] - 1, bz = n[2] - 1;
  if constexpr (D == 1) {
    float x[1][2], y[1][3], z[1][3], qy[NB], qz[NB];
#pragma unroll
    for (int f = 0; f < 2; ++f) {
      x[0][f] = cP[0][0][f];
      if constexpr (NB == 2) x[0][f] = __fadd_rn(x[0][f], cP[1][0][f]);
    }
    jput_block<D, DET, 1, 2>(Jx + bx, x, st);
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      qy[b] = qw[b] * v[b][1] * sc;
      qz[b] = qw[b] * v[b][2] * sc;
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      y[0][i] = __fmul_rn(qy[0], A[0][0][i]);
      z[0][i] = __fmul_rn(qz[0], A[0][0][i]);
      if constexpr (NB == 2) {
        y[0][i] = __fadd_rn(y[0][i], __fmul_rn(qy[1], A[1][0][i]));
        z[0][i] = __fadd_rn(z[0][i], __fmul_rn(qz[1], A[1][0][i]));
      }
    }
    jput_block<D, DET, 1, 3>(Jy + bx, y, st);
    jput_block<D, DET, 1, 3>(Jz + bx, z, st);
  } else if constexpr (D == 2) {
    float x[3][2], y[2][3], z[3][3], qz[NB];
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int f = 0; f < 2; ++f) {
        x[j][f] = __fmul_rn(cP[0][0][f], A[0][1][j]);
        if constexpr (NB == 2) x[j][f] = __fadd_rn(x[j][f], __fmul_rn(cP[1][0][f], A[1][1][j]));
      }
    jput_block<D, DET, 3, 2>(Jx + (bx + (long long)st.row * by), x, st);
#pragma unroll
    for (int g = 0; g < 2; ++g)
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        y[g][i] = __fmul_rn(cP[0][1][g], A[0][0][i]);
        if constexpr (NB == 2) y[g][i] = __fadd_rn(y[g][i], __fmul_rn(cP[1][1][g], A[1][0][i]));
      }
    jput_block<D, DET, 2, 3>(Jy + (bx + (long long)st.row * by), y, st);
#pragma unroll
    for (int b = 0; b < NB; ++b) qz[b] = qw[b] * v[b][2] * sc;
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        z[j][i] = __fmul_rn(qz[0], fmaf(A[0][0][i], A[0][1][j], DK[0][0][i] * DS[0][1][j]));
        if constexpr (NB == 2)
          z[j][i] = __fadd_rn(z[j][i], __fmul_rn(qz[1], fmaf(A[1][0][i], A[1][1][j], DK[1][0][i] * DS[1][1][j])));
      }
    jput_block<D, DET, 3, 3>(Jz + (bx + (long long)st.row * by), z, st);
  } else {
    // The outer loop of each pass stays rolled (its weights picked by
    // selects): the fully unrolled 54-node form is about three times the
    // code, and the kernel's hot path then outgrows the instruction caches.
#pragma unroll 1
    for (int k = 0; k < 3; ++k) {
      float azk[NB], dzk[NB];
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        azk[b] = k == 0 ? A[b][2][0] : (k == 1 ? A[b][2][1] : A[b][2][2]);
        dzk[b] = k == 0 ? DS[b][2][0] : (k == 1 ? DS[b][2][1] : DS[b][2][2]);
      }
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        float F[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) F[b] = fmaf(A[b][1][j], azk[b], DK[b][1][j] * dzk[b]);
#pragma unroll
        for (int f = 0; f < 2; ++f) {
          float jx = __fmul_rn(cP[0][0][f], F[0]);
          if constexpr (NB == 2) jx = __fadd_rn(jx, __fmul_rn(cP[1][0][f], F[1]));
          jput<D, DET, false>(Jx + Box<D>::ji(bx + f, by + j, bz + k), jx);
        }
      }
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        float F[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) F[b] = fmaf(A[b][0][i], azk[b], DK[b][0][i] * dzk[b]);
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          float jy = __fmul_rn(cP[0][1][g], F[0]);
          if constexpr (NB == 2) jy = __fadd_rn(jy, __fmul_rn(cP[1][1][g], F[1]));
          jput<D, DET, false>(Jy + Box<D>::ji(bx + i, by + g, bz + k), jy);
        }
      }
    }
#pragma unroll 1
    for (int j = 0; j < 3; ++j) {
      float ayj[NB], dyj[NB];
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        ayj[b] = j == 0 ? A[b][1][0] : (j == 1 ? A[b][1][1] : A[b][1][2]);
        dyj[b] = j == 0 ? DS[b][1][0] : (j == 1 ? DS[b][1][1] : DS[b][1][2]);
      }
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        float F[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) F[b] = fmaf(A[b][0][i], ayj[b], DK[b][0][i] * dyj[b]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float jz = __fmul_rn(cP[0][2][h], F[0]);
          if constexpr (NB == 2) jz = __fadd_rn(jz, __fmul_rn(cP[1][2][h], F[1]));
          jput<D, DET, false>(Jz + Box<D>::ji(bx + i, by + j, bz + h), jz);
        }
      }
    }
  }
}

__device__ __forceinline__ float2 sel3(int k, const float2 *a) { return k == 0 ? a[0] : (k == 1 ? a[1] : a[2]); }

// esirkepov3 for a two-body ion in 3D, sorted mode, on Blackwell's packed
// FP32 pairs (FFMA2): the two bodies in the lanes of every setup term and of
// each row's transverse factor F; a node's value is the bodies' two products
// (one packed multiply) added, and six nodes at a time go through the packed
// fixed-point split (fx_add6).  The outer loops stay rolled as in the scalar
// form (code size).
__device__ __forceinline__ void esirkepov3_p3(unsigned int *__restrict__ J, const int n[3], const float (*xi)[3],
                                              const float (*de)[3], const float *qw, const float dxdt[3],
                                              float scale) {
  constexpr int jcells = Box<3>::JCELLS;
  constexpr int hoff = 3 * jcells;
  const float2 K12 = make_float2(1.0f / 12.0f, 1.0f / 12.0f), H = make_float2(0.5f, 0.5f);
  const float2 M1 = make_float2(-1.0f, -1.0f), ONE = make_float2(1.0f, 1.0f);
  float2 A[3][3], DS[3][3], DK[3][3], cP[3][2];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float2 x = make_float2(xi[0][a], xi[1][a]), d = make_float2(de[0][a], de[1][a]);
    float2 S0[3];
    qweights2(x, S0);
    const float2 u = __fadd2_rn(__fadd2_rn(x, x), d);
    float2 dd[3];
    dd[0] = __fmul2_rn(__fmul2_rn(d, make_float2(-0.5f, -0.5f)), __ffma2_rn(u, M1, ONE));
    dd[1] = __fmul2_rn(__fmul2_rn(d, M1), u);
    dd[2] = __fmul2_rn(__fmul2_rn(d, H), __fadd2_rn(u, ONE));
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      A[a][i] = __ffma2_rn(H, dd[i], S0[i]);
      DS[a][i] = dd[i];
      DK[a][i] = __fmul2_rn(K12, dd[i]);
    }
    const float2 c = make_float2(-qw[0] * dxdt[a] * scale, -qw[1] * dxdt[a] * scale);
    cP[a][0] = __fmul2_rn(c, dd[0]);
    cP[a][1] = __fmul2_rn(__fmul2_rn(c, M1), dd[2]);
  }
  unsigned int *Jx = J, *Jy = J + jcells, *Jz = J + 2 * jcells;
  const int bx = n[0] - 1, by = n[1] - 1, bz = n[2] - 1;
#pragma unroll 1
  for (int k = 0; k < 3; ++k) {
    const float2 az = sel3(k, A[2]), dz = sel3(k, DS[2]);
    unsigned int *p = Jx + Box<3>::ji(bx, by, bz + k);
    float2 v[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const float2 F = __ffma2_rn(A[1][j], az, __fmul2_rn(DK[1][j], dz));
      const float2 t0 = __fmul2_rn(cP[0][0], F), t1 = __fmul2_rn(cP[0][1], F);
      v[j] = make_float2(__fadd_rn(t0.x, t0.y), __fadd_rn(t1.x, t1.y));
    }
    fx_add6(p, Box<3>::J0, 1, hoff, v);
    p = Jy + Box<3>::ji(bx, by, bz + k);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const float2 F = __ffma2_rn(A[0][i], az, __fmul2_rn(DK[0][i], dz));
      const float2 t0 = __fmul2_rn(cP[1][0], F), t1 = __fmul2_rn(cP[1][1], F);
      v[i] = make_float2(__fadd_rn(t0.x, t0.y), __fadd_rn(t1.x, t1.y));
    }
    fx_add6(p, 1, Box<3>::J0, hoff, v);
  }
#pragma unroll 1
  for (int j = 0; j < 3; ++j) {
    const float2 ay = sel3(j, A[1]), dy = sel3(j, DS[1]);
    unsigned int *p = Jz + Box<3>::ji(bx, by + j, bz);
    float2 v[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const float2 F = __ffma2_rn(A[0][i], ay, __fmul2_rn(DK[0][i], dy));
      const float2 t0 = __fmul2_rn(cP[2][0], F), t1 = __fmul2_rn(cP[2][1], F);
      v[i] = make_float2(__fadd_rn(t0.x, t0.y), __fadd_rn(t1.x, t1.y));
    }
    fx_add6(p, 1, Box<3>::JP, hoff, v);
  }
}

// General case of one body: its nearest node changes along some axis in this
// step, or the ion's two bodies have different nearest nodes.  Old and new
// shapes then span four nodes per axis (three where the node stays): node m of
// the window is base + m, base = n0 - 1, or n0 - 2 along an axis crossed
// downwards (n0 the old nearest node).  Along an axis that is not crossed the
// difference of the shapes has the closed form of the fast path; a crossed
// axis takes the difference of the two shapes, every node of which changes
// its polynomial piece.  The current of a face is the running sum of the
// differences, whose last one is minus the last difference.
//
// Bound by the shared-memory adds (40 in 2D); the body of a fast particle
// needs 21.  It replaces five-node records in a global buffer added by a
// kernel of its own, and a single thread's 75 rows from local memory once the
// buffer was full: 4.2 M electrons, many of them crossing in a strong pulse,
// push and records 1.07 ms a step before, 0.43 after; 32.5 M thermal ions in
// 3D, 4.26 ms before, 3.60 after (one record took its lane as long as several
// particles).
struct GenAxis {
  float A[4], DS[4], P[3];  // mid-step shape S0 + DS / 2, shape difference, face currents (charge factor included)
  int base;                 // window's first node relative to the cell
};
__device__ __forceinline__ GenAxis general_axis(float f, float de, float c) {
  GenAxis g;
  const float up = f >= 0.5f ? 1.0f : 0.0f;
  const float x = f - up, x1 = x + de;
  const bool hi = x1 >= 0.5f, lo = x1 < -0.5f;
  float w[3], W[3], d3[3];
  qweights(x, w);
  qweights(hi ? x1 - 1.0f : x1 + 1.0f, W);
  d3[0] = -0.5f * de * (1.0f - 2.0f * x - de);
  d3[1] = -de * (2.0f * x + de);
  d3[2] = 0.5f * de * (1.0f + 2.0f * x + de);
  g.DS[0] = hi ? -w[0] : (lo ? W[0] : d3[0]);
  g.DS[1] = hi ? W[0] - w[1] : (lo ? W[1] - w[0] : d3[1]);
  g.DS[2] = hi ? W[1] - w[2] : (lo ? W[2] - w[1] : d3[2]);
  g.DS[3] = hi ? W[2] : (lo ? -w[2] : 0.0f);
  g.A[0] = fmaf(0.5f, g.DS[0], lo ? 0.0f : w[0]);
  g.A[1] = fmaf(0.5f, g.DS[1], lo ? w[0] : w[1]);
  g.A[2] = fmaf(0.5f, g.DS[2], lo ? w[1] : w[2]);
  g.A[3] = fmaf(0.5f, g.DS[3], lo ? w[2] : 0.0f);
  g.P[0] = c * g.DS[0];
  g.P[1] = c * (g.DS[0] + g.DS[1]);
  g.P[2] = -c * g.DS[3];
  g.base = (int)up - 1 - (lo ? 1 : 0);
  return g;
}

// The same axis for an ion's body, in the arithmetic of the shape functions
// (qshape, qshape_delta) node by node: the terms of a co-moving neutral pair
// cancel to rounding, so how each is rounded shows in the sum.  Without
// branches: a node's difference is the closed form of the piece that old and
// new position share, else the difference of the two shapes.
struct PairAxis {
  float S[4], DS[4], P[4];  // old shape, shape difference, running sums of the differences times the charge factor
  int base;
};
// old nearest node's offset up, position x from it, and the window's first node
// o relative to it
__device__ __forceinline__ void pair_place(float f, float d, float &x, int &up, int &o) {
  up = f >= 0.5f ? 1 : 0;
  x = f - (float)up;
  o = x + d < -0.5f ? -2 : -1;
}
// old shape S and shape difference DS of the node k away from the old nearest one
__device__ __forceinline__ void pair_node(float x, float d, int k, float &S, float &DS) {
  const float u = x - (float)k, v = u + d;
  const float au = fabsf(u), av = fabsf(v);
  const float tu = 1.5f - au, tv = 1.5f - av;
  const float cu = fmaf(-u, u, 0.75f), cv = fmaf(-v, v, 0.75f);
  const float su = au <= 0.5f ? cu : (au < 1.5f ? __fmul_rn(__fmul_rn(0.5f, tu), tu) : 0.0f);
  const float sv = av <= 0.5f ? cv : (av < 1.5f ? __fmul_rn(__fmul_rn(0.5f, tv), tv) : 0.0f);
  const bool mid = au <= 0.5f && av <= 0.5f, right = u > 0.5f && v > 0.5f && u < 1.5f && v < 1.5f,
             left = u < -0.5f && v < -0.5f && u > -1.5f && v > -1.5f;
  const float w = mid ? u + v : (right ? __fsub_rn(__fsub_rn(3.0f, u), v) : __fadd_rn(__fadd_rn(3.0f, u), v));
  const float h = mid ? -d : (right ? __fmul_rn(-0.5f, d) : __fmul_rn(0.5f, d));
  S = su;
  DS = mid || right || left ? __fmul_rn(h, w) : __fsub_rn(sv, su);
}
__device__ __forceinline__ PairAxis pair_axis(float f, float d, float c) {
  PairAxis g;
  float x, run = 0.0f;
  int up, o;
  pair_place(f, d, x, up, o);
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    pair_node(x, d, o + m, g.S[m], g.DS[m]);
    run = __fadd_rn(run, g.DS[m]);
    g.P[m] = __fmul_rn(c, run);
  }
  if (o == -1) g.P[3] = 0.0f;  // no face beyond the nodes n0 - 2 .. n0 + 2
  g.base = up + o;
  return g;
}
// the Esirkepov factor of the two axes transverse to a component
__device__ __forceinline__ float pair_factor(float sp, float dp, float sq, float dq) {
  return sp * sq + 0.5f * (dp * sq + sp * dq) + (1.0f / 3.0f) * dp * dq;
}

__device__ __forceinline__ float sel4(int k, const float *a) {
  return k == 0 ? a[0] : (k == 1 ? a[1] : (k == 2 ? a[2] : a[3]));
}

// 1D and 2D: a free particle (and, body by body, the ions of a 2D grid with free
// particles, whose kernel has no registers left for the other form)
template <int D, bool DET, typename JT>
__device__ __forceinline__ void deposit_general(JT *__restrict__ J, const int d[3], const float f[3], const float de[3],
                                                float qw, const float v[3], const float dxdt[3], float scale) {
  static_assert(D < 3, "3D: deposit_general3");
  constexpr int jcells = Box<D>::JCELLS;
  constexpr float K12 = 1.0f / 12.0f;
  const float q = DET ? qw * scale : qw;
  JT *Jx = J, *Jy = J + jcells, *Jz = J + 2 * jcells;
  const GenAxis X = general_axis(f[0], de[0], -q * dxdt[0]);
  if constexpr (D == 1) {
    const int b0 = d[0] + Box<D>::OJ + X.base;
    const float qy = q * v[1], qz = q * v[2];
#pragma unroll
    for (int i = 0; i < 3; ++i) jput<D, DET>(Jx + b0 + i, X.P[i]);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      jput<D, DET>(Jy + b0 + i, qy * X.A[i]);
      jput<D, DET>(Jz + b0 + i, qz * X.A[i]);
    }
  } else {
    const GenAxis Y = general_axis(f[1], de[1], -q * dxdt[1]);
    const float qz = q * v[2];
    const int b0 = Box<D>::ji(d[0] + Box<D>::OJ + X.base, d[1] + Box<D>::OJ + Y.base, 0);
    // rows rolled (code size: the loop competes with the fast path for the
    // instruction cache)
#pragma unroll 1
    for (int j = 0; j < 4; ++j) {
      const float ay = sel4(j, Y.A), dy = K12 * sel4(j, Y.DS);
      const int r = b0 + Box<D>::ji(0, j, 0);
#pragma unroll
      for (int i = 0; i < 3; ++i) jput<D, DET>(Jx + r + i, X.P[i] * ay);
#pragma unroll
      for (int i = 0; i < 4; ++i) jput<D, DET>(Jz + r + i, qz * fmaf(X.A[i], ay, X.DS[i] * dy));
      if (j < 3) {
        const float py = j == 0 ? Y.P[0] : (j == 1 ? Y.P[1] : Y.P[2]);
#pragma unroll
        for (int i = 0; i < 4; ++i) jput<D, DET>(Jy + r + i, py * X.A[i]);
      }
    }
  }
}

// an ion in 1D and 2D (rare: its bodies stay close to each other and slow), both
// bodies one after the other, out of line
template <int D, bool DET, typename JT, typename ST = BoxStride<D>>
__device__ __noinline__ void deposit_general_pair(JT *__restrict__ J, const int *d1, const int *d2, const float *f1,
                                                  const float *f2, const float *e1, const float *e2, float qw1,
                                                  float qw2, const float *v1, const float *v2, const float *dxdt,
                                                  float scale, const ST st = ST()) {
#pragma unroll 1
  for (int b = 0; b < 2; ++b) {
    const float q = (b ? qw2 : qw1) * (DET ? scale : 1.0f);
    const float *v = b ? v2 : v1;
    PairAxis G[2];
    int n0[2] = {0, 0};
#pragma unroll
    for (int a = 0; a < D; ++a) {
      G[a] = pair_axis(b ? f2[a] : f1[a], b ? e2[a] : e1[a], -q * dxdt[a]);
      n0[a] = (b ? d2[a] : d1[a]) + Box<D>::OJ + G[a].base;
    }
    const PairAxis &X = G[0], &Y = G[1];
    const float qy = q * v[1], qz = q * v[2];
    JT *p = J + (n0[0] + (long long)st.row * (D == 2 ? n0[1] : 0));
#pragma unroll 1
    for (int j = 0; j < (D == 2 ? 4 : 1); ++j, p += st.row) {
      const float sy = D == 2 ? sel4(j, Y.S) : 1.0f, dy = D == 2 ? sel4(j, Y.DS) : 0.0f, py = D == 2 ? sel4(j, Y.P) : 0.0f;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float fx = pair_factor(X.S[i], X.DS[i], 1.0f, 0.0f);
        jput<D, DET>(p + i, X.P[i] * pair_factor(sy, dy, 1.0f, 0.0f));
        jput<D, DET>(p + st.comp + i, D == 2 ? py * fx : qy * fx);
        jput<D, DET>(p + 2 * st.comp + i, qz * pair_factor(X.S[i], X.DS[i], sy, dy));
      }
    }
  }
}

// one particle's deposit inputs, handed to its warp in shared memory (by value
// they cost the push its registers: 3D, 32.5 M ions, 3.75 ms a step by value,
// 3.60 this way)
struct PairJob {
  float f[2][3], e[2][3];  // the bodies' offsets and moves
  int d[2][3];             // their cells relative to the tile
  float q[2][3];           // minus charge factor times dx / dt along each axis
  int two;
};

// 3D: the whole warp shares out one such particle, first a node of a body's axis per lane (24 of them), then the rows of
// both bodies, three a lane.  A thermal medium has one such particle in some 15
// warps; alone, its lane's chain of some 3,000 dependent instructions held the
// warp as long as several runs of particles, and the tile with it when it came
// in one of the last runs.
template <bool DET, typename JT>
__device__ __noinline__ void deposit_general3_warp(JT *__restrict__ J, const PairJob *job) {
  constexpr unsigned ALL = 0xFFFFFFFFu;
  const PairJob &P = *job;
  const int lane = threadIdx.x & 31;
  // lanes 12 b + 4 a + m: node m of axis a of body b (the last eight lanes repeat)
  const int nl = lane < 24 ? lane : lane - 24, nbody = nl / 12, naxis = (nl % 12) >> 2;
  float x, S, DS;
  int up, o;
  const float d = P.e[nbody][naxis];
  pair_place(P.f[nbody][naxis], d, x, up, o);
  pair_node(x, d, o + (nl & 3), S, DS);
  const int base = P.d[nbody][naxis] + Box<3>::OJ + up + o;  // the window's first node along this lane's axis
#pragma unroll
  for (int w = 0; w < 3; ++w) {
    const int it = lane + 32 * w, b = it / 48, r = it - 48 * b, c = r >> 4, j = r & 3, k = (r >> 2) & 3;
    const int p = c == 0 ? 1 : 0, q = c == 2 ? 1 : 2;  // the other two axes
    const int lb = 12 * b, lc = lb + 4 * c, lp = lb + 4 * p + j, lq = lb + 4 * q + k;
    const float F = pair_factor(__shfl_sync(ALL, S, lp), __shfl_sync(ALL, DS, lp), __shfl_sync(ALL, S, lq),
                                __shfl_sync(ALL, DS, lq));
    const int n0 = __shfl_sync(ALL, base, lb), n1 = __shfl_sync(ALL, base, lb + 4), n2 = __shfl_sync(ALL, base, lb + 8);
    const int oc = __shfl_sync(ALL, o, lc);
    const int sc = c == 0 ? 1 : (c == 1 ? Box<3>::J0 : Box<3>::JP);
    JT *row = J + c * Box<3>::JCELLS + Box<3>::ji(n0, n1, n2) + j * (c == 0 ? Box<3>::J0 : 1) +
              k * (c == 2 ? Box<3>::J0 : Box<3>::JP);
    const float cq = P.q[b][c];
    float run = 0.0f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      run = __fadd_rn(run, __shfl_sync(ALL, DS, lc + i));
      const float v = __fmul_rn(__fmul_rn(cq, run), F);
      if ((i < 3 || oc == -2) && (b == 0 || P.two)) jput<3, DET>(row + i * sc, v);
    }
  }
}

// W lanes work on one far body: the whole warp on one after the other of an
// ion's bodies (32), a half warp on each (16, 1D and 2D), or one thread on both
// (1).  lanes: the deposit of a far body (a bound electron a cell or more from
// its nucleus, or that nucleus), four-node windows as above
// around its own cell c, each node's value rounded to the fixed-point unit as
// the shared-memory path rounds it and added to the global current (periodic
// axes wrapped, nodes beyond an open face dropped, as the push drops them).
template <int D, int W>
__device__ __forceinline__ void deposit_far(const GridP &g, const int c[3], const float f[3], const float de[3], float qw,
                                            const float v[3], unsigned long long *jfx, float scale) {
  constexpr int NODES = D == 3 ? 64 : (D == 2 ? 16 : 4);
  PairAxis G[3];
#pragma unroll
  for (int a = 0; a < D; ++a) G[a] = pair_axis(f[a], de[a], -qw * g.dxdt[a]);
#pragma unroll 1
  for (int it = W > 1 ? (int)(threadIdx.x & (W - 1)) : 0; it < 3 * NODES; it += W) {
    const int cc = it / NODES, m = it - cc * NODES;
    // shapes of the transverse axes (1 and 0 along cc and axes not simulated)
    float S[3] = {1.0f, 1.0f, 1.0f}, T[3] = {0.0f, 0.0f, 0.0f}, val = 0.0f;
    long long gi = 0, stride = 1;
    bool ok = true;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const int k = (m >> (2 * a)) & 3;
      if (a == cc) {
        val = sel4(k, G[a].P);
      } else {
        S[a] = sel4(k, G[a].S);
        T[a] = sel4(k, G[a].DS);
      }
      int x = c[a] + G[a].base + k;
      if (g.bc[a] == BP_PERIODIC) x = wrap_once(x, g.n[a]);
      else ok &= x >= 0 && x < g.n[a];
      gi += (long long)x * stride;
      stride *= g.n[a];
    }
    if (cc >= D) val = qw * (cc == 1 ? v[1] : v[2]);
    const float F = cc == 0 ? pair_factor(S[1], T[1], S[2], T[2])
                            : (cc == 1 ? pair_factor(S[0], T[0], S[2], T[2]) : pair_factor(S[0], T[0], S[1], T[1]));
    const float vs = val * F * scale;
    if (ok && fabsf(vs) > 0.5f) atomicAdd(jfx + (size_t)cc * g.ncell + gi, (unsigned long long)f2ll_rn(vs));
  }
}

// E and B of one body read from the global fields by its lanes (a body
// outside the tile's staged box): the staggered quadratic gather over the
// body's cell c and offset f, the stencil's nodes shared out over the lanes; periodic axes wrapped, zero beyond open faces
template <int D, int W>
__device__ __forceinline__ void gather_global(const GridP &g, const float *const *Eg, const float *const *Bg,
                                              const int c[3], const float f[3], float E[3], float B[3]) {
  constexpr int NODES = D == 3 ? 27 : (D == 2 ? 9 : 3);
#pragma unroll
  for (int cc = 0; cc < 6; ++cc) {
    // stagger pattern of component cc: bit a set when it sits half a cell along a
    const int pat = cc < 3 ? (1 << cc) : (7 & ~(1 << (cc - 3)));
    const float *F = cc < 3 ? Eg[cc] : Bg[cc - 3];
    float acc = 0.0f;
    for (int k = W > 1 ? (int)(threadIdx.x & (W - 1)) : 0; k < NODES; k += W) {
      const int o[3] = {k % 3, (k / 3) % 3, k / 9};
      long long gi = 0, stride = 1;
      float w = 1.0f;
      bool ok = true;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        const bool half = (pat >> a) & 1;
        const int up = half ? 0 : (f[a] >= 0.5f ? 1 : 0);
        float wa[3];
        qweights(half ? f[a] - 0.5f : f[a] - (float)up, wa);
        w *= o[a] == 0 ? wa[0] : (o[a] == 1 ? wa[1] : wa[2]);
        int x = c[a] + up - 1 + o[a];
        if (g.bc[a] == BP_PERIODIC) x = wrap_once(x, g.n[a]);
        else ok &= x >= 0 && x < g.n[a];
        gi += (long long)x * stride;
        stride *= g.n[a];
      }
      if (ok) acc = fmaf(w, F[gi], acc);
    }
#pragma unroll
    for (int q = W / 2; q > 0; q >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, q);
    if (cc < 3) E[cc] = acc;
    else B[cc - 3] = acc;
  }
}

// node bounding box of a thread's deposits, one byte per axis (box
// coordinates are below 256); axes the grid does not simulate stay at 0
template <int D>
__device__ __forceinline__ void bb_add(unsigned &lo, unsigned &hi, const int n[3], int below, int above) {
  unsigned l = 0, h = 0;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    l |= (unsigned)(n[a] - below) << (8 * a);
    h |= (unsigned)(n[a] + above) << (8 * a);
  }
  lo = __vminu4(lo, l);
  hi = __vmaxu4(hi, h);
}

// the centre node of a body's general window (it reaches two nodes either way)
template <int D>
__device__ __forceinline__ void window_centre(const float *f, const int *d, int n0[3]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) n0[a] = a < D ? d[a] + Box<D>::OJ + (f[a] >= 0.5f ? 1 : 0) : 0;
}

// a particle of (loaded) species s left its tile's margin: the species is
// sorted before the next push.  The flags are read first: in a hot plasma many
// particles set them in one step.
__device__ __forceinline__ void mark_sort(int *status, int s) {
  volatile int *const st = status;
  if (!(st[1] & (1 << s))) atomicOr(status + 1, 1 << s);
  if (!(st[0] & ST_NEED_SORT)) atomicOr(status, ST_NEED_SORT);
}

// 1 / gamma of a momentum u = p / (m c), one fixed evaluation order (the
// quiet pass and the full push must move a particle identically)
__device__ __forceinline__ float inv_gamma(const float u[3]) {
  return rsqrtf(fmaf(u[2], u[2], fmaf(u[1], u[1], fmaf(u[0], u[0], 1.0f))));
}

// body 1's offset after the drift x += dt v, in cells
__device__ __forceinline__ float drift_offset(const GridP &g, int a, float f, float v) {
  return fmaf(g.dt * v, g.idx[a], f);
}

// new cell of body 1 from its moved offset fn (renormalised to [0, 1)).  On
// open axes a free particle whose cell leaves [2, n-2) is removed (after its
// last deposit); a two-body ion leaving the grid is a domain error.
template <int D>
__device__ __forceinline__ void advance_cell(const GridP &g, const int T0[3], bool two, int c[3], float fn[3],
                                             bool &bad, bool &removed, bool &need_sort) {
#pragma unroll
  for (int a = 0; a < D; ++a) {
    if (fn[a] >= 1.0f) {
      fn[a] -= 1.0f;
      c[a] += 1;
    } else if (fn[a] < 0.0f) {
      fn[a] += 1.0f;
      c[a] -= 1;
      if (fn[a] >= 1.0f) { fn[a] = 0.0f; c[a] += 1; }
    }
    if (g.bc[a] == BP_PERIODIC) {
      c[a] = wrap_once(c[a], g.n[a]);
    } else if (two) {
      bad |= (c[a] < 0 || c[a] >= g.n[a]);
    } else {
      removed |= (c[a] < 2 || c[a] >= g.n[a] - 2);
    }
    const int dn = rel_cell<D>(g, a, c[a], T0[a]);
    need_sort |= outside_margin<D>(a, dn);
  }
}

// A quiet ion: a neutral two-body ion whose bodies coincide (r = 0) and move
// together (u1 = u2, finite) in a tile whose staged fields are all zero.  The
// full push leaves its momenta and r exactly as they are (zero internal force
// at r = 0, zero fields) and deposits nothing (its bodies' terms cancel), so
// only body 1's drift remains.
__device__ __forceinline__ bool quiet_state(const float r[3], const float u1[3], const float u2[3]) {
  bool q = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) q &= (r[a] == 0.0f) && (u1[a] == u2[a]) && isfinite(u1[a]);
  return q;
}

// The quiet pass over QB particles of a thread (i0, i0 + bs, ...): all loads
// first, so that many are in flight, then the drift of the quiet ones, which
// writes only the cell and the offset.  Returns true when one of them is not
// quiet (left for the full push).
template <int D, int QB>
__device__ __forceinline__ bool quiet_batch(const GridP &g, const PartP &P, long long i0, int bs, long long end,
                                            const int T0[3], int *status, int s, unsigned &moved) {
  const long long cap = P.cap;
  int cell[QB];
  float f[QB][3], u1[QB][3], u2[QB][3], r[QB][3];
#pragma unroll
  for (int q = 0; q < QB; ++q) {
    const long long i = i0 + (long long)q * bs;
    cell[q] = i < end ? P.cell[i] : -1;
    if (cell[q] >= 0) {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        f[q][a] = a < D ? P.off[a * cap + i] : 0.0f;
        u1[q][a] = P.u1[a * cap + i];
        u2[q][a] = P.u2[a * cap + i];
        r[q][a] = P.r[a * cap + i];
      }
    }
  }
  bool left = false;
#pragma unroll
  for (int q = 0; q < QB; ++q) {
    if (cell[q] < 0) continue;
    if (!quiet_state(r[q], u1[q], u2[q])) {
      left = true;
      continue;
    }
    const long long i = i0 + (long long)q * bs;
    int c[3];
    unpack_cell(g, cell[q], c);
    bool bad = false, removed = false, need_sort = false;
#pragma unroll
    for (int a = 0; a < D; ++a) bad |= outside_margin<D>(a, rel_cell<D>(g, a, c[a], T0[a]));
    if (bad) {
      atomicOr(status, ST_DOMAIN);
      continue;
    }
    const float gi = inv_gamma(u1[q]);
    float fn[3];
#pragma unroll
    for (int a = 0; a < D; ++a) fn[a] = drift_offset(g, a, f[q][a], u1[q][a] * gi);
    advance_cell<D>(g, T0, true, c, fn, bad, removed, need_sort);
    if (bad) {
      atomicOr(status, ST_DOMAIN);
      P.cell[i] = -1;
      continue;
    }
    if (need_sort) mark_sort(status, s);
    P.cell[i] = pack_cell(g, c[0], c[1], c[2]);
#pragma unroll
    for (int a = 0; a < D; ++a) P.off[a * cap + i] = fn[a];
    ++moved;
  }
  return left;
}

// add a per-thread count to a global work counter: one atomic per warp
__device__ __forceinline__ void count_work(unsigned long long *ctr, unsigned n) {
  const unsigned s = __reduce_add_sync(0xFFFFFFFFu, n);
  if ((threadIdx.x & 31u) == 0 && s) atomicAdd(ctr, (unsigned long long)s);
}

// whether the quiet pass has already moved particle i (its state is still
// quiet after the move: r, u1, u2 unchanged)
__device__ __forceinline__ bool quiet_done(const PartP &P, long long i) {
  const long long cap = P.cap;
  if (P.cell[i] < 0) return true;
  float r[3], u1[3], u2[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    r[a] = P.r[a * cap + i];
    u1[a] = P.u1[a * cap + i];
    u2[a] = P.u2[a * cap + i];
  }
  return quiet_state(r, u1, u2);
}

// The whole step of a two-body ion whose bound electron is a cell or more
// from its nucleus (a strong field pulls it into the Coulomb tail of the
// modified potential), sorted mode: outside the tile's boxes, so both bodies
// gather from the global E and B and deposit into the global fixed-point
// current.  The same arithmetic as push_particle's.
// A warp (W = 32 or 16 lanes a body; every lane holds the ion, lane 0 writes
// it) or a thread (W = 1) per ion.  Returns
// false when the ion cannot be moved this way (body 1 outside its tile's
// margin, body 2 beyond an open face or a displacement that is not finite): a
// domain error for the caller.
template <int D, int W>
__device__ __forceinline__ bool push_far(const GridP &g, const SpecP &sp, const PartP &P, int s, long long i, int t0x, int t0y,
                                      int t0z, int *status, const float *const *Eg, const float *const *Bg,
                                      unsigned long long *jfx, float scale) {
  const long long cap = P.cap;
  const int T0[3] = {t0x, t0y, t0z};
  int c[3];
  unpack_cell(g, P.cell[i], c);
  float f[3] = {0.0f, 0.0f, 0.0f}, r[3], u1[3], u2[3];
#pragma unroll
  for (int a = 0; a < D; ++a) f[a] = P.off[a * cap + i];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    r[a] = P.r[a * cap + i];
    u1[a] = P.u1[a * cap + i];
    u2[a] = P.u2[a * cap + i];
  }
  int c2[3] = {0, 0, 0};
  float f2[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
  for (int a = 0; a < D; ++a) {
    if (outside_margin<D>(a, rel_cell<D>(g, a, c[a], T0[a]))) return false;
    const float rc = r[a] * g.idx[a];
    if (!(fabsf(rc) < (float)g.n[a])) return false;
    const float X = f[a] - rc;
    const float fl = floorf(X);
    float fr = X - fl;
    int di = (int)fl;
    if (fr >= 1.0f) { fr = 0.0f; di += 1; }
    c2[a] = c[a] + di;
    if (g.bc[a] == BP_PERIODIC) c2[a] = wrap_mod(c2[a], g.n[a]);
    else if (c2[a] < 0 || c2[a] >= g.n[a]) return false;
    f2[a] = fr;
  }
  float E1[3], B1[3], E2[3], B2[3];
  const bool second = W == 16 && (threadIdx.x & 16);  // this half warp's body
  if constexpr (W != 16) {
    gather_global<D, W>(g, Eg, Bg, c, f, E1, B1);
    gather_global<D, W>(g, Eg, Bg, c2, f2, E2, B2);
  } else {
    int cb[3];
    float fb[3], Eo[3], Bo[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      cb[a] = second ? c2[a] : c[a];
      fb[a] = second ? f2[a] : f[a];
    }
    gather_global<D, W>(g, Eg, Bg, cb, fb, Eo, Bo);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float e = __shfl_xor_sync(0xFFFFFFFFu, Eo[a], 16), b = __shfl_xor_sync(0xFFFFFFFFu, Bo[a], 16);
      E1[a] = second ? e : Eo[a];
      B1[a] = second ? b : Bo[a];
      E2[a] = second ? Eo[a] : e;
      B2[a] = second ? Bo[a] : b;
    }
  }
  const int pi = P.pidx ? P.pidx[i] : 0;
  const float ac = sp.ac[pi];
  const float rr = r[0] * r[0] + r[1] * r[1] + r[2] * r[2] + ac * ac;
  const float rs = rsqrtf(rr);
  const float k3 = sp.kappa * rs * rs * rs;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    E1[a] = fmaf(sp.q2 * k3, r[a], E1[a]);
    E2[a] = fmaf(-sp.q1 * k3, r[a], E2[a]);
  }
  boris(sp.h2, E2, B2, u2);
  boris(sp.h1, E1, B1, u1);
  float v1[3], v2[3];
  const float g1 = inv_gamma(u1), g2 = inv_gamma(u2);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    v1[a] = u1[a] * g1;
    v2[a] = u2[a] * g2;
  }
  float fn[3] = {0.0f, 0.0f, 0.0f}, de1[3] = {0.0f, 0.0f, 0.0f}, de2[3] = {0.0f, 0.0f, 0.0f}, rn[3];
#pragma unroll
  for (int a = 0; a < D; ++a) {
    fn[a] = drift_offset(g, a, f[a], v1[a]);
    de1[a] = fn[a] - f[a];
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    rn[a] = r[a] + g.dt * (v1[a] - v2[a]);
    if (a < D) de2[a] = de1[a] - (rn[a] - r[a]) * g.idx[a];
  }
  // each body on its own, around its own cell
  if constexpr (W != 16) {
    deposit_far<D, W>(g, c, f, de1, sp.qw1, v1, jfx, scale);
    deposit_far<D, W>(g, c2, f2, de2, sp.qw2, v2, jfx, scale);
  } else {
    int cb[3];
    float fb[3], db[3], vb[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      cb[a] = second ? c2[a] : c[a];
      fb[a] = second ? f2[a] : f[a];
      db[a] = second ? de2[a] : de1[a];
      vb[a] = second ? v2[a] : v1[a];
    }
    deposit_far<D, W>(g, cb, fb, db, second ? sp.qw2 : sp.qw1, vb, jfx, scale);
  }
  if (W > 1 && (threadIdx.x & 31)) return true;
  bool bad = false, removed = false, need_sort = false, nonfinite = false;
  advance_cell<D>(g, T0, true, c, fn, bad, removed, need_sort);
#pragma unroll
  for (int a = 0; a < 3; ++a) nonfinite |= !isfinite(u1[a]) || !isfinite(u2[a]);
  if (bad) atomicOr(status, ST_DOMAIN);
  if (nonfinite) atomicOr(status, ST_NONFINITE);
  if (bad) {
    P.cell[i] = -1;
    return true;
  }
  if (need_sort) mark_sort(status, s);
  P.cell[i] = pack_cell(g, c[0], c[1], c[2]);
#pragma unroll
  for (int a = 0; a < D; ++a) P.off[a * cap + i] = fn[a];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    P.u1[a * cap + i] = u1[a];
    P.r[a * cap + i] = rn[a];
    P.u2[a * cap + i] = u2[a];
  }
  return true;
}

// How much a particle may add to one node of the box's two words (fx_add).
// High words: its bodies' currents q w v, of which a node gets at most 0.75 per
// simulated axis (the largest shape factor, and the largest flux of a shape
// through a face), in units of 2^16; the scale (bp_api.cu) keeps them at 2^21
// for two bodies.  Low words: two adds of up to 2^15 each; 2^16 is counted for
// them.  A warp drains the box when one of its lanes has put in kLaneLoad since
// its last drain, so a word holds at most that and one particle of every lane
// (512 in 3D, 256 else): high words stay below 1.61e9 + 0.49e9 < 2^31, and low
// words have at most 2 (24,576 + 512) < 2^16 adds.
template <int D>
constexpr unsigned kLaneLoad = (3u << 29) / push_threads(D);
template <int D>
__device__ __forceinline__ unsigned box_load(const SpecP &sp, const float v1[3], const float v2[3], float scale) {
  constexpr float SHAPE = D == 1 ? 0.7501f : (D == 2 ? 0.5627f : 0.4220f);
  const float m1 = fmaxf(fmaxf(fabsf(v1[0]), fabsf(v1[1])), fabsf(v1[2]));
  const float m2 = fmaxf(fmaxf(fabsf(v2[0]), fabsf(v2[1])), fabsf(v2[2]));
  return 65536u + (unsigned)(fmaf(fabsf(sp.qw1), m1, fabsf(sp.qw2) * m2) * (scale * (SHAPE / 65536.0f)));
}

// One particle's step.  In 3D every lane of the warp calls it, those without a
// particle with have = false: the general-case deposits are the whole warp's.
// JT fx64: fields and current are the global arrays (A.E, A.B at `at`; Jsm the
// current at the box's origin, strides st)
template <int D, bool DET, bool FREE, typename JT, typename ST = BoxStride<D>>
__device__ void push_particle(const GridP &g, const SpecP &sp, const PartP &P, bool have, long long i, const int T0[3],
                              const float *Gsm, JT *Jsm, int *status, float scale, unsigned &blo, unsigned &bhi,
                              unsigned &load, PairJob *jobs, bool nofield, int4 *far, int *far_n, int far_cap, int s, int t,
                              const PushArgs *A = nullptr, long long at = 0, const ST &st = ST()) {
  constexpr bool GLOBAL = std::is_same<JT, fx64>::value;
  const long long cap = P.cap;
  const bool two = sp.kind == BP_TWO_BODY;
  int c[3], d[3] = {0, 0, 0}, d2[3] = {0, 0, 0}, nn[3] = {2, 2, 2};
  float f[3] = {0.0f, 0.0f, 0.0f}, r[3] = {0.0f, 0.0f, 0.0f}, u1[3], u2[3] = {0.0f, 0.0f, 0.0f};
  float f2[3] = {0.0f, 0.0f, 0.0f}, v1[3], v2[3] = {0.0f, 0.0f, 0.0f};
  float fn[3] = {0.0f, 0.0f, 0.0f}, de1[3] = {0.0f, 0.0f, 0.0f}, de2[3] = {0.0f, 0.0f, 0.0f}, rn[3];
  float xi[2][3] = {{0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f}};
  float dxdt[3] = {g.dxdt[0], g.dxdt[1], g.dxdt[2]};  // (in 1D and 2D read further down: registers)
  bool bad = false, fast = true, silent = true;
  // kicks and moves; not live: no particle, or one that is left where it is
  bool live = false;
  do {
    if (D == 3 && !have) break;
    const int cell = P.cell[i];
    if (cell < 0) break;
    unpack_cell(g, cell, c);
#pragma unroll
    for (int a = 0; a < D; ++a) f[a] = P.off[a * cap + i];
#pragma unroll
    for (int a = 0; a < 3; ++a) u1[a] = P.u1[a * cap + i];
    if (two) {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        r[a] = P.r[a * cap + i];
        u2[a] = P.u2[a * cap + i];
      }
    }
#pragma unroll
    for (int a = 0; a < D; ++a) {
      d[a] = rel_cell<D>(g, a, c[a], T0[a]);
      bad |= outside_margin<D>(a, d[a]);
      // body 2 sits at x1 - r
      float rc = r[a] * g.idx[a];
      bad |= !(fabsf(rc) < 1.0f);
      float X = f[a] - rc;
      float fl = floorf(X);
      float fr = X - fl;
      int di = (int)fl;
      if (fr >= 1.0f) { fr = 0.0f; di += 1; }
      d2[a] = d[a] + di;
      f2[a] = fr;
    }
    if (bad) {
      // sorted mode: perhaps a bound electron a cell or more from its nucleus,
      // which k_push_far moves on the global grid after this kernel (it
      // reports a domain error for anything else); atomic mode: a domain error
      if (DET && two) {
        const int k = atomicAdd(far_n, 1);
        if (k < far_cap) {
          far[k] = make_int4(s, (int)i, t, 0);
          break;
        }
      }
      atomicOr(status, ST_DOMAIN);
      break;
    }
    // A tile whose staged box holds no field (ahead of the field front) gathers
    // exact zeros, so the gather is skipped.  A neutral ion there with r = 0 and
    // u1 = u2 also keeps its momenta exactly (no internal force at r = 0, Boris
    // rotation by zero fields), so its kicks are skipped too.
    bool quiet = nofield && two && sp.qw1 == -sp.qw2;
#pragma unroll
    for (int a = 0; a < 3; ++a) quiet &= (r[a] == 0.0f) && (u1[a] == u2[a]);
    float E1[3], B1[3], E2[3], B2[3];
    if (nofield) {
#pragma unroll
      for (int a = 0; a < 3; ++a) E1[a] = B1[a] = E2[a] = B2[a] = 0.0f;
    } else {
      if constexpr (D == 3) {
        Pos P1, P2;
        make_pos<D>(d, f, P1);
        make_pos<D>(two ? d2 : d, two ? f2 : f, P2);
        gather_all_p3(Gsm, P1, P2, E1, B1, E2, B2);
      } else {
        Loc L1, L2;
        make_loc<D>(d, f, L1);
        make_loc<D>(two ? d2 : d, two ? f2 : f, L2);
        if constexpr (GLOBAL) gather_all_few(A->E, A->B, at, st.row, L1, L2, E1, B1, E2, B2);
        else gather_all<D>(Gsm, L1, L2, E1, B1, E2, B2);
      }
    }
    if (two && !quiet) {
      // modified Coulomb field (Sec. 2): on the nucleus q2 kappa r / (r^2 + ac^2)^{3/2},
      // on the bound electron -q1 kappa r / (...), r = x1 - x2
      const int pi = P.pidx ? P.pidx[i] : 0;
      const float ac = sp.ac[pi];
      float rr = r[0] * r[0] + r[1] * r[1] + r[2] * r[2] + ac * ac;
      float rs = rsqrtf(rr);
      float s = sp.kappa * rs * rs * rs;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        E1[a] = fmaf(sp.q2 * s, r[a], E1[a]);
        E2[a] = fmaf(-sp.q1 * s, r[a], E2[a]);
      }
      boris(sp.h2, E2, B2, u2);
    }
    if (two) {
      const float g2 = inv_gamma(u2);
#pragma unroll
      for (int a = 0; a < 3; ++a) v2[a] = u2[a] * g2;
    }
    if (!quiet) boris(sp.h1, E1, B1, u1);
    {
      const float g1 = inv_gamma(u1);
#pragma unroll
      for (int a = 0; a < 3; ++a) v1[a] = u1[a] * g1;
    }
    // drift: body 1 moves in cells by dt v / dx; the internal displacement by
    // dt (v1 - v2) on all three axes; the deposited moves are the ones the
    // stored FP32 state actually makes
#pragma unroll
    for (int a = 0; a < D; ++a) {
      fn[a] = drift_offset(g, a, f[a], v1[a]);
      de1[a] = fn[a] - f[a];
    }
    if (two) {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        rn[a] = r[a] + g.dt * (v1[a] - v2[a]);
        float dr = rn[a] - r[a];
        if (a < D) de2[a] = de1[a] - dr * g.idx[a];
      }
    }
    if constexpr (D < 3) {
#pragma unroll
      for (int a = 0; a < 3; ++a) dxdt[a] = g.dxdt[a];
    }
    // fast path when every position keeps one nearest node per axis
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const float u1p = f[a] >= 0.5f ? 1.0f : 0.0f;
      xi[0][a] = f[a] - u1p;
      const float x1n = xi[0][a] + de1[a];
      fast &= (x1n >= -0.5f) && (x1n < 0.5f);
      nn[a] = d[a] + Box<D>::OJ + (int)u1p;
      if (two) {
        const float u2p = f2[a] >= 0.5f ? 1.0f : 0.0f;
        xi[1][a] = f2[a] - u2p;
        const float x2n = xi[1][a] + de2[a];
        fast &= (d2[a] == d[a]) && (u2p == u1p) && (x2n >= -0.5f) && (x2n < 0.5f);
      }
    }
    // a neutral ion whose bodies coincide and move together carries no
    // current (its two bodies' terms cancel exactly; Sec. 2 starts every ion
    // so, and it stays so until a field acts on it): nothing to deposit
    silent = two && sp.qw1 == -sp.qw2;
#pragma unroll
    for (int a = 0; a < 3; ++a) silent &= (r[a] == 0.0f) && (v1[a] == v2[a]);
    if (DET && !GLOBAL && !silent) load += box_load<D>(sp, v1, v2, scale);
    live = true;
  } while (false);
  if constexpr (D == 3) {
    // the general case in 3D: rare in a thermal medium, so the whole warp
    // shares out one such particle after the other.  Its lanes meet here
    // whatever became of their own particles: the slot is the warp's, and two
    // groups of it that arrived apart, each with its own active mask, would
    // share it.  (32.5 M ions: 3.69 ms a step, 3.63 with such masks.)
    unsigned gen = __ballot_sync(0xFFFFFFFFu, live && !silent && !fast);
    for (; gen; gen &= gen - 1) {
      PairJob &P = jobs[threadIdx.x >> 5];
      if ((int)(threadIdx.x & 31) == __ffs(gen) - 1) {
        const float sc = DET ? scale : 1.0f;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          P.f[0][a] = f[a];
          P.f[1][a] = f2[a];
          P.e[0][a] = de1[a];
          P.e[1][a] = de2[a];
          P.d[0][a] = d[a];
          P.d[1][a] = d2[a];
          P.q[0][a] = -(sp.qw1 * sc) * dxdt[a];
          P.q[1][a] = -(sp.qw2 * sc) * dxdt[a];
        }
        P.two = two;
      }
      __syncwarp();
      deposit_general3_warp<DET, JT>(Jsm, &P);
      __syncwarp();
    }
  }
  if (!live) return;
  if (!silent) {
    if (fast) {
      float qw[2] = {sp.qw1, sp.qw2};
      float vv[2][3];
      float dd[2][3];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        vv[0][a] = v1[a];
        vv[1][a] = v2[a];
        dd[0][a] = de1[a];
        dd[1][a] = de2[a];
      }
      if constexpr (D == 3 && DET) {
        if (two) esirkepov3_p3(Jsm, nn, xi, dd, qw, dxdt, scale);
        else esirkepov3<D, DET, 1>(Jsm, nn, xi, dd, qw, vv, dxdt, scale);
      } else if (two) esirkepov3<D, DET, 2>(Jsm, nn, xi, dd, qw, vv, dxdt, scale, st);
      else esirkepov3<D, DET, 1>(Jsm, nn, xi, dd, qw, vv, dxdt, scale, st);
      bb_add<D>(blo, bhi, nn, 1, 1);
    } else {
      if constexpr (D == 2 && FREE) {
        // body by body
#pragma unroll 1
        for (int b = 0; b < (two ? 2 : 1); ++b) {
          float fb[3], db[3], vb[3];
          int cb[3];
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            fb[a] = b ? f2[a] : f[a];
            db[a] = b ? de2[a] : de1[a];
            vb[a] = b ? v2[a] : v1[a];
            cb[a] = b ? d2[a] : d[a];
          }
          deposit_general<D, DET, JT>(Jsm, cb, fb, db, b ? sp.qw2 : sp.qw1, vb, dxdt, scale);
        }
      } else if constexpr (D < 3) {
        if (two) {
          float fb[2][3], db[2][3], vb[2][3], dd[3];
          int cb[2][3];
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            fb[0][a] = f[a]; fb[1][a] = f2[a];
            db[0][a] = de1[a]; db[1][a] = de2[a];
            vb[0][a] = v1[a]; vb[1][a] = v2[a];
            cb[0][a] = d[a]; cb[1][a] = d2[a];
            dd[a] = dxdt[a];
          }
          deposit_general_pair<D, DET, JT>(Jsm, cb[0], cb[1], fb[0], fb[1], db[0], db[1], sp.qw1, sp.qw2, vb[0], vb[1], dd,
                                           scale, st);
        } else if constexpr (D == 1) {
          deposit_general<D, DET, JT>(Jsm, d, f, de1, sp.qw1, v1, dxdt, scale);
        }
      }
      int n0[3];
      window_centre<D>(f, d, n0);
      bb_add<D>(blo, bhi, n0, 2, 2);
      if (two) {
        window_centre<D>(f2, d2, n0);
        bb_add<D>(blo, bhi, n0, 2, 2);
      }
    }
  }
  bool need_sort = false, nonfinite = false, removed = false;
  advance_cell<D>(g, T0, two, c, fn, bad, removed, need_sort);
#pragma unroll
  for (int a = 0; a < 3; ++a) nonfinite |= !isfinite(u1[a]) || !isfinite(u2[a]);
  if (bad) atomicOr(status, ST_DOMAIN);
  if (nonfinite) atomicOr(status, ST_NONFINITE);
  if (bad || removed) {
    P.cell[i] = -1;
    return;
  }
  if (need_sort) mark_sort(status, s);
  P.cell[i] = pack_cell(g, c[0], c[1], c[2]);
#pragma unroll
  for (int a = 0; a < D; ++a) P.off[a * cap + i] = fn[a];
#pragma unroll
  for (int a = 0; a < 3; ++a) P.u1[a * cap + i] = u1[a];
  if (two) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      P.r[a * cap + i] = rn[a];
      P.u2[a * cap + i] = u2[a];
    }
  }
}

// the state of the particle a thread takes next, brought into L1 while the
// current one is pushed (its loads would otherwise stall the warp at the
// start of the next iteration)
template <int D>
__device__ __forceinline__ void prefetch_particle(const PartP &P, long long j, bool two) {
  const long long cp = P.cap;
  asm volatile("prefetch.global.L1 [%0];" ::"l"(P.cell + j));
#pragma unroll
  for (int a = 0; a < D; ++a) asm volatile("prefetch.global.L1 [%0];" ::"l"(P.off + a * cp + j));
#pragma unroll
  for (int a = 0; a < 3; ++a) asm volatile("prefetch.global.L1 [%0];" ::"l"(P.u1 + a * cp + j));
  if (two) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      asm volatile("prefetch.global.L1 [%0];" ::"l"(P.r + a * cp + j));
      asm volatile("prefetch.global.L1 [%0];" ::"l"(P.u2 + a * cp + j));
    }
  }
}

// clear a shared-memory current box of n nodes (and the high words in the
// sorted mode), 16 bytes per store
template <bool DET, typename JT>
__device__ __forceinline__ void zero_box(JT *J, int n, int tid, int bs) {
  constexpr int W = DET ? 2 : 1;
  uint4 *p = reinterpret_cast<uint4 *>(J);
  const int n4 = (W * n) / 4;
  for (int q = tid; q < n4; q += bs) p[q] = make_uint4(0u, 0u, 0u, 0u);
  for (int q = 4 * n4 + tid; q < W * n; q += bs) reinterpret_cast<unsigned *>(J)[q] = 0u;
}

// A tile whose 3^D neighbouring tiles have never held a non-zero E or B has
// an all-zero field box (the box lies inside them).  This light kernel takes
// such tiles before the push: it moves their quiet ions (the drift alone) at
// high occupancy (eight 128-thread blocks per SM) and leaves a state per tile:
//   QS_PUSH  the push kernel does the whole tile (fields may be non-zero),
//   QS_DONE  every particle moved, nothing deposited (occ = 0),
//   QS_REST  the quiet ions moved; the push does the others without fields.
//   QS_COLD  no fields and no particle moved yet (grids that go without this
//            pass): the push does the whole tile without fields.
constexpr unsigned char QS_PUSH = 0, QS_DONE = 1, QS_REST = 2, QS_COLD = 3;

// lane's share (lanes 0..26) of whether a tile of t's 3^D neighbourhood has
// held a non-zero E or B
template <int D>
__device__ __forceinline__ bool near_mark(const GridP &g, int t, int lane) {
  if (lane >= 27) return false;
  const int tc[3] = {t % g.nt[0], (t / g.nt[0]) % g.nt[1], t / (g.nt[0] * g.nt[1])};
  const int o[3] = {lane % 3 - 1, (lane / 3) % 3 - 1, lane / 9 - 1};
  bool use = true;
  int nb[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    nb[a] = tc[a] + o[a];
    if (a >= D) use &= o[a] == 0;
    else if (g.bc[a] == BP_PERIODIC) nb[a] = wrap_once(nb[a], g.nt[a]);
    else use &= nb[a] >= 0 && nb[a] < g.nt[a];
  }
  return use && g.fnz[nb[0] + g.nt[0] * (nb[1] + g.nt[1] * nb[2])] != 0;
}

// Tiles of at most FEW ions go to k_push_few when their boxes lie within the
// grid (no wrap, no open face to look out for).  1024 x 1024 cells, ions at
// random places, step by box and from the global arrays: 133 and 71 us with 8
// ions a tile, 149 and 93 with 48, 154 and 104 with 64, 172 and 139 with 128;
// but ions that sit close together add to the same nodes, one after the other
// in L2 (128 a tile in 4 x 4 cells: 303 us a step, 312), so it stops at 64.
constexpr int FEW = 64;
template <int D>
__device__ __forceinline__ bool box_inside(const GridP &g, int t) {
  const int tc[3] = {t % g.nt[0], (t / g.nt[0]) % g.nt[1], t / (g.nt[0] * g.nt[1])};
  using BX = Box<D>;
  constexpr int L[3] = {Geo<D>::L0, Geo<D>::L1, Geo<D>::L2}, GN[3] = {BX::G0, BX::G1, BX::G2}, JN[3] = {BX::J0, BX::J1, BX::J2};
  bool in = true;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    const int x = tc[a] * L[a];
    in &= x >= BX::OG && x - BX::OG + GN[a] <= g.n[a] && x >= BX::OJ && x - BX::OJ + JN[a] <= g.n[a];
  }
  return in;
}

template <int D>
__global__ void __launch_bounds__(128, 8) k_push_quiet(const __grid_constant__ GridP g, PushArgs A, int qt, int few,
                                                       const __grid_constant__ AntArgs ant) {
  static_assert(Box<D>::OG <= Geo<D>::L0 && Box<D>::G0 - Box<D>::OG <= 2 * Geo<D>::L0 &&
                    (D < 2 || (Box<D>::OG <= Geo<D>::L1 && Box<D>::G1 - Box<D>::OG <= 2 * Geo<D>::L1)) &&
                    (D < 3 || (Box<D>::OG <= Geo<D>::L2 && Box<D>::G2 - Box<D>::OG <= 2 * Geo<D>::L2)),
                "field box within the neighbouring tiles");
  constexpr int QB = 2;  // particles in flight per thread (measured best of 1, 2, 4, 8)
  // qt (1 to 4) tiles per block: one warp classifies each, then the whole
  // block drifts the quiet ones in turn (several tiles per block on grids
  // with many tiles, where a block per tile spent its time waiting on the
  // classification loads; one on small grids, where tiles in turn would
  // lengthen the pass)
  __shared__ int quiet[4], nquiet;
  if ((int)blockIdx.x < ant.blocks) {
    antenna_block<D>(g, ant);
    return;
  }
  const int tid = threadIdx.x, bs = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const int t = ((int)blockIdx.x - ant.blocks) * qt + warp;
  if (tid == 0) nquiet = 0;
  bool marked = false, occupied = false;
  int ions = 0;
  const bool stop = timed_out(A.status);
  if (warp < qt && t < g.ntiles) {
    marked = near_mark<D>(g, t, lane);
    // a tile without particles has nothing to push or deposit, whatever its
    // fields: done here, so the push neither stages its fields nor visits it
    if (lane < A.nsp) ions = A.p[lane].tstart[t + 1] - A.p[lane].tstart[t];
  }
  marked = __any_sync(0xFFFFFFFFu, marked);
  ions = __reduce_add_sync(0xFFFFFFFFu, ions);
  occupied = ions > 0;
  // a sort gave up: the tiles' particle ranges may not fit together, and the
  // push's lists stay empty
  if (stop) return;
  __syncthreads();  // nquiet cleared
  if (warp < qt && t < g.ntiles && lane == 0) {
    if (!occupied) {
      A.qstate[t] = QS_DONE;
      A.occ[t] = 0;
    } else if (marked) {
      A.qstate[t] = QS_PUSH;
      if (few && ions <= FEW && box_inside<D>(g, t)) A.tile_list[g.ntiles - 1 - atomicAdd(A.tile_n + 1, 1)] = t;
      else A.tile_list[atomicAdd(A.tile_n, 1)] = t;
    } else {
      quiet[atomicAdd(&nquiet, 1)] = t;  // each quiet tile is drifted alone: their order changes nothing
    }
  }
  __syncthreads();
  const int nq = nquiet;
  unsigned moved = 0;
  for (int k = 0; k < nq; ++k) {
    const int tq = quiet[k];
    const int T0[3] = {(tq % g.nt[0]) * Geo<D>::L0, ((tq / g.nt[0]) % g.nt[1]) * Geo<D>::L1,
                       (tq / (g.nt[0] * g.nt[1])) * Geo<D>::L2};
    bool left = false;
    for (int s = 0; s < A.nsp; ++s) {
      const int beg = A.p[s].tstart[tq], end = A.p[s].tstart[tq + 1];
      if (A.sp[s].kind == BP_TWO_BODY && A.sp[s].qw1 == -A.sp[s].qw2) {
        for (long long i0 = beg + tid; i0 < end; i0 += (long long)QB * bs)
          left |= quiet_batch<D, QB>(g, A.p[s], i0, bs, end, T0, A.status, s, moved);
      } else {
        left |= end > beg;
      }
    }
    left = __syncthreads_or(left);
    if (tid == 0) {
      A.qstate[tq] = left ? QS_REST : QS_DONE;
      if (!left) A.occ[tq] = 0;
      else A.tile_list[atomicAdd(A.tile_n, 1)] = tq;
    }
  }
  if (A.work) count_work(A.work + 1, moved);
}

// Tiles whose cells the field updates can change: a tile of the 3^D
// neighbourhood has held a non-zero E or B (the sticky marks), or holds
// particles the push moved this step (QS_PUSH, QS_REST: their current reaches
// the neighbouring tiles), or an antenna plane lies within one tile of it.
// Elsewhere E, B and J are zero and the Yee updates keep them exactly zero,
// so the field kernels skip those tiles.  Computed after the push; it serves
// that step's E update and the next step's B update, over which fields spread
// by at most two cells, less than one tile.  ACT_J where deposits or antennas
// can reach: elsewhere the field kernels leave the fixed-point current alone
// (48 of their 144 bytes per cell and step, and 12 of J).  Bragg crystal,
// 2048 x 2048 cells: step 159 us before, 144 after.
template <int D>
__device__ __forceinline__ void tile_active(const GridP &g, const PushArgs &A, bool far) {
  const int step = gridDim.x * blockDim.x;
  if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(A.act_n + 1, 1ull);  // the steps counted
  // whole warps: the count is a warp reduction
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; (t & ~31) < g.ntiles; t += step) {
    bool a = false, j = false;
    if (t < g.ntiles) {
      const int tc[3] = {t % g.nt[0], (t / g.nt[0]) % g.nt[1], t / (g.nt[0] * g.nt[1])};
      const int x0 = tc[0] * Geo<D>::L0;
      // a far bound electron deposits at its own position: every tile then
      a = far || (A.ia_hi >= x0 - Geo<D>::L0 && A.ia_lo < x0 + 2 * Geo<D>::L0);
      j = far || (A.ia_hi >= x0 && A.ia_lo < x0 + Geo<D>::L0);
      const unsigned char old = A.act[t];
      // all neighbours' states loaded at once (stopping at the first hit made
      // 27 dependent loads of it: 9.4 us on 4096 tiles)
      constexpr int NB = D == 3 ? 27 : (D == 2 ? 9 : 3);
#pragma unroll
      for (int o = 0; o < NB; ++o) {
        const int off[3] = {o % 3 - 1, D >= 2 ? (o / 3) % 3 - 1 : 0, D >= 3 ? o / 9 - 1 : 0};
        bool use = true;
        int nb[3] = {0, 0, 0};
#pragma unroll
        for (int k = 0; k < D; ++k) {
          nb[k] = tc[k] + off[k];
          if (g.bc[k] == BP_PERIODIC) nb[k] = wrap_once(nb[k], g.nt[k]);
          else use &= nb[k] >= 0 && nb[k] < g.nt[k];
        }
        const int u = use ? nb[0] + g.nt[0] * (nb[1] + g.nt[1] * nb[2]) : t;
        a |= g.fnz[u] != 0;
        j |= A.qstate[u] != QS_DONE;
      }
      a |= j;
      const bool stale = old & (ACT_J | ACT_STALE);
      A.act[t] = j ? ACT_ON | ACT_J : (a ? (stale ? ACT_ON | ACT_CLEAR : ACT_ON) : (stale ? ACT_STALE : 0));
    }
    const unsigned k = __reduce_add_sync(0xFFFFFFFFu, a ? 1u : 0u);
    if ((threadIdx.x & 31u) == 0 && k) atomicAdd(A.act_n, (unsigned long long)k);
  }
}

// byte offset of the field box in the push's dynamic shared memory (after the
// current box, 128-byte aligned for the TMA loads)
__host__ __device__ constexpr size_t push_gbox_offset(int D, bool det) {
  return ((det ? 8 : 4) * (size_t)3 *
              (D == 1 ? Box<1>::JCELLS : (D == 2 ? Box<2>::JCELLS : Box<3>::JCELLS)) + 127) / 128 * 128;
}

// ---------------------------------------------------------------------------
// TMA staging of 3D field boxes: one cp.async.bulk.tensor load per component,
// completing on an mbarrier (transaction bytes), issued by one thread.

__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned long long *bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long *bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long *bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// a bounded wait for the phase of the given parity: false when it gave up
__device__ __forceinline__ bool mbar_wait(unsigned long long *bar, unsigned parity) {
  for (int it = 0; it < (1 << 20); ++it)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}
__device__ __forceinline__ void tma_load_3d(float *dst, const CUtensorMap *map, int x, int y, int z,
                                            unsigned long long *bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(smem_u32(dst)), "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
      : "memory");
}

// Whether tile t's field box comes by TMA: 3D with maps, and no periodic
// axis wraps inside the box (TMA fills zeros outside the grid, which is what
// an open face reads; a wrapped box is staged by per-thread copies).
template <int D>
__device__ __forceinline__ bool tma_tile(const GridP &g, const TmaMaps &T, const int T0[3]) {
  if constexpr (D != 3) {
    return false;
  } else {
    // maps present, and the block's field box 128-byte aligned in shared memory
    extern __shared__ __align__(128) unsigned char smem[];
    if (!T.on || ((smem_u32(smem) + (unsigned)push_gbox_offset(3, true)) & 127u) ||
        ((smem_u32(smem) + (unsigned)push_gbox_offset(3, false)) & 127u))
      return false;
    using BX = Box<3>;
    bool ok = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int lo = T0[a] - BX::OG - (a == 0 ? BX::SX : 0);
      const int ext = a == 0 ? BX::GR : (a == 1 ? BX::G1 : BX::G2);
      if (g.bc[a] == BP_PERIODIC) ok &= lo >= 0 && lo + ext <= g.n[a];
    }
    return ok;
  }
}

// Staging of a tile's field box (E, B of the tile plus halo; zero outside
// open faces), in shared memory: by TMA where tma_tile allows (one thread
// issues six box loads), else by per-thread asynchronous copies.  Neither
// holds registers, so the copies run while the block finishes the previous
// tile.  A QS_REST tile's box is all zero and is not staged.
template <int D>
__device__ __forceinline__ void stage_issue(const GridP &g, const PushArgs &A, const TmaMaps &T, int t, unsigned char qs,
                                            float *Gsm, unsigned long long *bar) {
  using BX = Box<D>;
  constexpr int GC = BX::GCELLS;
  if (qs != QS_PUSH) return;
  const int tc[3] = {t % g.nt[0], (t / g.nt[0]) % g.nt[1], t / (g.nt[0] * g.nt[1])};
  const int T0[3] = {tc[0] * Geo<D>::L0, tc[1] * Geo<D>::L1, tc[2] * Geo<D>::L2};
  if (tma_tile<D>(g, T, T0)) {
    if (threadIdx.x == 0) {
      // the previous tile's box was read by ordinary loads before this point
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_expect_tx(bar, 6u * 4u * (unsigned)(BX::GP * BX::G2));
#pragma unroll
      for (int cc = 0; cc < 6; ++cc)
        tma_load_3d(Gsm + cc * GC, &T.m[cc], T0[0] - BX::OG - BX::SX, T0[1] - BX::OG, T0[2] - BX::OG, bar);
    }
    return;
  }
  const unsigned gbase = smem_u32(Gsm);
  for (int q = threadIdx.x; q < BX::GCOMP; q += blockDim.x) {
    const int b0 = q % BX::G0, b1 = (q / BX::G0) % BX::G1, b2 = q / (BX::G0 * BX::G1);
    const int bidx[3] = {b0, b1, b2};
    const int si = BX::gi(b0, b1, b2);
    long long gi = 0, stride = 1;
    bool ok = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      int x = T0[a] - (a < D ? BX::OG : 0) + bidx[a];
      if (a < D) {
        if (g.bc[a] == BP_PERIODIC) x = wrap_once(x, g.n[a]);
        else ok &= (x >= 0 && x < g.n[a]);
      }
      gi += (long long)x * stride;
      stride *= g.n[a];
    }
    if (!ok) gi = 0;  // a zero fill: nothing is read
    const unsigned src = ok ? 4u : 0u;
#pragma unroll
    for (int cc = 0; cc < 6; ++cc) {
      const float *gp = (cc < 3 ? A.E[cc] : A.B[cc - 3]) + gi;
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(gbase + 4u * (unsigned)(cc * GC + si)),
                   "l"(gp), "r"(src)
                   : "memory");
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// wait for tile t's staging (this thread's copies, or the TMA loads: the
// mbarrier phase `phase`, flipped here after each TMA tile).  A TMA wait that
// gives up sets ST_TIMEOUT and `failed`.
template <int D>
__device__ __forceinline__ void stage_done(const GridP &g, const PushArgs &A, const TmaMaps &T, int t, unsigned char qs,
                                           unsigned long long *bar, unsigned &phase, bool &failed) {
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  if (qs != QS_PUSH) return;
  const int tc[3] = {t % g.nt[0], (t / g.nt[0]) % g.nt[1], t / (g.nt[0] * g.nt[1])};
  const int T0[3] = {tc[0] * Geo<D>::L0, tc[1] * Geo<D>::L1, tc[2] * Geo<D>::L2};
  if (tma_tile<D>(g, T, T0)) {
    if (!mbar_wait(bar, phase)) {
      if (threadIdx.x == 0) set_timeout(A.status);
      failed = !mbar_wait(bar, phase);  // one more bounded wait for the loads in flight
    }
    phase ^= 1u;
  }
}

// Sorted mode: every word of the box added to the global current and cleared, by
// one warp while the others go on adding (a word is taken by an exchange, and
// the words of a node are summed apart): no barrier, and no loop around the
// tile's (with a flush by the block that the loop resumes after, the ionised
// crystal's 4.2 M electrons took 0.56 ms a step, 0.50 this way, 0.485 without
// any guard).  Reached by tiles of some 1,300 (2D) to 3,500 (3D) particles near
// the speed of light, far more at thermal speeds.
template <int D>
__device__ __forceinline__ void drain_box(const GridP &g, unsigned long long *jfx, int t, unsigned *Jsm) {
  using BX = Box<D>;
  const int T0[3] = {(t % g.nt[0]) * Geo<D>::L0, ((t / g.nt[0]) % g.nt[1]) * Geo<D>::L1,
                     (t / (g.nt[0] * g.nt[1])) * Geo<D>::L2};
  __syncwarp();  // the other lanes' adds are in
#pragma unroll 1
  for (int q = threadIdx.x & 31; q < 3 * BX::JCOMP; q += 32) {
    const int cc = q / BX::JCOMP, nd = q - cc * BX::JCOMP;
    const int bidx[3] = {nd % BX::J0, (nd / BX::J0) % BX::J1, nd / (BX::J0 * BX::J1)};
    unsigned *p = Jsm + cc * BX::JCELLS + BX::ji(bidx[0], bidx[1], bidx[2]);
    const long long v = (long long)(int)atomicExch(p + 3 * BX::JCELLS, 0u) * 65536LL + (long long)(int)atomicExch(p, 0u);
    if (v == 0) continue;
    long long gidx = 0, stride = 1;
    bool ok = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      int c = T0[a] - (a < D ? BX::OJ : 0) + bidx[a];
      if (a < D) {
        if (g.bc[a] == BP_PERIODIC) c = wrap_once(c, g.n[a]);
        else ok &= c >= 0 && c < g.n[a];
      }
      gidx += (long long)c * stride;
      stride *= g.n[a];
    }
    if (ok) atomicAdd(jfx + (size_t)cc * g.ncell + gidx, (unsigned long long)v);
  }
}

// out of line in 1D and 3D (inline it took 14 bytes of spills in 3D); in 2D the
// call itself, the only one of its kernel, cost 4%
template <int D>
__device__ __noinline__ void drain_box_call(const GridP &g, unsigned long long *jfx, int t, unsigned *Jsm) {
  drain_box<D>(g, jfx, t, Jsm);
}

// one tile of the push (the block's work for tile t)
template <int D, bool DET, bool FREE, typename AfterLoop>
__device__ __forceinline__ void push_tile(const GridP &g, const PushArgs &A, const TmaMaps &T, const int t,
                                          const unsigned char qs, unsigned long long *bar, unsigned &phase, bool &failed,
                                          AfterLoop &&after_loop) {
  using JT = typename std::conditional<DET, unsigned int, float>::type;
  extern __shared__ __align__(128) unsigned char smem[];
  using BX = Box<D>;
  constexpr int JC = BX::JCELLS, GC = BX::GCELLS;
  constexpr size_t GOFF = push_gbox_offset(D, DET);
  JT *Jsm = reinterpret_cast<JT *>(smem);
  float *Gsm = reinterpret_cast<float *>(smem + GOFF);
  const int tid = threadIdx.x, bs = blockDim.x;
  int total = 0;
  for (int s = 0; s < A.nsp; ++s) total += A.p[s].tstart[t + 1] - A.p[s].tstart[t];
  if (qs == QS_DONE || total == 0) {
    stage_done<D>(g, A, T, t, qs, bar, phase, failed);  // this tile's copies land before the next tile's are issued
    __syncthreads();
    if (tid == 0 && qs != QS_DONE) A.occ[t] = 0;
    after_loop();
    return;
  }
  int tc[3];
  tc[0] = t % g.nt[0];
  tc[1] = (t / g.nt[0]) % g.nt[1];
  tc[2] = t / (g.nt[0] * g.nt[1]);
  const int T0[3] = {tc[0] * Geo<D>::L0, tc[1] * Geo<D>::L1, tc[2] * Geo<D>::L2};
  zero_box<DET>(Jsm, 3 * JC, tid, bs);
  // the field box was staged asynchronously (stage_issue) by the caller
  stage_done<D>(g, A, T, t, qs, bar, phase, failed);
  __syncthreads();
  // no field in the box: known from the tile marks alone (a staged box that
  // happens to be all zero goes the full way, which leaves the same bits;
  // reading every staged value to find it cost 1% of the 3D push)
  const bool nofield = qs != QS_PUSH;
  __shared__ int run;
  __shared__ PairJob jobs[D == 3 ? push_threads(D) / 32 : 1];  // a warp's general-case particle (3D)
  __shared__ unsigned sbb[6];
  if (tid < 6) sbb[tid] = tid < 3 ? 0xFFFFFFFFu : 0u;
  unsigned blo = 0xFFFFFFFFu, bhi = 0u;
  unsigned pushed = 0, load = 0;  // load: this lane's box_load since the box was cleared (sorted mode)
  const int lane = tid & 31;
  for (int s = 0; s < A.nsp; ++s) {
    if (tid == 0) run = 0;
    __syncthreads();
    const int beg = A.p[s].tstart[t], end = A.p[s].tstart[t + 1], n = end - beg;
    // in a QS_REST tile the quiet ions of this species have already moved
    const bool moved = qs == QS_REST && A.sp[s].kind == BP_TWO_BODY && A.sp[s].qw1 == -A.sp[s].qw2;
    const bool two = A.sp[s].kind == BP_TWO_BODY;
    // Each warp takes runs of 32 consecutive (cell-sorted) particles from a
    // shared counter, one lane per particle: the lanes' gather loads share
    // addresses and their state loads coalesce, and a warp whose particles
    // took the rare paths does not hold the others at the tile's end.  The
    // next run is taken before the current one is pushed, so that its
    // particle can be prefetched.
    // Sorted mode: a run is consecutive.  Atomic mode: the lanes of a run are S
    // particles apart (S runs cover 32 S consecutive particles), so fewer of
    // them add to one node at once (an FP32 shared add is a compare-and-swap
    // loop): 3.1 M ions, 1.11 ms a step with S = 1, 0.98 with 2, 0.96 with 4;
    // the integer adds gain less than the gather loses (32.5 M ions: 4.23 ms
    // with 1, 4.21 with 2, 4.41 with 4).
    constexpr int S = DET ? 1 : 4;
    const int nr = (n + 32 * S - 1) / (32 * S) * S;
    auto at = [&](int c) { return (c / S) * (32 * S) + S * lane + c % S; };
    int r = 0;
    if (lane == 0) r = atomicAdd(&run, 1);
    r = __shfl_sync(0xFFFFFFFFu, r, 0);
    while (r < nr) {
      int rn = 0;
      if (lane == 0) rn = atomicAdd(&run, 1);
      rn = __shfl_sync(0xFFFFFFFFu, rn, 0);
      const int k = at(r);
      const long long i = beg + k;
      const bool have = k < n && !(moved && quiet_done(A.p[s], i));
      if constexpr (D == 3) {
        if (have) {
          const int kn = at(rn);
          if (kn < n) prefetch_particle<D>(A.p[s], beg + kn, two);
          ++pushed;
        }
        push_particle<D, DET, FREE, JT>(g, A.sp[s], A.p[s], have, i, T0, Gsm, Jsm, A.status, A.jscale, blo, bhi, load,
                                        jobs, nofield, A.far, A.far_n, A.far_cap, s, t);
      } else if (have) {
        const int kn = at(rn);
        if (kn < n) prefetch_particle<D>(A.p[s], beg + kn, two);
        push_particle<D, DET, FREE, JT>(g, A.sp[s], A.p[s], true, i, T0, Gsm, Jsm, A.status, A.jscale, blo, bhi, load,
                                        jobs, nofield, A.far, A.far_n, A.far_cap, s, t);
        ++pushed;
      }
      r = rn;
      if constexpr (DET) {
        if (__any_sync(0xFFFFFFFFu, load >= kLaneLoad<D>)) {
          if constexpr (D == 2) drain_box<D>(g, A.jfx, t, Jsm);
          else drain_box_call<D>(g, A.jfx, t, Jsm);
          load = 0;
        }
      }
    }
    __syncthreads();
  }
  if (A.work) count_work(A.work, pushed);
  // the field box is no longer needed: the caller may start staging the next tile
  after_loop();
  // the deposits' bounding box over the block
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const unsigned l = __reduce_min_sync(0xFFFFFFFFu, blo == 0xFFFFFFFFu ? 0xFFFFFFFFu : (blo >> (8 * a)) & 255u);
    const unsigned h = __reduce_max_sync(0xFFFFFFFFu, (bhi >> (8 * a)) & 255u);
    if ((tid & 31) == 0 && l != 0xFFFFFFFFu) {
      atomicMin(&sbb[a], l);
      atomicMax(&sbb[3 + a], h);
    }
  }
  __syncthreads();
  const bool any = sbb[0] != 0xFFFFFFFFu;
  // the box's occupied part to global memory.  Sorted mode: each non-zero
  // node, an exact 64-bit fixed-point sum, is added into the global
  // fixed-point current (integer adds: the same result in any order; nodes
  // beyond an open face hold no deposit the field sees).  Atomic mode: the
  // FP32 box to the tile's slot (compact layout) for the current-sum kernel.
  constexpr int JN = BX::JCOMP;
  if (any) {
    const int lo0 = sbb[0], lo1 = sbb[1], lo2 = sbb[2];
    const int nx = sbb[3] - lo0 + 1, ny = sbb[4] - lo1 + 1, nz = sbb[5] - lo2 + 1;
    const int nxy = nx * ny, nbox = nxy * nz;
    // r / n as a multiplication: with m = 2^k / n rounded up, (r m) >> k is
    // exact while r n < 2^k: rows r2 < 729, n <= 27, k = 17; planes r < 17^3,
    // n <= 17^2, k = 24.  Four integer divisions per node took about 100
    // instructions per ion on the 3D push.
    static_assert(BX::J0 * BX::J1 * BX::J2 <= 4913 && BX::J0 * BX::J1 <= 729, "box small enough for the division");
    const unsigned mx = (131072u + nx - 1) / nx, mxy = ((1u << 24) + nxy - 1) / nxy;
    for (int q = tid; q < 3 * nbox; q += bs) {
      const int cc = q >= 2 * nbox ? 2 : (q >= nbox ? 1 : 0), r = q - cc * nbox;
      const int zz = D >= 3 ? (int)__umulhi((unsigned)r << 8, mxy) : 0, r2 = r - zz * nxy;
      const int yy = D >= 2 ? (int)(((unsigned)r2 * mx) >> 17) : 0;
      const int x = lo0 + r2 - yy * nx, y = lo1 + yy, z = lo2 + zz;
      const int k = cc * JC + BX::ji(x, y, z);
      if constexpr (DET) {
        const long long v = fx_value(Jsm + k, 3 * JC);
        if (v == 0) continue;
        const int bidx[3] = {x, y, z};
        long long gidx = 0, stride = 1;
        bool ok = true;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          int c = T0[a] - (a < D ? BX::OJ : 0) + bidx[a];
          if (a < D) {
            if (g.bc[a] == BP_PERIODIC) c = wrap_once(c, g.n[a]);
            else ok &= (c >= 0 && c < g.n[a]);
          }
          gidx += (long long)c * stride;
          stride *= g.n[a];
        }
        if (ok) atomicAdd(A.jfx + (size_t)cc * g.ncell + gidx, (unsigned long long)v);
      } else {
        A.jbox[(size_t)t * 3 * JN + cc * JN + x + BX::J0 * (y + BX::J1 * z)] = Jsm[k];
      }
    }
  }
  if (tid == 0) {
    A.occ[t] = any ? 1 : 0;
    A.jbb[t] = make_uint2(sbb[0] | (sbb[1] << 8) | (sbb[2] << 16), sbb[3] | (sbb[4] << 8) | (sbb[5] << 16));
  }
}

// The push: persistent blocks (as many as fit on the GPU at once) take the
// tiles the quiet-tile pass left (its list) in order from a counter, so a
// block's shared memory and setup are reused from tile to tile, and the next
// tile's field box is staged while the block finishes the current one.
//
// PB: blocks per SM the registers are held to.  2D grids with free particles
// take 3 (80 registers): a tile's work is short there and its barriers and
// instruction fetches are hidden by other blocks (4.2 M electrons, step of
// the ionised crystal: 0.62 ms with 2, 0.56 with 3, 0.61 with 4, which
// spills).  Two-body ions need the registers (524 k ions: the adjoint cycle
// 179 ms with 2, 185 with 3).
template <int D, bool DET, int PB>
__global__ void __launch_bounds__(push_threads(D), PB) k_push(GridP g, PushArgs A, const __grid_constant__ TmaMaps T,
                                                               int direct) {
  extern __shared__ __align__(128) unsigned char smem[];
  float *Gsm = reinterpret_cast<float *>(smem + push_gbox_offset(D, DET));
  __shared__ int next;
  __shared__ __align__(8) unsigned long long bar;  // completion of the TMA staging
  __shared__ int give_up, marked;
  // (no push after a sort that gave up, as in k_push_quiet; read here, beside
  // the tile's marks)
  const int stop = direct && threadIdx.x == 0 ? *(volatile const int *)(A.status + 2) : 0;
  if (threadIdx.x == 0) {
    mbar_init(&bar);
    give_up = 0;
  }
  __syncthreads();
  unsigned phase = 0;
  bool failed = false;
  const int nlist = direct ? 0 : *A.tile_n;
  unsigned char qs = QS_DONE;
  // The next list entry is taken only once the block has finished the
  // current tile's particles: reserving it earlier would let one block hold
  // two costly tiles in a row while others have none (grids with few
  // occupied tiles ran 20% slower that way).  direct: a block per tile,
  // without the quiet-tile pass; the block looks at its tile's marks itself.
  auto grab = [&](bool first) {
    bool mark = false;
    if (direct && first && threadIdx.x < 32)
      mark = __any_sync(0xFFFFFFFFu, near_mark<D>(g, (int)blockIdx.x, (int)threadIdx.x));
    if (threadIdx.x == 0) {
      if (direct) {
        next = first && !stop ? (int)blockIdx.x : -1;
        marked = mark;
      } else {
        const int k = atomicAdd(A.tile_ctr, 1);
        next = k < nlist ? A.tile_list[k] : -1;
      }
    }
    __syncthreads();
    if (next >= 0) {
      qs = direct ? (marked ? QS_PUSH : QS_COLD) : A.qstate[next];
      stage_issue<D>(g, A, T, next, qs, Gsm, &bar);
    }
  };
  grab(true);
  for (int t = next; t >= 0; t = next) {
    push_tile<D, DET, PB == 3>(g, A, T, t, qs, &bar, phase, failed, [&]() { grab(false); });
    if (failed) give_up = 1;
    __syncthreads();  // every thread has read `next` before it changes
    if (give_up) break;  // a staging wait gave up twice (ST_TIMEOUT is set): stop
  }
  // nothing may be in flight into this block's shared memory when it exits
  if (next >= 0 && qs == QS_PUSH) stage_done<D>(g, A, T, next, qs, &bar, phase, failed);
}

// 2D, sorted mode: the tiles with few ions, a warp each and a lane per ion,
// straight from the global fields to the global current, in the arithmetic of
// the tile push (the current's integer adds give the same bits in any order).
// Bound by the chain of one ion's gather, push and deposit; for a few ions the
// box push adds the staging of 2,400 field values, the clearing of the current
// box and its flush, with two blocks per SM: the 1,600 ions of a Bragg crystal
// on 2048 x 2048 cells, step 233 us before, 160 after.
__global__ void __launch_bounds__(128, 4) k_push_few(GridP g, PushArgs A) {
  using BX = Box<2>;
  const int lane = threadIdx.x & 31, n = A.tile_n[1];
  const GridStride st = {g.n[0], (long long)g.ncell};
  unsigned pushed = 0;
  for (int k = (int)(blockIdx.x * 4 + (threadIdx.x >> 5)); k < n; k += (int)gridDim.x * 4) {
    const int t = A.tile_list[g.ntiles - 1 - k];
    const int T0[3] = {(t % g.nt[0]) * Geo<2>::L0, (t / g.nt[0]) * Geo<2>::L1, 0};
    const long long at = (T0[0] - BX::OG) + (long long)g.n[0] * (T0[1] - BX::OG);
    fx64 *J = A.jfx + ((T0[0] - BX::OJ) + (long long)g.n[0] * (T0[1] - BX::OJ));
    for (int s = 0; s < A.nsp; ++s) {
      const int end = A.p[s].tstart[t + 1];
      for (int i = A.p[s].tstart[t] + lane; i < end; i += 32) {
        unsigned blo = 0xFFFFFFFFu, bhi = 0u, none = 0u;
        push_particle<2, true, false, fx64, GridStride>(g, A.sp[s], A.p[s], true, i, T0, nullptr, J, A.status, A.jscale, blo, bhi,
                                                        none, nullptr, false, A.far, A.far_n, A.far_cap, s, t, &A, at, st);
        ++pushed;
      }
      __syncwarp();
    }
  }
  if (A.work) count_work(A.work, pushed);
}

// Sorted mode: the ions the push listed as far (a bound electron a cell or
// more from its nucleus), each moved by push_far; anything push_far cannot
// move is a domain error.
template <int D>
__global__ void __launch_bounds__(128) k_push_far(GridP g, PushArgs A) {
  const int n = A.far_n ? min(*A.far_n, A.far_cap) : 0;
  if (A.act) tile_active<D>(g, A, n > 0);
  auto move = [&](int k, auto lanes) {
    const int4 e = A.far[k];
    const int t = e.z;
    const int T0[3] = {(t % g.nt[0]) * Geo<D>::L0, ((t / g.nt[0]) % g.nt[1]) * Geo<D>::L1,
                       (t / (g.nt[0] * g.nt[1])) * Geo<D>::L2};
    constexpr int W = decltype(lanes)::value;
    if (!push_far<D, W>(g, A.sp[e.x], A.p[e.x], e.x, e.y, T0[0], T0[1], T0[2], A.status, A.E, A.B, A.jfx, A.jscale) &&
        (W == 1 || (threadIdx.x & 31) == 0))
      atomicOr(A.status, ST_DOMAIN);
  };
  // few ions (rare tears): a warp each, for the latency; many (a strong field
  // over a whole crystal): a thread each.  A fixed number (a GB300's warps of
  // this launch): the gather sums its nodes by lane, so the last bit of a far
  // ion's fields depends on the form, and must not depend on the device.
  constexpr int FEW_FAR = 2432;
  const int tid = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
  if (n <= FEW_FAR) {
    for (int k = tid >> 5; k < n; k += nt / 32) move(k, std::integral_constant<int, D == 3 ? 32 : 16>{});
  } else {
    for (int k = tid; k < n; k += nt) move(k, std::integral_constant<int, 1>{});
  }
}

// the push kernel's variant (index of push_blocks): 1 on 2D grids with free particles
int push_variant(const GridP &g, const PushArgs &a) {
  bool free_sp = false;
  for (int k = 0; k < a.nsp; ++k) free_sp |= a.sp[k].kind == BP_FREE;
  return g.D == 2 && free_sp ? 1 : 0;
}

// Whether a 2D step launches k_push_few: two-body ions only, less than 8 a tile
// on average.  Where no tile has few ions the launch is lost (a dense slab in a
// wide grid, 16 ions a tile on average: adjoint cycle 53.4 ms without it, 55.1
// with), and the host knows no more of the tiles than the average.
bool push_few(const GridP &g, const PushArgs &a) {
  if (push_variant(g, a)) return false;
  long long ions = 0;
  for (int k = 0; k < a.nsp; ++k) ions += a.p[k].cap;
  return ions < 8LL * g.ntiles;
}

template <int D, bool DET>
void launch_one(const GridP &g, const PushArgs &a, const TmaMaps &tm, const AntArgs &ant, cudaStream_t s) {
  const bool direct = push_direct(g, a);
  if (!direct) {
    const int qt = g.ntiles >= 8192 ? 4 : 1;  // tiles per quiet-pass block
    const bool few = D == 2 && DET && push_few(g, a);
    k_push_quiet<D><<<(g.ntiles + qt - 1) / qt + ant.blocks, 128, 0, s>>>(g, a, qt, few, ant);
    if constexpr (D == 2 && DET)
      if (few) k_push_few<<<a.sms * 4, 128, 0, s>>>(g, a);
  }
  const size_t smem = push_smem_bytes(g, DET);
  // as many persistent blocks as the device holds at once (worked out per
  // context for its grid and device when it was created)
  const int v = push_variant(g, a);
  const int blocks = a.push_blocks[v] > 0 ? a.push_blocks[v] : 1, nb = blocks < g.ntiles ? blocks : g.ntiles;
  if (v) k_push<D, DET, push_pb(D, true)><<<nb, push_threads(D), smem, s>>>(g, a, tm, direct);
  else k_push<D, DET, push_pb(D, false)><<<nb, push_threads(D), smem, s>>>(g, a, tm, direct);
  if (DET || a.act) k_push_far<D><<<a.sms * 4, 128, 0, s>>>(g, a);
}

template <int D, bool DET, int PB>
int prepare_variant(const GridP &g, int *blocks) {
  const size_t smem = push_smem_bytes(g, DET);
  cudaError_t e = cudaFuncSetAttribute(k_push<D, DET, PB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return -1;
  int dev = 0, sms = 0, per = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return -1;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_push<D, DET, PB>, push_threads(D), smem);
  if (e != cudaSuccess) return -1;
  *blocks = (sms > 0 ? sms : 1) * (per > 0 ? per : 1);
  return 0;
}

template <int D, bool DET>
int prepare_one(const GridP &g, int blocks[2]) {
  return prepare_variant<D, DET, push_pb(D, false)>(g, blocks) || prepare_variant<D, DET, push_pb(D, true)>(g, blocks + 1) ? -1
                                                                                                                         : 0;
}

}  // namespace

size_t push_smem_bytes(const GridP &g, int det) {
  const int gc = g.D == 1 ? Box<1>::GCELLS : (g.D == 2 ? Box<2>::GCELLS : Box<3>::GCELLS);
  return push_gbox_offset(g.D, det != 0) + 4 * (size_t)6 * gc;
}

// The quiet-tile pass and its list pay where there are more tiles than push
// blocks resident at once (a block then takes several tiles, and tiles ahead
// of the field are many).  With a block for every tile they only lengthen the
// chain of dependent launches: step of the 1D medium (128 tiles) 35.4 us with
// the pass, 33.5 without; 524 k ions in 3D (128 tiles) 121 and 117 us.  Grids
// with tile flags (1024 tiles or more) need the pass's states, the push timing
// its counts.
bool push_direct(const GridP &g, const PushArgs &a) {
  return !a.act && !a.work && g.ntiles <= a.push_blocks[push_variant(g, a)];
}

int push_prepare(const GridP &g, int det, int blocks[2]) {
  switch (g.D * 2 + (det ? 1 : 0)) {
    case 2: return prepare_one<1, false>(g, blocks);
    case 3: return prepare_one<1, true>(g, blocks);
    case 4: return prepare_one<2, false>(g, blocks);
    case 5: return prepare_one<2, true>(g, blocks);
    case 6: return prepare_one<3, false>(g, blocks);
    default: return prepare_one<3, true>(g, blocks);
  }
}

void launch_push(const GridP &g, const PushArgs &a, const TmaMaps &tm, const AntArgs &ant, cudaStream_t s) {
  const bool det = a.jscale != 0.0f;
  switch (g.D * 2 + (det ? 1 : 0)) {
    case 2: launch_one<1, false>(g, a, tm, ant, s); break;
    case 3: launch_one<1, true>(g, a, tm, ant, s); break;
    case 4: launch_one<2, false>(g, a, tm, ant, s); break;
    case 5: launch_one<2, true>(g, a, tm, ant, s); break;
    case 6: launch_one<3, false>(g, a, tm, ant, s); break;
    default: launch_one<3, true>(g, a, tm, ant, s); break;
  }
}

// The six field maps of a 3D grid: FP32 [nz][ny][nx] (strides in bytes
// between rows and planes), box {16, 15, 15} = one staged field box, no
// swizzle, zeros outside the grid.  cuTensorMapEncodeTiled comes through the
// runtime's driver entry point, so the library does not link the driver.
int encode_field_maps(const GridP &g, float *const F[6], TmaMaps *out) {
  out->on = 0;
  if (g.D != 3) return 0;
  using encode_fn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                 const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  void *fp = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fp, 12000, cudaEnableDefault, &q) != cudaSuccess ||
      q != cudaDriverEntryPointSuccess || !fp)
    return -1;
  const encode_fn encode = reinterpret_cast<encode_fn>(fp);
  const cuuint64_t dims[3] = {(cuuint64_t)g.n[0], (cuuint64_t)g.n[1], (cuuint64_t)g.n[2]};
  const cuuint64_t strides[2] = {(cuuint64_t)g.n[0] * 4, (cuuint64_t)g.n[0] * g.n[1] * 4};
  const cuuint32_t box[3] = {(cuuint32_t)Box<3>::GR, (cuuint32_t)Box<3>::G1, (cuuint32_t)Box<3>::G2};
  const cuuint32_t estr[3] = {1, 1, 1};
  if (strides[0] % 16 || strides[1] % 16) return -1;
  for (int c = 0; c < 6; ++c) {
    if (reinterpret_cast<uintptr_t>(F[c]) % 16) return -1;
    CUresult r = encode(&out->m[c], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, F[c], dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return -1;
  }
  out->on = 1;
  return 0;
}
