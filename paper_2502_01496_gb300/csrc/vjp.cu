// Vector-Jacobian product of one force evaluation with respect to positions
// and masses, through the same tree and interaction lists (topology, lists
// and smoothing lengths held fixed).  The paper has no adjoint; this is the
// derivative of the evaluation of Sec. 2 (Eqs. 3, 6, 7, 8, 13).  FP64 mode
// runs every step in float64; mixed mode runs the M2L and P2P reverses with
// float32 terms (as its forward does) and sums of float64 or wider (a source's
// terms over the particles of one target leaf are added in float32 first).
//
// a_i = sum_{j in near(leaf i), j != i} m_j K(x_i - x_j)            (P2P)
//     + L(C_alpha, x_i - com_alpha)                                (L2P, Eq. 8)
// C_alpha = sum_{beta in far(alpha)} C(com_alpha - com_beta, M_beta, Q_beta)   (M2L, Eq. 6)
// with M, com = S/M (S = sum m x) and Q (Eq. 7) functions of the particles.
//
// Reverse order: L2P (cotangents of each leaf's expansion and of x_i, com),
// M2L (cotangents of r = com_alpha - com_beta, M_beta, Q_beta: C is linear in M
// and Q, its r-derivatives come from dual numbers), P2P on the target side and
// on the source side, then the moments: per cell the
// cotangents (M_bar, com_bar, Q_bar) give m_bar_i and x_bar_i as a quadratic
// polynomial in x_i, summed over the leaf's chain of ancestors.
#include <algorithm>
#include <climits>
#include <type_traits>

#include "kdfmm_internal.cuh"

namespace kdfmm {

namespace {

inline unsigned blocks_for(int64_t n, int threads) { return (unsigned)((n + threads - 1) / threads); }

// ---------------------------------------------------------------------------
// M2L coefficients (same closed forms as the forward) on float32 dual numbers
// ---------------------------------------------------------------------------
// d: the derivatives with respect to the three components of r.
struct Dual {
  float v, d[3];
};
__device__ __forceinline__ Dual operator+(const Dual& a, const Dual& b) {
  return Dual{a.v + b.v, {a.d[0] + b.d[0], a.d[1] + b.d[1], a.d[2] + b.d[2]}};
}
__device__ __forceinline__ Dual operator-(const Dual& a, const Dual& b) {
  return Dual{a.v - b.v, {a.d[0] - b.d[0], a.d[1] - b.d[1], a.d[2] - b.d[2]}};
}
__device__ __forceinline__ Dual operator-(const Dual& a) {
  return Dual{-a.v, {-a.d[0], -a.d[1], -a.d[2]}};
}
__device__ __forceinline__ Dual operator*(const Dual& a, const Dual& b) {
  return Dual{a.v * b.v,
              {a.d[0] * b.v + a.v * b.d[0], a.d[1] * b.v + a.v * b.d[1], a.d[2] * b.v + a.v * b.d[2]}};
}
__device__ __forceinline__ Dual& operator+=(Dual& a, const Dual& b) { return a = a + b; }

__device__ __forceinline__ float rsq(float v) { return rsqrtf(v); }

__device__ __forceinline__ Dual rsqrt_dual(const Dual& a) {
  const float r = rsq(a.v);
  const float dr = -0.5f * r / a.v;
  return Dual{r, {dr * a.d[0], dr * a.d[1], dr * a.d[2]}};
}
// A constant.
__device__ __forceinline__ Dual lift(float v) { return Dual{v, {0.f, 0.f, 0.f}}; }

__device__ __forceinline__ Dual c2e(int a, int b, const Dual R[3], const Dual u[3],
                                    const Dual Qm[3][3], Dual s1, Dual s2, Dual t2, Dual t3) {
  Dual v = s2 * R[a] * R[b] + t3 * (R[a] * u[b] + R[b] * u[a]) + t2 * Qm[a][b];
  if (a == b) v += s1;
  return v;
}

__device__ __forceinline__ Dual c3e(int a, int b, int c, const Dual R[3], const Dual u[3],
                                    const Dual Qm[3][3], Dual s2, Dual s3, Dual t3, Dual t4) {
  Dual d = lift(0.0f), du = lift(0.0f);
  if (a == b) { d += R[c]; du += u[c]; }
  if (a == c) { d += R[b]; du += u[b]; }
  if (b == c) { d += R[a]; du += u[a]; }
  return s3 * R[a] * R[b] * R[c] + s2 * d +
         t4 * (R[b] * R[c] * u[a] + R[a] * R[c] * u[b] + R[a] * R[b] * u[c]) +
         t3 * (R[a] * Qm[b][c] + R[b] * Qm[a][c] + R[c] * Qm[a][b] + du);
}

// sum_j w_j C_j over the 20 compact coefficients C0, C1 (3), C2 (6), C3 (10)
// of the potential Phi = -M/R - Q_jk R_j R_k / (2 R^5) and its derivatives
// (the closed forms of m2l.cu); contracting as each coefficient is formed
// keeps one accumulator instead of twenty.
// STD: the standard p = 3 series -- the quadrupole keeps only its C0 and C1
// terms (as in m2l.cu).
template <bool STD>
__device__ Dual m2l_contract(const Dual R[3], float M, const float Q[6], const float w[20]) {
  const Dual Qm[3][3] = {{lift(Q[0]), lift(Q[1]), lift(Q[2])},
                         {lift(Q[1]), lift(Q[3]), lift(Q[4])},
                         {lift(Q[2]), lift(Q[4]), lift(Q[5])}};
  const Dual R2 = R[0] * R[0] + R[1] * R[1] + R[2] * R[2];
  const Dual g0 = rsqrt_dual(R2);
  const Dual i2 = g0 * g0;
  const Dual g1 = -(g0 * i2);
  const Dual g2 = lift(-3.0f) * g1 * i2;
  const Dual g3 = lift(-5.0f) * g2 * i2;
  const Dual g4 = lift(-7.0f) * g3 * i2;
  const Dual g5 = lift(-9.0f) * g4 * i2;
  Dual u[3];
  for (int i = 0; i < 3; ++i) u[i] = Qm[i][0] * R[0] + Qm[i][1] * R[1] + Qm[i][2] * R[2];
  const Dual q = R[0] * u[0] + R[1] * u[1] + R[2] * u[2];
  const Dual qs = q * lift((float)(1.0 / 6.0));
  const Dual Mt = lift(M);
  const Dual s1 = -(Mt * g1) - g3 * qs;
  const Dual t2 = g2 * lift((float)(-1.0 / 3.0));
  Dual acc = lift(w[0]) * (-(Mt * g0) - g2 * qs);
  for (int i = 0; i < 3; ++i) acc += lift(w[1 + i]) * (s1 * R[i] + t2 * u[i]);
  const Dual s1h = STD ? -(Mt * g1) : s1;
  const Dual s2 = STD ? -(Mt * g2) : -(Mt * g2) - g4 * qs;
  const Dual s3 = STD ? -(Mt * g3) : -(Mt * g3) - g5 * qs;
  const Dual t2h = STD ? lift(0.0f) : t2;
  const Dual t3 = STD ? lift(0.0f) : g3 * lift((float)(-1.0 / 3.0));
  const Dual t4 = STD ? lift(0.0f) : g4 * lift((float)(-1.0 / 3.0));
  const int c2a[6] = {0, 0, 0, 1, 1, 2}, c2b[6] = {0, 1, 2, 1, 2, 2};
#pragma unroll
  for (int k = 0; k < 6; ++k) acc += lift(w[4 + k]) * c2e(c2a[k], c2b[k], R, u, Qm, s1h, s2, t2h, t3);
  const int c3a[10] = {0, 0, 0, 0, 0, 0, 1, 1, 1, 2}, c3b[10] = {0, 0, 0, 1, 1, 2, 1, 1, 2, 2},
            c3c[10] = {0, 1, 2, 1, 2, 2, 1, 2, 2, 2};
#pragma unroll
  for (int k = 0; k < 10; ++k)
    acc += lift(w[10 + k]) * c3e(c3a[k], c3b[k], c3c[k], R, u, Qm, s2, s3, t3, t4);
  return acc;
}

// ---------------------------------------------------------------------------
// kernels
// ---------------------------------------------------------------------------
struct VjpArgs {
  int64_t n;
  int nleaves, ncells;
  bool mixed;
  const int32_t* leaf_sys;
  const double* sys_eps;
  const int32_t* leaf_cells;
  const int32_t* leaf_rank;
  Cells c;
  PCols tp;
  const float4* ph;                     // (1/h, 1/h^3, h, (2h)^2) float32
  const float* lexp32;
  const double* lexp64;
  const int32_t *far_cnt, *far_idx, *near_cnt, *near_idx;
  const int64_t *far_off, *near_off;
  int64_t cap_far, cap_near;            // entries a list may hold
  double* ab;                           // cotangent in tree order (N x 3; FP64 mode)
  double* hinv;                         // 1 / h in tree order (FP64 mode, M4 kernel)
  const int32_t* sys_root;
  // mixed mode, tree order: the position on three float32 grids (split_grid),
  // q0 = (x0, m), q1 = (x1, 1 / h), q2 = (x2, first component of a_bar), q3 the other two
  float4 *q0, *q1, *q2;
  float2* q3;
  double* xbar;                         // tree order (N x 3)
  double* xsrc;                         // P2P source-side part of x_bar (N x 3, atomics)
  double* msrc;                         // P2P source-side part of m_bar (N, atomics)
  double* cbar;                         // per leaf: 20 expansion cotangents
  double* cell_bar;                     // per cell: M_bar, com_bar (3), Q_bar (6)
  // near lists and transposed near lists are cut into pieces of `entries`:
  // piece 0 is the leaf's own work item, the others extra items after the leaves
  // (seg_leaf: their leaf; seg_first: a leaf's first extra item); the targets'
  // partial sums of the extra items (seg_part) are added in piece order
  int entries;
  int32_t *seg_first, *seg_leaf;
  double* seg_part;
  int64_t seg_cap;
  // transposed near lists: leaf ordinal r is a source of the target leaves
  // tidx[toff[r] ...) (ordinals), tcnt[r] of them
  int32_t *tcnt, *tcur, *tidx;
  int64_t* toff;
  int64_t tcap;                         // entries of tidx
  int32_t *tseg_leaf, *tseg_first;
  int64_t tseg_cap;
  // [0] entries reserved, [1] extra source items, [2] extra target items, [3] and
  // [4] target and source items with close pairs (mixed mode), listed in close_t, close_s
  unsigned long long* tctr;
  int32_t *close_t, *close_s;
};

// A coordinate as x0 + x1 + x2 on the grids 2^(k-22), 2^(k-45) and 2^(k-68) of
// its system (|x| <= 2^k): the difference of two coordinates is then three
// exact float32 subtractions, and grid_diff their sum rounded to float32, without
// the float64 pipe (1/64 rate).  A coordinate below 2^(k-16) may have bits under
// the last grid: the difference is off by less than 2^(k-68), so pairs closer
// than 2^(k-36) take the float64 difference, and for the others that is 2^-32 of
// their distance at most, against the 2^-25 of float32's rounding.  An item that
// meets such a pair (close_pairs) is left to the float64-difference form of its
// kernel: the branch within the loop cost the 2^20 Plummer sphere's call 5 % by
// the registers it took.
__device__ __forceinline__ int grid_exponent(double bound) {
  return max(((__double2hiint(bound) >> 20) & 0x7ff) - 1022, -900);           // bound < 2^k
}
// Bound on the |coordinates| of a leaf's system.
__device__ __forceinline__ double system_bound(const VjpArgs& V, int leaf) {
  const int root = V.sys_root[V.leaf_sys[leaf]];
  return fmax(fabs(V.c.cx[root]), fmax(fabs(V.c.cy[root]), fabs(V.c.cz[root]))) + V.c.s[root];
}
// Whether an item whose smallest r^2 is `lowest` has a pair closer than that: its
// r^2 is below 2^(2 (k - 36)), but no less than the smallest normal number (the
// grids' own underflow is 2^-149).  Always from 2^100 on, where a coordinate may
// leave float32.
__device__ __forceinline__ bool close_pairs(float lowest, double bound) {
  const int e = 2 * (grid_exponent(bound) - 36);
  return e > 127 || lowest < __int_as_float((max(e, -126) + 127) << 23);
}
struct GridScale {
  double c0, c1, c2;                    // adding and subtracting rounds to the grid
};
__device__ __forceinline__ GridScale grid_scale(double bound) {
  const int k = grid_exponent(bound);
  GridScale g;
  g.c0 = __hiloint2double((min(k + 30, 1023) + 1023) << 20 | 0x80000, 0);     // 1.5 * 2^(k+30)
  g.c1 = __hiloint2double((k + 7 + 1023) << 20 | 0x80000, 0);
  g.c2 = __hiloint2double((k - 16 + 1023) << 20 | 0x80000, 0);
  return g;
}
__device__ __forceinline__ void split_grid(double x, const GridScale& g, float& x0, float& x1,
                                           float& x2) {
  const double a = __dsub_rn(__dadd_rn(x, g.c0), g.c0), r = __dsub_rn(x, a);
  const double b = __dsub_rn(__dadd_rn(r, g.c1), g.c1), q = __dsub_rn(r, b);
  x0 = (float)a;
  x1 = (float)b;
  x2 = (float)__dsub_rn(__dadd_rn(q, g.c2), g.c2);
}
__device__ __forceinline__ float grid_diff(float a0, float a1, float a2, float b0, float b1,
                                           float b2) {
  const float d0 = __fsub_rn(a0, b0), d1 = __fsub_rn(a1, b1), d2 = __fsub_rn(a2, b2);
  const float s = __fadd_rn(d0, d1);
  const float e = __fsub_rn(d1, __fsub_rn(s, d0));            // |d0| >= |d1| or d0 = 0
  // s + e + d2 rounded once: the tail is cut off with its last bit set when
  // anything was lost, so that it cannot make a tie of what is none
  float r = __fadd_rz(e, d2);
  if (__fsub_rn(d2, __fsub_rn(r, e)) != 0.0f) r = __int_as_float(__float_as_int(r) | 1);
  return __fadd_rn(s, r);
}

// L2P reverse: warp per leaf, lane per particle.  a_i = -(C1 + C2 x + C3 x x / 2)
// with x = x_i - com_alpha.  Also brings the cotangent into tree order and
// prepares the particle records of the P2P reverse.
// Bound by the float64 pipe (1/64 rate): the lanes form the particles' 19
// monomials b x x in parallel (29 float64 operations a warp), and lane j sums
// monomial j over the leaf's particles from shared memory (11 additions a
// leaf of 11), instead of butterflies over 23 values (115 additions).
constexpr int kL2PWarps = 4;
__global__ void __launch_bounds__(kL2PWarps * 32) k_vjp_l2p(const double* __restrict__ abar, VjpArgs V,
                                                         bool m4) {
  __shared__ double s_c[kL2PWarps][20];
  __shared__ double s_v[kL2PWarps][22][33];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k = blockIdx.x * kL2PWarps + w;
  if (k >= V.nleaves) return;
  const int a = V.leaf_cells[k];
  const int f = V.c.first[a], cnt = V.c.count[a];
  double* C = s_c[w];
  if (lane < 20) {
    if (V.mixed) {
      const float* e = V.lexp32 + 24 * (int64_t)k;
      double v = (double)e[lane];
      if (lane < 4) v += (double)e[20 + lane];
      C[lane] = v;
    } else {
      C[lane] = V.lexp64[20 * (int64_t)k + lane];
    }
  }
  __syncwarp();
  double (*vals)[33] = s_v[w];
  if (lane < cnt) {
    const int64_t p = (int64_t)f + lane, i = V.tp.idx[p];
    const double x = V.tp.x[p] - V.c.cx[a], y = V.tp.y[p] - V.c.cy[a], z = V.tp.z[p] - V.c.cz[a];
    const double b0 = abar[3 * i], b1 = abar[3 * i + 1], b2 = abar[3 * i + 2];
    if (V.mixed) {
      const GridScale g = grid_scale(system_bound(V, k));
      float4 u0, u1, u2;
      split_grid(V.tp.x[p], g, u0.x, u1.x, u2.x);
      split_grid(V.tp.y[p], g, u0.y, u1.y, u2.y);
      split_grid(V.tp.z[p], g, u0.z, u1.z, u2.z);
      u0.w = (float)V.tp.m[p];
      u1.w = m4 ? 1.0f / (float)V.tp.h[p] : 0.0f;
      u2.w = (float)b0;
      V.q0[p] = u0;
      V.q1[p] = u1;
      V.q2[p] = u2;
      V.q3[p] = make_float2((float)b1, (float)b2);
    } else {
      V.ab[3 * p] = b0;
      V.ab[3 * p + 1] = b1;
      V.ab[3 * p + 2] = b2;
      if (m4) V.hinv[p] = 1.0 / V.tp.h[p];
    }
    // (d a_i / d x_j) = -N_ij, N_ij = C2_ij + C3_ijk x_k: g_j = -sum_i b_i N_ij
    const double n00 = C[4] + C[10] * x + C[11] * y + C[12] * z;
    const double n01 = C[5] + C[11] * x + C[13] * y + C[14] * z;
    const double n02 = C[6] + C[12] * x + C[14] * y + C[15] * z;
    const double n11 = C[7] + C[13] * x + C[16] * y + C[17] * z;
    const double n12 = C[8] + C[14] * x + C[17] * y + C[18] * z;
    const double n22 = C[9] + C[15] * x + C[18] * y + C[19] * z;
    const double g0 = -(b0 * n00 + b1 * n01 + b2 * n02);
    const double g1 = -(b0 * n01 + b1 * n11 + b2 * n12);
    const double g2 = -(b0 * n02 + b1 * n12 + b2 * n22);
    V.xbar[3 * p] = g0;
    V.xbar[3 * p + 1] = g1;
    V.xbar[3 * p + 2] = g2;
    // expansion cotangents: a_i depends on C1_i, C2_ij x_j, 1/2 C3_ijk x_j x_k
    // (monomials here; their factors -1, -1/2 follow the sum)
    const double xx = b0 * x, xy = b0 * y, xz = b0 * z, yx = b1 * x, yy = b1 * y, yz = b1 * z,
                 zx = b2 * x, zy = b2 * y, zz = b2 * z;
    const double sxy = xy + yx, sxz = xz + zx, syz = yz + zy;
    vals[1][lane] = b0; vals[2][lane] = b1; vals[3][lane] = b2;
    vals[4][lane] = xx; vals[5][lane] = sxy; vals[6][lane] = sxz;
    vals[7][lane] = yy; vals[8][lane] = syz; vals[9][lane] = zz;
    vals[10][lane] = xx * x;
    vals[11][lane] = x * (sxy + xy);
    vals[12][lane] = x * (sxz + xz);
    vals[13][lane] = y * (sxy + yx);
    vals[14][lane] = xy * z + x * syz;
    vals[15][lane] = z * (sxz + zx);
    vals[16][lane] = yy * y;
    vals[17][lane] = y * (syz + yz);
    vals[18][lane] = z * (syz + zy);
    vals[19][lane] = zz * z;
    vals[0][lane] = g0; vals[20][lane] = g1; vals[21][lane] = g2;
  }
  __syncwarp();
  if (lane < 22) {
    double s = 0.0;
    for (int j = 0; j < cnt; ++j) s += vals[lane][j];
    if (lane >= 1 && lane < 20) {
      const double scale = lane < 10 || lane == 14 ? -1.0 : -0.5;
      V.cbar[20 * (int64_t)k + lane] = scale * s;
    } else {
      // x = x_i - com_alpha: the com receives minus the particles' share
      if (lane == 0) V.cbar[20 * (int64_t)k] = 0.0;
      atomicAdd(&V.cell_bar[10 * (int64_t)a + (lane == 0 ? 1 : lane - 18)], -s);
    }
  }
}

// M2L reverse: warp per sink leaf, lanes over its far cells.  Mixed mode is bound
// by float32 issue (some 2500 instructions a pair, three quarters of them the
// dual numbers): the cotangents of M and Q, which needed seven contractions with
// mostly zero terms (15.8 ms on the 2^20 Plummer sphere, 1.32e8 pairs; 12.5 now), are
// written without those terms.  A far cell's ten
// cotangents (M_bar, com_bar, Q_bar) go to float64 atomics through shared
// memory, so that a warp instruction adds 32 consecutive values (about three
// cells) instead of one value of 32 scattered cells.
constexpr int kM2LWarps = 4;
struct CellBuf {
  double v[32 * 11];                    // 10 per lane, stride 11 against bank conflicts
  int cell[32];
};
__device__ __forceinline__ void cell_buf_add(const VjpArgs& V, CellBuf& B, int lane, int n) {
  __syncwarp();
  for (int i = lane; i < 10 * n; i += 32) {
    const int c = i / 10, q = i - 10 * c;
    atomicAdd(&V.cell_bar[10 * (int64_t)B.cell[c] + q], B.v[11 * c + q]);
  }
  __syncwarp();
}

// The cotangent of M: sum_j w_j C_j for M = 1, Q = 0, in the operations and
// the order of m2l_contract (float32) without its terms that are exactly zero.
struct GTerms {
  float g[6];                           // g_n of R
  float t2, t3, t4;
};
__device__ __forceinline__ GTerms g_terms(const float R[3]) {
  GTerms G;
  const float R2 = __fadd_rn(__fadd_rn(__fmul_rn(R[0], R[0]), __fmul_rn(R[1], R[1])),
                             __fmul_rn(R[2], R[2]));
  G.g[0] = rsqrtf(R2);
  const float i2 = __fmul_rn(G.g[0], G.g[0]);
  G.g[1] = -__fmul_rn(G.g[0], i2);
#pragma unroll
  for (int n = 2; n < 6; ++n) G.g[n] = __fmul_rn(__fmul_rn((float)(1 - 2 * n), G.g[n - 1]), i2);
  const float third = (float)(-1.0 / 3.0);
  G.t2 = __fmul_rn(G.g[2], third);
  G.t3 = __fmul_rn(G.g[3], third);
  G.t4 = __fmul_rn(G.g[4], third);
  return G;
}

constexpr int kC2[6][2] = {{0, 0}, {0, 1}, {0, 2}, {1, 1}, {1, 2}, {2, 2}};
constexpr int kC3[10][3] = {{0, 0, 0}, {0, 0, 1}, {0, 0, 2}, {0, 1, 1}, {0, 1, 2},
                            {0, 2, 2}, {1, 1, 1}, {1, 1, 2}, {1, 2, 2}, {2, 2, 2}};

// s3 R_a R_b R_c + s2 (d_ab R_c + d_ac R_b + d_bc R_a)
template <int a, int b, int c>
__device__ __forceinline__ float c3_radial(const float R[3], float s2, float s3) {
  const float p = __fmul_rn(__fmul_rn(s3, R[a]), R[b]);
  if constexpr (a == b && b == c) {
    return __fmaf_rn(s2, __fadd_rn(__fadd_rn(R[a], R[a]), R[a]), __fmul_rn(p, R[c]));
  } else if constexpr (a == b || b == c) {
    return __fmaf_rn(s2, a == b ? R[c] : R[a], __fmul_rn(p, R[c]));
  } else {
    return __fmul_rn(p, R[c]);
  }
}

template <int K>
__device__ __forceinline__ float mass_c2(const float R[3], float s1, float s2, const float* w, float acc) {
  constexpr int a = kC2[K][0], b = kC2[K][1];
  float v = __fmul_rn(__fmul_rn(s2, R[a]), R[b]);
  if (a == b) v = __fadd_rn(v, s1);
  return __fmaf_rn(w[4 + K], v, acc);
}
template <int K>
__device__ __forceinline__ float mass_c3(const float R[3], float s2, float s3, const float* w, float acc) {
  return __fmaf_rn(w[10 + K], c3_radial<kC3[K][0], kC3[K][1], kC3[K][2]>(R, s2, s3), acc);
}
__device__ __forceinline__ float mass_cotangent(const float R[3], const GTerms& G, const float w[20]) {
  const float s1 = -G.g[1], s2 = -G.g[2], s3 = -G.g[3];
  float acc = 0.0f;
#pragma unroll
  for (int i = 0; i < 3; ++i) acc = __fmaf_rn(w[1 + i], __fmul_rn(s1, R[i]), acc);
  acc = mass_c2<0>(R, s1, s2, w, acc); acc = mass_c2<1>(R, s1, s2, w, acc);
  acc = mass_c2<2>(R, s1, s2, w, acc); acc = mass_c2<3>(R, s1, s2, w, acc);
  acc = mass_c2<4>(R, s1, s2, w, acc); acc = mass_c2<5>(R, s1, s2, w, acc);
  acc = mass_c3<0>(R, s2, s3, w, acc); acc = mass_c3<1>(R, s2, s3, w, acc);
  acc = mass_c3<2>(R, s2, s3, w, acc); acc = mass_c3<3>(R, s2, s3, w, acc);
  acc = mass_c3<4>(R, s2, s3, w, acc); acc = mass_c3<5>(R, s2, s3, w, acc);
  acc = mass_c3<6>(R, s2, s3, w, acc); acc = mass_c3<7>(R, s2, s3, w, acc);
  acc = mass_c3<8>(R, s2, s3, w, acc); acc = mass_c3<9>(R, s2, s3, w, acc);
  return acc;
}

// The cotangent of Q_ij (i = A, j = B, A <= B): sum_j w_j C_j for M = 0 and the
// unit Q_ij = Q_ji = 1, likewise.  u = Q R has u_A = R_B, u_B = R_A.
template <int A, int B>
struct UnitQ {
  // u_i is R[ui(i)], or zero (-1)
  __host__ __device__ static constexpr int ui(int i) { return i == A ? B : (i == B ? A : -1); }
  __host__ __device__ static constexpr bool q(int i, int j) {
    return (i == A && j == B) || (i == B && j == A);
  }
};
// sum of the non-zero of two terms x y, contracted as fma(x0, y0, x1 y1)
template <bool Z0, bool Z1>
__device__ __forceinline__ float sum2(float x0, float y0, float x1, float y1) {
  if constexpr (Z0 && Z1) return 0.0f;
  else if constexpr (Z0) return __fmul_rn(x1, y1);
  else if constexpr (Z1) return __fmul_rn(x0, y0);
  else return __fmaf_rn(x0, y0, __fmul_rn(x1, y1));
}
template <int A, int B, int K>
__device__ __forceinline__ float q_c2(const float R[3], const GTerms& G, float s1, float s2,
                                      const float* w, float acc) {
  using U = UnitQ<A, B>;
  constexpr int a = kC2[K][0], b = kC2[K][1], ua = U::ui(a), ub = U::ui(b);
  const float p = __fmul_rn(s2, R[a]);
  float v;
  if constexpr (ua < 0 && ub < 0) {
    v = __fmul_rn(p, R[b]);
  } else {
    const float in = sum2<(ub < 0), (ua < 0)>(R[a], R[ub < 0 ? 0 : ub], R[b], R[ua < 0 ? 0 : ua]);
    v = __fmaf_rn(p, R[b], __fmul_rn(G.t3, in));
  }
  if (U::q(a, b)) v = __fadd_rn(v, G.t2);
  if (a == b) v = __fadd_rn(v, s1);
  return __fmaf_rn(w[4 + K], v, acc);
}
template <int A, int B, int K>
__device__ __forceinline__ float q_c3(const float R[3], const GTerms& G, float s2, float s3,
                                      const float* w, float acc) {
  using U = UnitQ<A, B>;
  constexpr int a = kC3[K][0], b = kC3[K][1], c = kC3[K][2];
  constexpr int ua = U::ui(a), ub = U::ui(b), uc = U::ui(c);
  float v = c3_radial<a, b, c>(R, s2, s3);
  if constexpr (ua >= 0 || ub >= 0 || uc >= 0) {
    float x = sum2<(ua < 0), (ub < 0)>(__fmul_rn(R[b], R[c]), R[ua < 0 ? 0 : ua],
                                       __fmul_rn(R[a], R[c]), R[ub < 0 ? 0 : ub]);
    if constexpr (uc >= 0) {
      if constexpr (ua < 0 && ub < 0) x = __fmul_rn(__fmul_rn(R[a], R[b]), R[uc]);
      else x = __fmaf_rn(__fmul_rn(R[a], R[b]), R[uc], x);
    }
    v = __fmaf_rn(G.t4, x, v);
  }
  constexpr bool e0 = U::q(b, c), e1 = U::q(a, c), e2 = U::q(a, b);
  constexpr bool d0 = a == b && uc >= 0, d1 = a == c && ub >= 0, d2 = b == c && ua >= 0;
  if constexpr (e0 || e1 || e2 || d0 || d1 || d2) {
    float y = 0.0f, du = 0.0f;
    if constexpr (e0) y = R[a];
    if constexpr (e1) y = __fadd_rn(y, R[b]);
    if constexpr (e2) y = __fadd_rn(y, R[c]);
    if constexpr (d0) du = R[uc];
    if constexpr (d1) du = __fadd_rn(du, R[ub]);
    if constexpr (d2) du = __fadd_rn(du, R[ua]);
    v = __fmaf_rn(G.t3, __fadd_rn(y, du), v);
  }
  return __fmaf_rn(w[10 + K], v, acc);
}
template <int A, int B, bool STD>
__device__ __forceinline__ float q_cotangent(const float R[3], const GTerms& G, const float w[20]) {
  using U = UnitQ<A, B>;
  const float q = A == B ? __fmul_rn(R[A], R[A]) : __fmaf_rn(R[A], R[B], __fmul_rn(R[A], R[B]));
  const float qs = __fmul_rn(q, (float)(1.0 / 6.0));
  const float s1 = -__fmul_rn(G.g[3], qs);
  float acc = 0.0f;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    float t = __fmul_rn(s1, R[i]);
    if (U::ui(i) >= 0) t = __fmaf_rn(s1, R[i], __fmul_rn(G.t2, R[U::ui(i) < 0 ? 0 : U::ui(i)]));
    acc = __fmaf_rn(w[1 + i], t, acc);
  }
  if constexpr (!STD) {
    const float s2 = -__fmul_rn(G.g[4], qs), s3 = -__fmul_rn(G.g[5], qs);
    acc = q_c2<A, B, 0>(R, G, s1, s2, w, acc); acc = q_c2<A, B, 1>(R, G, s1, s2, w, acc);
    acc = q_c2<A, B, 2>(R, G, s1, s2, w, acc); acc = q_c2<A, B, 3>(R, G, s1, s2, w, acc);
    acc = q_c2<A, B, 4>(R, G, s1, s2, w, acc); acc = q_c2<A, B, 5>(R, G, s1, s2, w, acc);
    acc = q_c3<A, B, 0>(R, G, s2, s3, w, acc); acc = q_c3<A, B, 1>(R, G, s2, s3, w, acc);
    acc = q_c3<A, B, 2>(R, G, s2, s3, w, acc); acc = q_c3<A, B, 3>(R, G, s2, s3, w, acc);
    acc = q_c3<A, B, 4>(R, G, s2, s3, w, acc); acc = q_c3<A, B, 5>(R, G, s2, s3, w, acc);
    acc = q_c3<A, B, 6>(R, G, s2, s3, w, acc); acc = q_c3<A, B, 7>(R, G, s2, s3, w, acc);
    acc = q_c3<A, B, 8>(R, G, s2, s3, w, acc); acc = q_c3<A, B, 9>(R, G, s2, s3, w, acc);
  }
  return acc;
}

// Mixed mode: coefficients in float32 (as in the forward), r formed in
// float64, sums in float64.
template <bool STD>
__global__ void __launch_bounds__(kM2LWarps * 32) k_vjp_m2l32(VjpArgs V) {
  __shared__ CellBuf s_buf[kM2LWarps];
  const int k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (k >= V.nleaves) return;
  CellBuf& B = s_buf[threadIdx.x >> 5];
  const int a = V.leaf_cells[k];
  const float mine = lane < 20 ? (float)V.cbar[20 * (int64_t)k + lane] : 0.0f;
  float cb[20];
#pragma unroll
  for (int j = 0; j < 20; ++j) cb[j] = __shfl_sync(0xffffffffu, mine, j);
  const double ax = V.c.cx[a], ay = V.c.cy[a], az = V.c.cz[a];
  double rx = 0.0, ry = 0.0, rz = 0.0;
  const int64_t off = V.far_off[k];
  const int nf = (int)min((int64_t)V.far_cnt[k], V.cap_far);
  for (int e0 = 0; e0 < nf; e0 += 32) {
    const int n = min(32, nf - e0);
    if (lane < n) {
      const int b = V.far_idx[off + e0 + lane];
      const double* s64 = V.c.src64 + 10 * (int64_t)b;
      const float r[3] = {(float)(ax - s64[0]), (float)(ay - s64[1]), (float)(az - s64[2])};
      const float4 q0 = V.c.src32[4 * (int64_t)b + 2], q1 = V.c.src32[4 * (int64_t)b + 3];
      const float Qb[6] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y};
      // r-derivatives of sum_j cb_j C_j by dual numbers; M and Q enter linearly
      const Dual R[3] = {Dual{r[0], {1.f, 0.f, 0.f}}, Dual{r[1], {0.f, 1.f, 0.f}}, Dual{r[2], {0.f, 0.f, 1.f}}};
      const Dual cr = m2l_contract<STD>(R, V.c.src32[4 * (int64_t)b].w, Qb, cb);
      double* v = B.v + 11 * lane;
      B.cell[lane] = b;
#pragma unroll
      for (int i = 0; i < 3; ++i) v[1 + i] = -(double)cr.d[i];
      rx -= v[1]; ry -= v[2]; rz -= v[3];
      const GTerms G = g_terms(r);
      v[0] = (double)mass_cotangent(r, G, cb);
      v[4] = (double)q_cotangent<0, 0, STD>(r, G, cb);
      v[5] = (double)q_cotangent<0, 1, STD>(r, G, cb);
      v[6] = (double)q_cotangent<0, 2, STD>(r, G, cb);
      v[7] = (double)q_cotangent<1, 1, STD>(r, G, cb);
      v[8] = (double)q_cotangent<1, 2, STD>(r, G, cb);
      v[9] = (double)q_cotangent<2, 2, STD>(r, G, cb);
    }
    cell_buf_add(V, B, lane, n);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    rx += __shfl_xor_sync(0xffffffffu, rx, o);
    ry += __shfl_xor_sync(0xffffffffu, ry, o);
    rz += __shfl_xor_sync(0xffffffffu, rz, o);
  }
  if (lane < 3)
    atomicAdd(&V.cell_bar[10 * (int64_t)a + 1 + lane], lane == 0 ? rx : (lane == 1 ? ry : rz));
}

// FP64 mode.  With W1, W2, W3 the leaf's cotangents as symmetric tensors, their
// traces removed (1/R is harmonic), A(R) = W1.D1 + W2:D2 + W3:D3 of 1/R is
//   A = g1 l1 + g2 l2 + g3 l3,  l1 = W1.R, l2 = R.W2.R, l3 = W3 R R R,
// harmonic and homogeneous in each l_n, and the sum of the coefficients is
// -M A - Q:(grad grad A) / 6.  So M_bar = -A, Q_bar = -(grad grad A) / 6 (an
// isotropic part, which a traceless Q does not see, left out) and r_bar =
// -M grad A - grad(Q:grad grad A) / 6, with grad g_n = g_(n+1) R, v = W2 R,
// Y = W3 R, z = Y R, u = Q R: some 200 float64 operations a pair where the
// dual numbers and the seven contractions took 3000.
struct LeafW {
  double w1[3], w2[6], w3[10];          // compact: xx xy xz yy yz zz; xxx xxy xxz xyy xyz xzz yyy yyz yzz zzz
};
template <bool STD>
__global__ void __launch_bounds__(kM2LWarps * 32) k_vjp_m2l64(VjpArgs V) {
  __shared__ CellBuf s_buf[kM2LWarps];
  const int k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (k >= V.nleaves) return;
  CellBuf& B = s_buf[threadIdx.x >> 5];
  const int a = V.leaf_cells[k];
  LeafW W;
  {
    const double* cb = V.cbar + 20 * (int64_t)k;
#pragma unroll
    for (int i = 0; i < 3; ++i) W.w1[i] = cb[1 + i];
    const double tr = (cb[4] + cb[7] + cb[9]) * (1.0 / 3.0);
    W.w2[0] = cb[4] - tr; W.w2[3] = cb[7] - tr; W.w2[5] = cb[9] - tr;
    W.w2[1] = 0.5 * cb[5]; W.w2[2] = 0.5 * cb[6]; W.w2[4] = 0.5 * cb[8];
    const double third = 1.0 / 3.0;
    double x[10] = {cb[10], cb[11] * third, cb[12] * third, cb[13] * third, cb[14] * (1.0 / 6.0),
                    cb[15] * third, cb[16], cb[17] * third, cb[18] * third, cb[19]};
    const double t0 = 0.2 * (x[0] + x[3] + x[5]), t1 = 0.2 * (x[1] + x[6] + x[8]),
                 t2 = 0.2 * (x[2] + x[7] + x[9]);
    W.w3[0] = x[0] - 3.0 * t0; W.w3[1] = x[1] - t1; W.w3[2] = x[2] - t2; W.w3[3] = x[3] - t0;
    W.w3[4] = x[4]; W.w3[5] = x[5] - t0; W.w3[6] = x[6] - 3.0 * t1; W.w3[7] = x[7] - t2;
    W.w3[8] = x[8] - t1; W.w3[9] = x[9] - 3.0 * t2;
  }
  const double ax = V.c.cx[a], ay = V.c.cy[a], az = V.c.cz[a];
  double rx = 0.0, ry = 0.0, rz = 0.0;
  const int64_t off = V.far_off[k];
  const int nf = (int)min((int64_t)V.far_cnt[k], V.cap_far);
  constexpr int s3[3][6] = {{0, 1, 2, 3, 4, 5}, {1, 3, 4, 6, 7, 8}, {2, 4, 5, 7, 8, 9}};   // W3 slice of an axis
  for (int e0 = 0; e0 < nf; e0 += 32) {
    const int n = min(32, nf - e0);
    if (lane < n) {
      const int b = V.far_idx[off + e0 + lane];
      const double* s = V.c.src64 + 10 * (int64_t)b;
      const double R[3] = {ax - s[0], ay - s[1], az - s[2]};
      const double M = s[3];
      const double Q[6] = {s[4], s[5], s[6], s[7], s[8], s[9]};
      const double g0 = rsqrt64(R[0] * R[0] + R[1] * R[1] + R[2] * R[2]);
      const double i2 = g0 * g0, g1 = -g0 * i2, g2 = -3.0 * g1 * i2, g3 = -5.0 * g2 * i2,
                   g4 = -7.0 * g3 * i2, g5 = -9.0 * g4 * i2, g6 = -11.0 * g5 * i2;
      auto mul = [](const double S[6], const double x[3], double out[3]) {
        out[0] = S[0] * x[0] + S[1] * x[1] + S[2] * x[2];
        out[1] = S[1] * x[0] + S[3] * x[1] + S[4] * x[2];
        out[2] = S[2] * x[0] + S[4] * x[1] + S[5] * x[2];
      };
      auto dot = [](const double x[3], const double y[3]) { return x[0] * y[0] + x[1] * y[1] + x[2] * y[2]; };
      auto con = [](const double S[6], const double T[6]) {
        return S[0] * T[0] + S[3] * T[3] + S[5] * T[5] + 2.0 * (S[1] * T[1] + S[2] * T[2] + S[4] * T[4]);
      };
      double v[3], Y[6], z[3], u[3];
      mul(W.w2, R, v);
#pragma unroll
      for (int q = 0; q < 6; ++q)
        Y[q] = W.w3[s3[0][q]] * R[0] + W.w3[s3[1][q]] * R[1] + W.w3[s3[2][q]] * R[2];
      mul(Y, R, z);
      mul(Q, R, u);
      const double l1 = dot(W.w1, R), l2 = dot(v, R), l3 = dot(z, R), q = dot(u, R);
      const double S2 = g2 * l1 + g3 * l2 + g4 * l3;
      // the quadrupole sees all orders, or the first alone (standard series)
      double P[3], P4[3], H[6], K[6], dA[3];
      const double S4 = STD ? g3 * l1 : g3 * l1 + g4 * l2 + g5 * l3;
      const double S5 = STD ? g4 * l1 : g4 * l1 + g5 * l2 + g6 * l3;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        dA[i] = S2 * R[i] + g1 * W.w1[i] + 2.0 * (g2 * v[i]) + 3.0 * (g3 * z[i]);
        P[i] = STD ? g2 * W.w1[i] : g2 * W.w1[i] + 2.0 * (g3 * v[i]) + 3.0 * (g4 * z[i]);
        P4[i] = STD ? g3 * W.w1[i] : g3 * W.w1[i] + 2.0 * (g4 * v[i]) + 3.0 * (g5 * z[i]);
      }
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        H[c] = STD ? 0.0 : 2.0 * (g2 * W.w2[c]) + 6.0 * (g3 * Y[c]);
        K[c] = STD ? 0.0 : 2.0 * (g3 * W.w2[c]) + 6.0 * (g4 * Y[c]);
      }
      double QP[3], Ku[3], WQ[3] = {0.0, 0.0, 0.0};
      mul(Q, P, QP);
      mul(K, u, Ku);
      if (!STD) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          const double T[6] = {W.w3[s3[i][0]], W.w3[s3[i][1]], W.w3[s3[i][2]],
                               W.w3[s3[i][3]], W.w3[s3[i][4]], W.w3[s3[i][5]]};
          WQ[i] = 6.0 * g3 * con(Q, T);
        }
      }
      const double cR = q * S5 + 2.0 * dot(u, P4) + con(Q, K);
      double* out = B.v + 11 * lane;
      B.cell[lane] = b;
      out[0] = -(g1 * l1 + g2 * l2 + g3 * l3);
      double gr[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const double t = cR * R[i] + 2.0 * (S4 * u[i] + QP[i] + Ku[i]) + q * P4[i] + WQ[i];
        gr[i] = -(M * dA[i]) - t * (1.0 / 6.0);
        out[1 + i] = -gr[i];
      }
      rx += gr[0]; ry += gr[1]; rz += gr[2];
      const double sx = S4 * R[0], sy = S4 * R[1], sz = S4 * R[2];
      out[4] = (sx * R[0] + 2.0 * (R[0] * P[0]) + H[0]) * (-1.0 / 6.0);
      out[5] = (sx * R[1] + (R[0] * P[1] + R[1] * P[0]) + H[1]) * (-1.0 / 3.0);
      out[6] = (sx * R[2] + (R[0] * P[2] + R[2] * P[0]) + H[2]) * (-1.0 / 3.0);
      out[7] = (sy * R[1] + 2.0 * (R[1] * P[1]) + H[3]) * (-1.0 / 6.0);
      out[8] = (sy * R[2] + (R[1] * P[2] + R[2] * P[1]) + H[4]) * (-1.0 / 3.0);
      out[9] = (sz * R[2] + 2.0 * (R[2] * P[2]) + H[5]) * (-1.0 / 6.0);
    }
    cell_buf_add(V, B, lane, n);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    rx += __shfl_xor_sync(0xffffffffu, rx, o);
    ry += __shfl_xor_sync(0xffffffffu, ry, o);
    rz += __shfl_xor_sync(0xffffffffu, rz, o);
  }
  if (lane < 3)
    atomicAdd(&V.cell_bar[10 * (int64_t)a + 1 + lane], lane == 0 ? rx : (lane == 1 ? ry : rz));
}

// ---------------------------------------------------------------------------
// Transposed near lists.  The leaf-only walk is one-sided (b near a does not
// imply a near b), so the target leaves of a source leaf are collected from
// the near lists: counts, room reserved per leaf, fill.  A source then sums
// its own cotangents in registers; with the pairs walked by target alone they
// took four float64 atomics per (target leaf, source) and butterflies over
// the leaf's targets per pair (47 ms of the 2^20 Plummer sphere's adjoint).
// ---------------------------------------------------------------------------
// Extra items of the near lists (any order: a leaf's are contiguous).
__global__ void k_near_plan(VjpArgs V) {
  KD_GRID_STRIDE(k, V.nleaves) {
    const int x = extra_segments(min((int64_t)V.near_cnt[k], V.cap_near), V.entries);
    const int64_t first = x > 0 ? (int64_t)atomicAdd(&V.tctr[2], (unsigned long long)x) : 0;
    V.seg_first[k] = (int32_t)first;
    for (int q = 0; q < x; ++q)
      if (first + q < V.seg_cap) V.seg_leaf[first + q] = k;
  }
}

// The entries of a target item.
__device__ __forceinline__ int near_items(const VjpArgs& V) {
  return V.nleaves + (int)min((int64_t)V.tctr[2], V.seg_cap);
}
__device__ __forceinline__ int near_item(const VjpArgs& V, int item, int* k, int64_t* e0) {
  const bool seg = item >= V.nleaves;
  const int g = item - V.nleaves;
  *k = seg ? V.seg_leaf[g] : item;
  const int64_t piece = seg ? (int64_t)(g - V.seg_first[*k] + 1) : 0;
  *e0 = V.near_off[*k] + piece * V.entries;
  return (int)(min(min((int64_t)V.near_cnt[*k], V.cap_near), (piece + 1) * V.entries) - piece * V.entries);
}

__global__ void k_tr_count(VjpArgs V) {
  const int lane = threadIdx.x & 31;
  const int nitems = near_items(V);
  for (int item = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); item < nitems;
       item += (int)((gridDim.x * blockDim.x) >> 5)) {
    int k;
    int64_t e0 = 0;
    const int nn = near_item(V, item, &k, &e0);
    for (int e = lane; e < nn; e += 32) atomicAdd(&V.tcnt[V.leaf_rank[V.near_idx[e0 + e]]], 1);
  }
}

// Room for each leaf's entries and extra items (any order), reserved once per warp.
__global__ void k_tr_plan(VjpArgs V) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r - lane >= V.nleaves) return;
  const int cnt = r < V.nleaves ? V.tcnt[r] : 0;
  const int extra = extra_segments(cnt, V.entries);
  long long ic = cnt;
  int ie = extra;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long uc = __shfl_up_sync(full, ic, o);
    const int ue = __shfl_up_sync(full, ie, o);
    if (lane >= o) { ic += uc; ie += ue; }
  }
  unsigned long long bc = 0, be = 0;
  if (lane == 31) {
    bc = atomicAdd(&V.tctr[0], (unsigned long long)ic);
    be = ie ? atomicAdd(&V.tctr[1], (unsigned long long)ie) : 0;
  }
  bc = __shfl_sync(full, bc, 31);
  be = __shfl_sync(full, be, 31);
  if (r >= V.nleaves) return;
  V.toff[r] = (int64_t)bc + ic - cnt;
  const int64_t first = (int64_t)be + ie - extra;
  V.tseg_first[r] = (int32_t)first;
  for (int q = 0; q < extra; ++q)
    if (first + q < V.tseg_cap) V.tseg_leaf[first + q] = r;
}

__global__ void k_tr_fill(VjpArgs V) {
  const int lane = threadIdx.x & 31;
  const int nitems = near_items(V);
  for (int item = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); item < nitems;
       item += (int)((gridDim.x * blockDim.x) >> 5)) {
    int k;
    int64_t e0 = 0;
    const int nn = near_item(V, item, &k, &e0);
    for (int e = lane; e < nn; e += 32) {
      const int r = V.leaf_rank[V.near_idx[e0 + e]];
      const int64_t at = V.toff[r] + atomicAdd(&V.tcur[r], 1);
      if (at < V.tcap) V.tidx[at] = k;
    }
  }
}

// ---------------------------------------------------------------------------
// P2P reverse.  Pair kernel K (a_i += m_j K(d), d = x_i - x_j), K = -f(r) d,
// J = dK/dd = -f I - g d d^T, g = f'(r) / r.  Plummer: f = (r^2 + eps^2)^(-3/2),
// g = -3 (r^2 + eps^2)^(-5/2).  M4 (Eq. 13, symmetrised): the mean of the two
// sides' terms; one side, q = r/h:
//   q < 1:       f = (4/3 - 6/5 q^2 + q^3/2) / h^3,   g = (-12/5 + 3/2 q) / h^5
//   1 <= q < 2:  f = F(q) / (q^3 h^3),  g = (F'(q) q - 3 F(q)) / (q^5 h^5), F' = 4 pi w q^2
//   q >= 2:      f = 1 / r^3,           g = -3 / r^5
// (the q < 1 forms are the polynomials themselves, finite at r = 0, where g
// multiplies d = 0).  F: M4 mass fraction for 1 <= q < 2; 4 pi w(q) = t^3
// there, t = 2 - q.
// Target side:  x_bar_i += sum_j m_j J(d) a_bar_i;
// source side:  x_bar_j -= m_j sum_i J(d) a_bar_i,  m_bar_j += sum_i K(d).a_bar_i.
// ---------------------------------------------------------------------------
// The rounding order of a pair's terms is fixed, so that both sides of a pair
// (and any version of these kernels) form the same float32 values.
__device__ __forceinline__ float dot_rn(float a0, float b0, float a1, float b1, float a2, float b2) {
  return __fmaf_rn(a2, b2, __fmaf_rn(a0, b0, __fmul_rn(a1, b1)));
}
// Differences of a pair that its system's grids are too coarse for: float64,
// rounded to float32.
__device__ __forceinline__ void exact_diff(const VjpArgs& V, int i, int j, float& d0, float& d1,
                                           float& d2) {
  d0 = (float)(V.tp.x[i] - V.tp.x[j]);
  d1 = (float)(V.tp.y[i] - V.tp.y[j]);
  d2 = (float)(V.tp.z[i] - V.tp.z[j]);
}
// One component of J b = -f b - g d (d.b).
__device__ __forceinline__ float jb_term(float f, float b, float g, float d, float db) {
  return __fmaf_rn(-f, b, -__fmul_rn(__fmul_rn(g, d), db));
}

__device__ __forceinline__ float m4_F_outer(float q) {
  const float t = 2.0f - q;
  return 1.0f - t * t * t * t * (1.0f - 0.8f * t + t * t / 6.0f);
}

template <int SOFT>
__device__ __forceinline__ void pair_fg32(float r2, float eps2, float hinv_i, float hinv_j, float& f,
                                          float& g) {
  if (SOFT == KDFMM_SOFT_PLUMMER) {
    const float inv = rsq(__fadd_rn(r2, eps2));
    const float inv3 = __fmul_rn(__fmul_rn(inv, inv), inv);
    f = inv3;
    g = -3.0f * inv3 * inv * inv;
    return;
  }
  const float r = sqrtf(r2);
  float fs = 0.0f, gs = 0.0f;
  const float hs[2] = {hinv_i, hinv_j};
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    const float hinv = hs[side];
    const float q = r * hinv;
    const float h3inv = hinv * hinv * hinv;
    if (q >= 2.0f) {
      const float rinv = 1.0f / r;
      const float r3inv = rinv * rinv * rinv;
      fs += r3inv;
      gs += -3.0f * r3inv * rinv * rinv;
    } else if (q < 1.0f) {
      fs += (4.0f / 3.0f + q * q * (-1.2f + 0.5f * q)) * h3inv;
      gs += (-2.4f + 1.5f * q) * h3inv * hinv * hinv;
    } else {
      const float q2 = q * q, F = m4_F_outer(q);
      const float t = 2.0f - q;
      fs += F / (q2 * q) * h3inv;
      gs += (t * t * t * q2 * q - 3.0f * F) / (q2 * q2 * q) * h3inv * hinv * hinv;
    }
  }
  f = 0.5f * fs;
  g = 0.5f * gs;
}

// A chunk of list entries in shared memory: up to 32 leaves whose particles fit
// in kVjpStage records.
constexpr int kVjpStage = 128;
struct LeafChunk {
  float4 p0[kVjpStage], p1[kVjpStage], p2[kVjpStage];
  int beg[33];                          // staged start of each leaf
  int first[32];
};
// Stages the records of the leading leaves of the entries' cells (cell: this
// lane's, or -1) that fit; returns their number.  The loads of a batch of rounds
// are issued before any is used (L2 gathers: latency-bound).
template <class Chunk, class Put>
__device__ __forceinline__ int stage_chunk(const VjpArgs& V, Chunk& B, int lane, int cell, Put put) {
  const unsigned full = 0xffffffffu;
  int cnt = 0;
  __syncwarp();
  if (cell >= 0) {
    cnt = V.c.count[cell];
    B.first[lane] = V.c.first[cell];
  }
  int incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int w = __shfl_up_sync(full, incl, o);
    if (lane >= o) incl += w;
  }
  B.beg[lane] = incl - cnt;
  const int L = __popc(__ballot_sync(full, cell >= 0 && incl <= kVjpStage));
  if (lane == L - 1) B.beg[L] = incl;
  __syncwarp();
  const int total = B.beg[L];
#pragma unroll 2
  for (int i = lane; i < total; i += 32) {
    int l = 0;
#pragma unroll
    for (int step = 16; step > 0; step >>= 1)
      if (l + step < L && B.beg[l + step] <= i) l += step;
    put(i, B.first[l] + i - B.beg[l]);
  }
  __syncwarp();
  return L;
}

constexpr int kVjpWarps = 4;

// A sum of float32 terms in three float32 numbers: what the first two lose is
// carried exactly (two-sums), so n terms of magnitude v are off by some
// n^2 2^-73 v, where a float64 sum loses up to n^2 2^-54 v.
struct Sum72 {
  float h, m, l;
  __device__ __forceinline__ void add(float v) {
    float e, e2;
    two_sum(h, v, h, e);
    two_sum(m, e, m, e2);
    l = __fadd_rn(l, e2);
  }
  __device__ __forceinline__ double value() const { return (double)h + ((double)m + (double)l); }
  // false once a term or the sum has left float32
  __device__ __forceinline__ bool holds() const { return fabsf(h) < __int_as_float(0x7f800000); }
};
struct Sum64 {
  double s;
  __device__ __forceinline__ void add(float v) { s += float_to_double(v); }
  __device__ __forceinline__ double value() const { return s; }
  __device__ __forceinline__ bool holds() const { return true; }
};

// Mixed mode, target side: warp per target leaf (or segment of a long near
// list), lanes = (target, slice) as in the forward; a leaf's sources are read
// by broadcast (a warp instruction touches the slices' few records).  Terms in
// float32, the same operations as the source side's; each is added to a sum of
// three float32 numbers, in the place of a float64 sum (three float64 additions a
// pair would keep the 1/64-rate pipe busy for longer than the rest of the pair)
// and with less rounding than it.  2^20 Plummer sphere, 1.17e9 pairs: 5.2 ms
// here and 5.4 ms on the source side (4.3 and 5.1 with two float32 numbers a sum;
// one of the three sums in float64: 0.5 ms more), against 47.3 ms for the two
// together when one kernel walked the pairs by target.
// EXACT: the items of close_t, with float64 differences and sums.
template <int SOFT, bool EXACT>
__device__ __forceinline__ void target32_items(const VjpArgs& V, LeafChunk& B) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int nwork = EXACT ? (int)V.tctr[3] : near_items(V);
  for (int at0 = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); at0 < nwork;
       at0 += (int)((gridDim.x * blockDim.x) >> 5)) {
    const int item = EXACT ? V.close_t[at0] : at0;
    const bool seg = item >= V.nleaves;
    const int gi = item - V.nleaves;
    int k;
    int64_t e0 = 0;
    const int nn = near_item(V, item, &k, &e0);
    const int a = V.leaf_cells[k];
    const int fa = V.c.first[a], nt = V.c.count[a];
    const int K = 32 / nt, t = lane % nt, sl = lane / nt;
    const bool act = sl < K;
    const int pi = fa + t;
    const float4 o0 = V.q0[pi], o1 = V.q1[pi], o2 = V.q2[pi];
    const float2 o3 = V.q3[pi];
    const float3 b = make_float3(o2.w, o3.x, o3.y);
    const double eps = V.sys_eps[V.leaf_sys[k]];
    float eps2 = (float)(eps * eps);
    asm("" : "+f"(eps2));
    float lowest = __int_as_float(0x7f800000);
    typename std::conditional<EXACT, Sum64, Sum72>::type sx{}, sy{}, sz{};
    for (int eb = 0; eb < nn;) {
      const int L = stage_chunk(V, B, lane, eb + lane < nn ? V.near_idx[e0 + eb + lane] : -1,
                                [&](int at, int pj) {
                                  B.p0[at] = V.q0[pj];
                                  B.p1[at] = V.q1[pj];
                                  float4 s = V.q2[pj];
                                  s.w = __int_as_float(pj);
                                  B.p2[at] = s;
                                });
      const int total = B.beg[L];
      if (act) {
#pragma unroll 2
        for (int j = sl; j < total; j += K) {
          const float4 s0 = B.p0[j], s1 = B.p1[j], s2 = B.p2[j];
          if (__float_as_int(s2.w) == pi) continue;
          float d0, d1, d2;
          if constexpr (EXACT) {
            exact_diff(V, pi, __float_as_int(s2.w), d0, d1, d2);
          } else {
            d0 = grid_diff(o0.x, o1.x, o2.x, s0.x, s1.x, s2.x);
            d1 = grid_diff(o0.y, o1.y, o2.y, s0.y, s1.y, s2.y);
            d2 = grid_diff(o0.z, o1.z, o2.z, s0.z, s1.z, s2.z);
          }
          const float r2 = dot_rn(d0, d0, d1, d1, d2, d2);
          if constexpr (!EXACT) lowest = fminf(lowest, r2);
          float f, g;
          pair_fg32<SOFT>(r2, eps2, o1.w, s1.w, f, g);
          const float db = dot_rn(d0, b.x, d1, b.y, d2, b.z);
          // J b = -f b - (f'/r) d (d.b)
          const float jx = jb_term(f, b.x, g, d0, db);
          const float jy = jb_term(f, b.y, g, d1, db);
          const float jz = jb_term(f, b.z, g, d2, db);
          sx.add(__fmul_rn(s0.w, jx));
          sy.add(__fmul_rn(s0.w, jy));
          sz.add(__fmul_rn(s0.w, jz));
        }
      }
      eb += L;
    }
    if (!EXACT && __any_sync(full, close_pairs(lowest, system_bound(V, k)) || !sx.holds() ||
                                       !sy.holds() || !sz.holds())) {
      if (lane == 0) V.close_t[atomicAdd(&V.tctr[3], 1ull)] = item;
      continue;
    }
    double gx = sx.value(), gy = sy.value(), gz = sz.value();
    for (int s = 1; s < K; ++s) {
      const int src = t + s * nt;
      const double ox = __shfl_sync(full, gx, src), oy = __shfl_sync(full, gy, src),
                   oz = __shfl_sync(full, gz, src);
      if (sl == 0) { gx += ox; gy += oy; gz += oz; }
    }
    if (act && sl == 0) {
      if (seg) {
        double* P = V.seg_part + (int64_t)gi * 128 + 4 * t;
        P[0] = gx; P[1] = gy; P[2] = gz;
      } else {
        V.xbar[3 * (int64_t)pi] += gx;
        V.xbar[3 * (int64_t)pi + 1] += gy;
        V.xbar[3 * (int64_t)pi + 2] += gz;
      }
    }
  }
}

// Mixed mode, source side: warp per source leaf (or piece of a long
// transposed list), lanes = (source, slice), a slice taking every K-th target
// leaf.  A leaf's terms are summed over its targets in float32 as a perfect
// binary tree (four at a time, then a carry stack), then added in float64; one
// float64 atomic per source and item at the end.
// EXACT: the items of close_s, with float64 differences.
template <int SOFT, bool EXACT>
__device__ __forceinline__ void source32_items(const VjpArgs& V, LeafChunk& B, float2* sb) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int nwork = EXACT ? (int)V.tctr[4] : V.nleaves + (int)min((int64_t)V.tctr[1], V.tseg_cap);
  for (int at0 = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); at0 < nwork;
       at0 += (int)((gridDim.x * blockDim.x) >> 5)) {
    const int item = EXACT ? V.close_s[at0] : at0;
    const bool seg = item >= V.nleaves;
    const int r = seg ? V.tseg_leaf[item - V.nleaves] : item;
    const int piece = seg ? item - V.nleaves - V.tseg_first[r] + 1 : 0;
    const int a = V.leaf_cells[r];
    const int fa = V.c.first[a], ns = V.c.count[a];
    const int K = 32 / ns, j = lane % ns, sl = lane / ns;
    const bool act = sl < K;
    const int pj = fa + j;
    const float4 o0 = V.q0[pj], o1 = V.q1[pj], o2 = V.q2[pj];
    const float mj = o0.w;
    const double eps = V.sys_eps[V.leaf_sys[r]];
    float eps2 = (float)(eps * eps);
    asm("" : "+f"(eps2));
    float lowest = __int_as_float(0x7f800000);
    double g[4] = {0.0, 0.0, 0.0, 0.0};
    const int64_t e0 = V.toff[r] + (int64_t)piece * V.entries;
    const int nn = min(V.tcnt[r] - piece * V.entries, V.entries);
    for (int eb = 0; eb < nn;) {
      const int L = stage_chunk(V, B, lane, eb + lane < nn ? V.leaf_cells[V.tidx[e0 + eb + lane]] : -1,
                                [&](int at, int pi) {
                                  float4 s = V.q0[pi];
                                  const float2 b = V.q3[pi];
                                  s.w = __int_as_float(pi);
                                  B.p0[at] = s;
                                  B.p1[at] = V.q1[pi];
                                  B.p2[at] = V.q2[pi];
                                  sb[at] = b;
                                });
      for (int q = sl; act && q < L; q += K) {
        const int fb = B.beg[q], nb = B.beg[q + 1] - fb;
        float h1[4], h2[4], h3[4], acc[4];
        for (int i0 = 0; i0 < nb; i0 += 4) {
          float s[4][4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int at = fb + i0 + u;
            s[u][0] = s[u][1] = s[u][2] = s[u][3] = 0.0f;
            if (i0 + u < nb && __float_as_int(B.p0[at].w) != pj) {
              const float4 t0 = B.p0[at], t1 = B.p1[at], t2 = B.p2[at];
              const float2 t3 = sb[at];
              const float3 b = make_float3(t2.w, t3.x, t3.y);
              float d0, d1, d2;
              if constexpr (EXACT) {
                exact_diff(V, __float_as_int(t0.w), pj, d0, d1, d2);
              } else {
                d0 = grid_diff(t0.x, t1.x, t2.x, o0.x, o1.x, o2.x);
                d1 = grid_diff(t0.y, t1.y, t2.y, o0.y, o1.y, o2.y);
                d2 = grid_diff(t0.z, t1.z, t2.z, o0.z, o1.z, o2.z);
              }
              const float r2 = dot_rn(d0, d0, d1, d1, d2, d2);
              if constexpr (!EXACT) lowest = fminf(lowest, r2);
              float f, g;
              pair_fg32<SOFT>(r2, eps2, t1.w, o1.w, f, g);
              const float db = dot_rn(d0, b.x, d1, b.y, d2, b.z);
              const float jx = jb_term(f, b.x, g, d0, db);
              const float jy = jb_term(f, b.y, g, d1, db);
              const float jz = jb_term(f, b.z, g, d2, db);
              s[u][0] = __fmul_rn(-mj, jx);
              s[u][1] = __fmul_rn(-mj, jy);
              s[u][2] = __fmul_rn(-mj, jz);
              s[u][3] = __fmul_rn(-f, db);    // K(d) . a_bar_i
            }
          }
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            float v = __fadd_rn(__fadd_rn(s[0][c], s[1][c]), __fadd_rn(s[2][c], s[3][c]));
            const int blk = i0 >> 2;
            const bool last = i0 + 4 >= nb;
            // the tree over the blocks of four: odd blocks join the one held
            // below; what is held is joined at the end
            if (blk & 1) {
              v = __fadd_rn(h1[c], v);
              if (blk & 2) {
                v = __fadd_rn(h2[c], v);
                if (blk & 4) v = __fadd_rn(h3[c], v); else h3[c] = v;
              } else {
                h2[c] = v;
              }
            } else {
              h1[c] = v;
            }
            if (last) {
              if (!(blk & 1)) {
                if (blk & 2) v = __fadd_rn(h2[c], v);
                if (blk & 4) v = __fadd_rn(h3[c], v);
              } else if (!(blk & 2)) {
                if (blk & 4) v = __fadd_rn(h3[c], v);
              }
              acc[c] = v;
            }
          }
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) g[c] += float_to_double(acc[c]);
      }
      eb += L;
    }
    if (!EXACT && __any_sync(full, close_pairs(lowest, system_bound(V, r)))) {
      if (lane == 0) V.close_s[atomicAdd(&V.tctr[4], 1ull)] = item;
      continue;
    }
    for (int s = 1; s < K; ++s) {
      const int src = j + s * ns;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const double o = __shfl_sync(full, g[c], src);
        if (sl == 0) g[c] += o;
      }
    }
    if (act && sl == 0) {
      atomicAdd(&V.xsrc[3 * (int64_t)pj], g[0]);
      atomicAdd(&V.xsrc[3 * (int64_t)pj + 1], g[1]);
      atomicAdd(&V.xsrc[3 * (int64_t)pj + 2], g[2]);
      atomicAdd(&V.msrc[pj], g[3]);
    }
  }
}

template <int SOFT>
__global__ void __launch_bounds__(kVjpWarps * 32, SOFT == KDFMM_SOFT_M4 ? 7 : 8) k_vjp_target32(VjpArgs V) {
  __shared__ LeafChunk s_chunk[kVjpWarps];
  target32_items<SOFT, false>(V, s_chunk[threadIdx.x >> 5]);
}
template <int SOFT>
__global__ void __launch_bounds__(kVjpWarps * 32, SOFT == KDFMM_SOFT_M4 ? 5 : 6) k_vjp_source32(VjpArgs V) {
  __shared__ LeafChunk s_chunk[kVjpWarps];
  __shared__ float2 s_b[kVjpWarps][kVjpStage];
  source32_items<SOFT, false>(V, s_chunk[threadIdx.x >> 5], s_b[threadIdx.x >> 5]);
}
// The items that both left (none, as a rule).
template <int SOFT>
__global__ void __launch_bounds__(kVjpWarps * 32) k_vjp_close32(VjpArgs V) {
  __shared__ LeafChunk s_chunk[kVjpWarps];
  __shared__ float2 s_b[kVjpWarps][kVjpStage];
  target32_items<SOFT, true>(V, s_chunk[threadIdx.x >> 5]);
  __syncwarp();
  source32_items<SOFT, true>(V, s_chunk[threadIdx.x >> 5], s_b[threadIdx.x >> 5]);
}

// One side of the symmetrised M4 pair in float64, added to f and g: the branches
// of q < 1 (v = q) and q >= 1 (v = 2 - q, 0 outside the support) as one
// evaluation with selected constants.
__device__ __forceinline__ void m4_fg64(double r, double inv3, double inv5, double hinv, double& f,
                                        double& g) {
  const double q = r * hinv, h2inv = hinv * hinv, h3inv = h2inv * hinv;
  const bool in = __double2hiint(q) < 0x3ff00000;            // q < 1 (q >= 0)
  const double t = 2.0 - q;
  const bool outside = __double2hiint(t) < 0;                // its q^3 may overflow
  const double v = in ? q : (outside ? 0.0 : t), v2 = v * v, qs = outside ? 0.0 : q;
  const double p1 = fma(v, fma(v, in ? 0.0 : -1.0 / 6.0, in ? 0.5 : 0.8), in ? -1.2 : -1.0);
  const double F = fma(in ? v2 : v2 * v2, p1, in ? 4.0 / 3.0 : 1.0);
  const double G = in ? fma(1.5, q, -2.4) : fma(-3.0, F, v2 * v * (qs * qs * qs));
  f = fma(F, in ? h3inv : inv3, f);
  g = fma(G, in ? h3inv * h2inv : inv5, g);
}
__device__ __forceinline__ void m4_pair_fg64(double r2, double hinv_i, double hinv_j, double& f, double& g) {
  const double inv = rsqrt64(r2), inv2 = inv * inv, inv3 = inv2 * inv, inv5 = inv3 * inv2, r = far_sqrt(r2, inv);
  f = g = 0.0;
  m4_fg64(r, inv3, inv5, hinv_i, f, g);
  m4_fg64(r, inv3, inv5, hinv_j, f, g);
  f *= 0.5;
  g *= 0.5;
}

// A chunk of list entries in float64: positions, w (the target side: m in w0;
// the source side: a_bar), 1/h, (2h)^2, particle; the pairs inside a support
// queued for the warp as in the evaluation's P2P.
struct Chunk64 {
  double x[kVjpStage], y[kVjpStage], z[kVjpStage], w0[kVjpStage], w1[kVjpStage], w2[kVjpStage],
      hinv[kVjpStage];
  float h2[kVjpStage];
  int id[kVjpStage];
  int beg[33], first[32];
  double term[4][32];
  unsigned own[32];
  uint16_t queue[512];
};

// FP64 mode, one kernel for both sides (SOURCE: the source side), warp per own
// leaf and piece, lanes = (own particle, slice).  With d = x_i - x_j (i the
// target), f and g of the pair: the target side sums m_j f and m_j g (d.b_i) d,
// the source side f b_i + g (d.b_i) d and -f d.b_i.  Pairs outside both supports
// first (f = r^-3, g = -3 r^-5); those that may be inside follow 32 at a time
// from a queue, whatever lanes they belong to.  Bound by the float64 pipe (28
// operations a pair outside the supports, some 60 inside).
template <int SOFT, bool SOURCE>
__global__ void __launch_bounds__(kVjpWarps * 32) k_vjp_pairs64(VjpArgs V) {
  constexpr bool M4 = SOFT == KDFMM_SOFT_M4;
  __shared__ Chunk64 s_chunk[kVjpWarps];
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  Chunk64& B = s_chunk[threadIdx.x >> 5];
  const int nitems = SOURCE ? V.nleaves + (int)min((int64_t)V.tctr[1], V.tseg_cap) : near_items(V);
  for (int item = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); item < nitems;
       item += (int)((gridDim.x * blockDim.x) >> 5)) {
    const bool seg = item >= V.nleaves;
    const int gi = item - V.nleaves;
    int k, nn;
    int64_t e0 = 0;
    if (SOURCE) {
      k = seg ? V.tseg_leaf[gi] : item;
      const int piece = seg ? gi - V.tseg_first[k] + 1 : 0;
      e0 = V.toff[k] + (int64_t)piece * V.entries;
      nn = min(V.tcnt[k] - piece * V.entries, V.entries);
    } else {
      nn = near_item(V, item, &k, &e0);
    }
    const int a = V.leaf_cells[k];
    const int fa = V.c.first[a], nt = V.c.count[a];
    const int K = 32 / nt, t = lane % nt, sl = lane / nt;
    const bool act = sl < K;
    const int64_t own = (int64_t)fa + t;
    const double xo = V.tp.x[own], yo = V.tp.y[own], zo = V.tp.z[own];
    const double b0 = SOURCE ? 0.0 : V.ab[3 * own], b1 = SOURCE ? 0.0 : V.ab[3 * own + 1],
                 b2 = SOURCE ? 0.0 : V.ab[3 * own + 2];
    const float h2o = M4 ? V.ph[own].w : 0.0f;
    const double hinv_o = M4 ? V.hinv[own] : 0.0;
    const double eps = V.sys_eps[V.leaf_sys[k]];
    const double soft2 = M4 ? 0.0 : eps * eps;       // added to r^2
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;   // vector sum and scalar sum
    // a pair's terms: f, g, own or partner's b, d, partner's mass
    auto terms = [&](double f, double g, double c0, double c1, double c2, double d0, double d1, double d2,
                     double m, double out[4]) {
      const double db = d0 * c0 + d1 * c1 + d2 * c2;
      if (SOURCE) {
        const double u = g * db;
        out[0] = fma(f, c0, u * d0);
        out[1] = fma(f, c1, u * d1);
        out[2] = fma(f, c2, u * d2);
        out[3] = -f * db;
      } else {
        const double u = m * g * db;
        out[0] = u * d0;
        out[1] = u * d1;
        out[2] = u * d2;
        out[3] = m * f;
      }
    };
    auto kernel_pairs = [&](int nq) {
      __syncwarp();
      for (int i0 = 0; i0 < nq; i0 += 32) {
        const bool v = i0 + lane < nq;
        const int e = v ? B.queue[i0 + lane] : 0, o = e >> 8, j = e & 255;
        const double ox = __shfl_sync(full, xo, o), oy = __shfl_sync(full, yo, o),
                     oz = __shfl_sync(full, zo, o), oh = __shfl_sync(full, hinv_o, o);
        double c0 = 0.0, c1 = 0.0, c2 = 0.0;
        if (!SOURCE) {
          c0 = __shfl_sync(full, b0, o);
          c1 = __shfl_sync(full, b1, o);
          c2 = __shfl_sync(full, b2, o);
        }
        B.own[lane] = 0u;
        const unsigned mine = __match_any_sync(full, v ? o : 32);
        __syncwarp();
        if (v) {
          if ((mine & lt) == 0u) B.own[o] = mine;
          if (SOURCE) { c0 = B.w0[j]; c1 = B.w1[j]; c2 = B.w2[j]; }
          const double d0 = SOURCE ? B.x[j] - ox : ox - B.x[j], d1 = SOURCE ? B.y[j] - oy : oy - B.y[j],
                       d2 = SOURCE ? B.z[j] - oz : oz - B.z[j];
          double f, g, out[4];
          m4_pair_fg64(fma(d2, d2, fma(d1, d1, fma(d0, d0, soft2))), oh, B.hinv[j], f, g);
          terms(f, g, c0, c1, c2, d0, d1, d2, B.w0[j], out);
          for (int q = 0; q < 4; ++q) B.term[q][lane] = out[q];
        }
        __syncwarp();
        for (unsigned m = B.own[lane]; m != 0u; m &= m - 1u) {
          const int q = __ffs(m) - 1;
          s0 += B.term[0][q]; s1 += B.term[1][q]; s2 += B.term[2][q]; s3 += B.term[3][q];
        }
        __syncwarp();
      }
    };
    for (int eb = 0; eb < nn;) {
      int cell = -1;
      if (eb + lane < nn)
        cell = SOURCE ? V.leaf_cells[V.tidx[e0 + eb + lane]] : V.near_idx[e0 + eb + lane];
      const int L = stage_chunk(V, B, lane, cell, [&](int at, int p) {
        B.x[at] = V.tp.x[p]; B.y[at] = V.tp.y[p]; B.z[at] = V.tp.z[p];
        if (SOURCE) {
          B.w0[at] = V.ab[3 * (int64_t)p];
          B.w1[at] = V.ab[3 * (int64_t)p + 1];
          B.w2[at] = V.ab[3 * (int64_t)p + 2];
        } else {
          B.w0[at] = V.tp.m[p];
        }
        if (M4) { B.hinv[at] = V.hinv[p]; B.h2[at] = V.ph[p].w; }
        B.id[at] = p;
      });
      const int total = B.beg[L];
      int nq = 0;
      for (int j0 = 0; j0 < total; j0 += K) {
        const int j = j0 + sl;
        bool in = false;
        if (act && j < total && B.id[j] != (int)own) {
          const double d0 = SOURCE ? B.x[j] - xo : xo - B.x[j], d1 = SOURCE ? B.y[j] - yo : yo - B.y[j],
                       d2 = SOURCE ? B.z[j] - zo : zo - B.z[j];
          const double r2 = fma(d2, d2, fma(d1, d1, fma(d0, d0, soft2)));
          in = M4 && maybe_inside(r2, h2o, B.h2[j]);
          if (!in) {
            const double inv = rsqrt64(r2), inv2 = inv * inv;
            if (SOURCE) {
              const double c0 = B.w0[j], c1 = B.w1[j], c2 = B.w2[j], f = inv2 * inv;
              const double fdb = f * (d0 * c0 + d1 * c1 + d2 * c2), u = -3.0 * inv2 * fdb;
              s0 = fma(f, c0, fma(u, d0, s0));
              s1 = fma(f, c1, fma(u, d1, s1));
              s2 = fma(f, c2, fma(u, d2, s2));
              s3 -= fdb;
            } else {
              const double mf = B.w0[j] * (inv2 * inv);
              const double u = -3.0 * (mf * inv2) * (d0 * b0 + d1 * b1 + d2 * b2);
              s3 += mf;
              s0 = fma(u, d0, s0); s1 = fma(u, d1, s1); s2 = fma(u, d2, s2);
            }
          }
        }
        if constexpr (M4) {
          const unsigned marks = __ballot_sync(full, in);
          if (marks != 0u) {
            if (in) B.queue[nq + __popc(marks & lt)] = (uint16_t)(lane << 8 | j);
            nq += __popc(marks);
            if (nq > 512 - 32) {
              kernel_pairs(nq);
              nq = 0;
            }
          }
        }
      }
      if constexpr (M4) {
        if (nq > 0) kernel_pairs(nq);
      }
      eb += L;
    }
    if (!SOURCE) {                     // x_bar_i: -(b_i sum m f + sum m g (d.b_i) d)
      s0 = -fma(s3, b0, s0); s1 = -fma(s3, b1, s1); s2 = -fma(s3, b2, s2);
    }
    for (int s = 1; s < K; ++s) {
      const int src = t + s * nt;
      const double q0 = __shfl_sync(full, s0, src), q1 = __shfl_sync(full, s1, src),
                   q2 = __shfl_sync(full, s2, src), q3 = __shfl_sync(full, s3, src);
      if (sl == 0) { s0 += q0; s1 += q1; s2 += q2; s3 += q3; }
    }
    if (act && sl == 0) {
      if (SOURCE) {
        const double mj = V.tp.m[own];
        atomicAdd(&V.xsrc[3 * own], mj * s0);
        atomicAdd(&V.xsrc[3 * own + 1], mj * s1);
        atomicAdd(&V.xsrc[3 * own + 2], mj * s2);
        atomicAdd(&V.msrc[own], s3);
      } else if (seg) {
        double* P = V.seg_part + (int64_t)gi * 128 + 4 * t;
        P[0] = s0; P[1] = s1; P[2] = s2;
      } else {
        V.xbar[3 * own] += s0;
        V.xbar[3 * own + 1] += s1;
        V.xbar[3 * own + 2] += s2;
      }
    }
  }
}

// Adds the extra items' target-side sums to x_bar, in piece order, warp per leaf
// (the warp of its first extra item), lane per target; eight pieces' loads in
// flight.
__global__ void k_vjp_seg_combine(VjpArgs V) {
  const int lane = threadIdx.x & 31;
  const int nseg = (int)min((int64_t)V.tctr[2], V.seg_cap);
  for (int g = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); g < nseg;
       g += (int)((gridDim.x * blockDim.x) >> 5)) {
    const int k = V.seg_leaf[g];
    const int f = V.seg_first[k];
    if (g != f) continue;
    const int a = V.leaf_cells[k];
    if (lane >= V.c.count[a]) continue;
    const int x = extra_segments(min((int64_t)V.near_cnt[k], V.cap_near), V.entries);
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
#pragma unroll 8
    for (int q = 0; q < x; ++q) {
      const double* P = V.seg_part + (int64_t)(f + q) * 128 + 4 * lane;
      const double2 p01 = *reinterpret_cast<const double2*>(P);
      const double p2 = P[2];
      s0 += p01.x; s1 += p01.y; s2 += p2;
    }
    const int64_t pi = (int64_t)V.c.first[a] + lane;
    V.xbar[3 * pi] += s0;
    V.xbar[3 * pi + 1] += s1;
    V.xbar[3 * pi + 2] += s2;
  }
}

// Moments reverse.  For a cell with cotangents (M_bar, com_bar, Q_bar):
// com = S / M gives S_bar = com_bar / M and M_bar' = M_bar - com_bar.com / M;
// Q (Eq. 7) gives, with G = [[4q0-2q3-2q5, 3q1, 3q2], [., 4q3-2q0-2q5, 3q4],
// [., ., 4q5-2q0-2q3]] and y = x - com:
//   m_bar_i += M_bar' + x.S_bar + y^T G y / 2,   x_bar_i += m_i (S_bar + G y).
// As polynomials in x: a0 + a1.x + x^T (G/2) x and m_i (a1 + G x), with
// a1 = S_bar - G com, a0 = M_bar' + com^T G com / 2; summed over ancestors.
// Each cell's polynomial once, in place of its cotangents (every leaf formed all
// its ancestors' before: four divisions a level and leaf).
__global__ void k_vjp_cell_poly(VjpArgs V) {
  KD_GRID_STRIDE(c, V.ncells) {
    double* cb = V.cell_bar + 10 * (int64_t)c;
    const double inv = 1.0 / V.c.M[c];
    const double com[3] = {V.c.cx[c], V.c.cy[c], V.c.cz[c]};
    const double Sb[3] = {cb[1] * inv, cb[2] * inv, cb[3] * inv};
    const double Mb = cb[0] - (Sb[0] * com[0] + Sb[1] * com[1] + Sb[2] * com[2]);
    const double q0 = cb[4], q1 = cb[5], q2 = cb[6], q3 = cb[7], q4 = cb[8], q5 = cb[9];
    const double g[6] = {4 * q0 - 2 * q3 - 2 * q5, 3 * q1, 3 * q2, 4 * q3 - 2 * q0 - 2 * q5, 3 * q4,
                         4 * q5 - 2 * q0 - 2 * q3};
    const double Gc[3] = {g[0] * com[0] + g[1] * com[1] + g[2] * com[2],
                          g[1] * com[0] + g[3] * com[1] + g[4] * com[2],
                          g[2] * com[0] + g[4] * com[1] + g[5] * com[2]};
    cb[0] = Mb + 0.5 * (com[0] * Gc[0] + com[1] * Gc[1] + com[2] * Gc[2]);
    for (int d = 0; d < 3; ++d) cb[1 + d] = Sb[d] - Gc[d];
    for (int d = 0; d < 6; ++d) cb[4 + d] = g[d];
  }
}

// Half a warp per leaf: lanes 0..9 sum a coefficient each over the leaf and its
// ancestors, then every lane takes particles, adds the parts of x_bar and m_bar
// and writes them in the caller's order.
__global__ void __launch_bounds__(128) k_vjp_moments(VjpArgs V, double* __restrict__ x_bar,
                                                     double* __restrict__ m_bar) {
  const int lane = threadIdx.x & 31, l = lane & 15, g0 = lane & 16;
  const unsigned half = 0xffffu << g0;
  const int k = (blockIdx.x * blockDim.x + threadIdx.x) >> 4;
  if (k >= V.nleaves) return;
  const int leaf = V.leaf_cells[k];
  double s = 0.0;
  for (int c = leaf; c >= 0; c = V.c.parent[c])
    if (l < 10) s += V.cell_bar[10 * (int64_t)c + l];
  double w[10];
#pragma unroll
  for (int j = 0; j < 10; ++j) w[j] = __shfl_sync(half, s, g0 + j);
  const double *a1 = w + 1, *G = w + 4;
  const int f = V.c.first[leaf], cnt = V.c.count[leaf];
  for (int j = l; j < cnt; j += 16) {
    const int64_t p = (int64_t)f + j, i = V.tp.idx[p];
    const double x = V.tp.x[p], y = V.tp.y[p], z = V.tp.z[p], m = V.tp.m[p];
    const double gx = G[0] * x + G[1] * y + G[2] * z, gy = G[1] * x + G[3] * y + G[4] * z,
                 gz = G[2] * x + G[4] * y + G[5] * z;
    m_bar[i] = V.msrc[p] + (w[0] + a1[0] * x + a1[1] * y + a1[2] * z + 0.5 * (x * gx + y * gy + z * gz));
    x_bar[3 * i] = V.xbar[3 * p] + V.xsrc[3 * p] + m * (a1[0] + gx);
    x_bar[3 * i + 1] = V.xbar[3 * p + 1] + V.xsrc[3 * p + 1] + m * (a1[1] + gy);
    x_bar[3 * i + 2] = V.xbar[3 * p + 2] + V.xsrc[3 * p + 2] + m * (a1[2] + gz);
  }
}

}  // namespace

// Scratch of the adjoint, kept with the handle (grows by an eighth more than
// asked for: near lists change with the particles; freed with it).  The calls of
// a handle follow one another on it, whatever streams they are on: each waits for
// the event that the one before recorded.
static int ensure_vjp_scratch(kdfmm_tree_s* t, size_t bytes, cudaStream_t s) {
  int rc;
  if (!t->vjp_done &&
      (rc = check_cuda(cudaEventCreateWithFlags(&t->vjp_done, cudaEventDisableTiming), "adjoint event")))
    return rc;
  if (t->vjp_cap >= bytes) return check_cuda(cudaStreamWaitEvent(s, t->vjp_done, 0), "adjoint order");
  if ((rc = check_cuda(cudaEventSynchronize(t->vjp_done), "adjoint order"))) return rc;
  cudaFree(t->vjp_buf);
  t->vjp_buf = nullptr;
  t->vjp_cap = 0;
  bytes += bytes / 8;
  rc = check_cuda(cudaMalloc(&t->vjp_buf, bytes), "adjoint scratch");
  if (!rc) t->vjp_cap = bytes;
  else cudaGetLastError();
  return rc;
}

int run_vjp(kdfmm_tree_s* t, const double* a_bar, double* x_bar, double* m_bar, cudaStream_t s) {
  const int64_t n = t->n;
  const int nl = t->nleaves, nc = t->ncells;
  const int64_t nnear = t->host_stats[KDFMM_STAT_NNEAR];
  VjpArgs V{};
  V.n = n;
  V.nleaves = nl;
  V.ncells = nc;
  V.leaf_sys = t->leaf_sys;
  V.sys_root = t->sys_root;
  V.sys_eps = t->sys_eps;
  V.mixed = t->p.precision == KDFMM_MIXED;
  V.leaf_cells = t->leaf_cells;
  V.leaf_rank = t->leaf_rank;
  V.c = t->c;
  V.tp = t->tp;
  V.ph = t->ph;
  V.lexp32 = t->lexp32;
  V.lexp64 = t->lexp64;
  V.far_cnt = t->L.far_cnt; V.far_idx = t->L.far_idx;
  V.near_cnt = t->L.near_cnt; V.near_idx = t->L.near_idx;
  V.far_off = t->L.far_off; V.near_off = t->L.near_off;
  V.cap_far = t->L.exact ? INT64_MAX : t->L.cap_far;
  V.cap_near = t->L.exact ? INT64_MAX : t->L.cap_near;
  // pieces short enough for a dozen warps on each of the SMs' four schedulers,
  // between 8 and 256 leaves
  V.entries = 256;
  while (V.entries > 8 && nnear / V.entries < (int64_t)sm_count() * 48) V.entries >>= 1;
  V.tcap = nnear;
  V.seg_cap = V.tseg_cap = nnear / V.entries + 1;
  // scratch, in two parts: what starts at zero first (one memset), then the
  // rest; every array on a 16-byte boundary
  size_t at = 0, zeroed = 0;
  auto take = [&](size_t bytes) {
    const size_t was = at;
    at += (bytes + 15) / 16 * 16;
    return was;
  };
  const size_t o_cell = take((size_t)nc * 10 * 8), o_xsrc = take((size_t)n * 3 * 8),
               o_msrc = take((size_t)n * 8),
               o_tcnt = take((size_t)nl * 4), o_tcur = take((size_t)nl * 4), o_tctr = take(64);
  zeroed = at;
  const size_t o_xbar = take((size_t)n * 3 * 8), o_cbar = take((size_t)nl * 20 * 8),
               o_toff = take((size_t)nl * 8), o_tfirst = take((size_t)nl * 4),
               o_tidx = take((size_t)nnear * 4), o_tseg = take((size_t)V.tseg_cap * 4),
               o_nfirst = take((size_t)nl * 4), o_nseg = take((size_t)V.seg_cap * 4),
               o_npart = take((size_t)V.seg_cap * 128 * 8);
  const size_t o_close = V.mixed ? take((size_t)(2 * nl + V.seg_cap + V.tseg_cap) * 4) : 0;
  const size_t o_q = V.mixed ? take((size_t)n * 56) : take((size_t)n * 32);
  // a call that is being captured takes its scratch from the stream's pool (a
  // graph must not refer to memory that the handle may replace)
  cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
  int rc = check_cuda(cudaStreamIsCapturing(s, &capturing), "adjoint stream");
  if (rc) return rc;
  const bool pooled = capturing != cudaStreamCaptureStatusNone;
  char* buf = nullptr;
  if (pooled) rc = check_cuda(cudaMallocAsync((void**)&buf, at, s), "adjoint scratch");
  else if (!(rc = ensure_vjp_scratch(t, at, s))) buf = static_cast<char*>(t->vjp_buf);
  if (rc) return rc;
  V.cell_bar = (double*)(buf + o_cell);
  V.xsrc = (double*)(buf + o_xsrc);
  V.msrc = (double*)(buf + o_msrc);
  V.tcnt = (int32_t*)(buf + o_tcnt);
  V.tcur = (int32_t*)(buf + o_tcur);
  V.tctr = (unsigned long long*)(buf + o_tctr);
  V.xbar = (double*)(buf + o_xbar);
  V.cbar = (double*)(buf + o_cbar);
  V.toff = (int64_t*)(buf + o_toff);
  V.tseg_first = (int32_t*)(buf + o_tfirst);
  V.tidx = (int32_t*)(buf + o_tidx);
  V.tseg_leaf = (int32_t*)(buf + o_tseg);
  V.seg_first = (int32_t*)(buf + o_nfirst);
  V.seg_leaf = (int32_t*)(buf + o_nseg);
  V.seg_part = (double*)(buf + o_npart);
  V.close_t = (int32_t*)(buf + o_close);
  V.close_s = V.close_t + nl + V.seg_cap;
  V.q0 = (float4*)(buf + o_q);
  V.q1 = V.q0 + n;
  V.q2 = V.q1 + n;
  V.q3 = (float2*)(V.q2 + n);
  V.ab = (double*)(buf + o_q);
  V.hinv = V.ab + 3 * n;
  cudaMemsetAsync(buf, 0, zeroed, s);
  const bool m4 = t->p.soft_kind == KDFMM_SOFT_M4;
  const unsigned gw = blocks_for((int64_t)nl * 32, 128);
  const unsigned gi = blocks_for((nl + V.seg_cap) * 32, 128);    // a warp per item that there may be
  const unsigned gclose = std::min<unsigned>(gi, grid_blocks(5));   // (resident blocks: found work in a loop)
  k_vjp_l2p<<<gw, kL2PWarps * 32, 0, s>>>(a_bar, V, m4);
  const bool std_exp = t->p.expansion == KDFMM_EXPANSION_STANDARD;
  if (V.mixed) {
    if (std_exp) k_vjp_m2l32<true><<<gw, kM2LWarps * 32, 0, s>>>(V);
    else k_vjp_m2l32<false><<<gw, kM2LWarps * 32, 0, s>>>(V);
  } else {
    if (std_exp) k_vjp_m2l64<true><<<gw, kM2LWarps * 32, 0, s>>>(V);
    else k_vjp_m2l64<false><<<gw, kM2LWarps * 32, 0, s>>>(V);
  }
  k_near_plan<<<std::min<unsigned>(blocks_for(nl, 128), grid_blocks()), 128, 0, s>>>(V);
  k_tr_count<<<grid_blocks(), 256, 0, s>>>(V);
  k_tr_plan<<<blocks_for(nl, 128), 128, 0, s>>>(V);
  k_tr_fill<<<grid_blocks(), 256, 0, s>>>(V);
  if (V.mixed) {
    if (m4) {
      k_vjp_target32<KDFMM_SOFT_M4><<<gi, kVjpWarps * 32, 0, s>>>(V);
      k_vjp_source32<KDFMM_SOFT_M4><<<gi, kVjpWarps * 32, 0, s>>>(V);
      k_vjp_close32<KDFMM_SOFT_M4><<<gclose, kVjpWarps * 32, 0, s>>>(V);
    } else {
      k_vjp_target32<KDFMM_SOFT_PLUMMER><<<gi, kVjpWarps * 32, 0, s>>>(V);
      k_vjp_source32<KDFMM_SOFT_PLUMMER><<<gi, kVjpWarps * 32, 0, s>>>(V);
      k_vjp_close32<KDFMM_SOFT_PLUMMER><<<gclose, kVjpWarps * 32, 0, s>>>(V);
    }
    t->launches += 1;
  } else {
    if (m4) {
      k_vjp_pairs64<KDFMM_SOFT_M4, false><<<gi, kVjpWarps * 32, 0, s>>>(V);
      k_vjp_pairs64<KDFMM_SOFT_M4, true><<<gi, kVjpWarps * 32, 0, s>>>(V);
    } else {
      k_vjp_pairs64<KDFMM_SOFT_PLUMMER, false><<<gi, kVjpWarps * 32, 0, s>>>(V);
      k_vjp_pairs64<KDFMM_SOFT_PLUMMER, true><<<gi, kVjpWarps * 32, 0, s>>>(V);
    }
  }
  k_vjp_seg_combine<<<grid_blocks(2), 256, 0, s>>>(V);
  k_vjp_cell_poly<<<std::min<unsigned>(blocks_for(nc, 128), grid_blocks()), 128, 0, s>>>(V);
  k_vjp_moments<<<blocks_for((int64_t)nl * 16, 128), 128, 0, s>>>(V, x_bar, m_bar);
  t->launches += 11;
  rc = check_cuda(cudaGetLastError(), "adjoint launch");
  if (pooled) {
    cudaFreeAsync(buf, s);
  } else {
    const int err = check_cuda(cudaEventRecord(t->vjp_done, s), "adjoint order");
    rc = rc ? rc : err;
  }
  return rc;
}

}  // namespace kdfmm
