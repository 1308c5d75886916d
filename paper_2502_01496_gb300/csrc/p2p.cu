// Short-range direct summation (P2P) over each leaf's near list, L2P (Eq. 8)
// of its local expansion, and the assembly a = a_short + a_long (Eq. 3) in
// the caller's particle order.
//
// Pair interaction on particle i from j (d = x_i - x_j, j != i):
//   Plummer:   a = -m_j d / (d^2 + eps^2)^(3/2),  phi = -m_j / sqrt(d^2 + eps^2);
//   M4 kernel: the symmetrised Green's function of Eq. 13,
//              a = -m_j [g(r,h_i) + g(r,h_j)]/2 d/r,  phi = -m_j [psi(r,h_i) + psi(r,h_j)]/2,
//              with g = F(q)/r^2 (F the mass fraction of the cubic spline inside
//              q = r/h) and psi = P(q)/h; outside q = 2 they are 1/r^2 and 1/r
//              (Eq. 15).  Written here as g/r = h^-3 F(q)/q^3.
//
// One warp per target leaf.  A leaf of n_t <= 32 targets uses K = 32 / n_t
// source slices: lane = target + n_t * slice, slice k takes sources k, k+K, ...
// of every near leaf, and the slices are combined at the end.  A near list
// longer than a work item (256 leaves; fewer in small float64 calls) is split
// (a large leaf in the sparse outskirts of a centrally condensed system can have
// most of the system in it): the leaf's warp takes the first item, the others are
// for other warps, and their partial sums are added afterwards in order, so the
// result does not depend on scheduling.
//
// Mixed mode: positions are float32 offsets from each particle's own leaf
// centre of mass; the target is shifted by the difference of the two leaf
// centres (from (high, low) float pairs), so no large coordinate enters the
// float32 arithmetic.  Each near leaf's contribution is summed in float32 and
// folded into a (high, low) accumulator with two-sum; the long-range part is
// added to the (high, low) pairs and the result converted to float64 once.
// FP64 mode uses float64 absolute positions.
#include <algorithm>
#include <climits>

#include "kdfmm_internal.cuh"

namespace kdfmm {

namespace {

struct P2PArgs {
  const int32_t* leaf_cells;
  const int32_t* counters;   // counters[C_LEAVES]: leaves
  int64_t cap_near;          // entries a list may hold (slot size, or no limit)
  int max_leaves;            // leaves the lists were made for
  const int32_t *cfirst, *ccount;
  const int32_t* near_cnt;
  const int32_t* near_idx;
  const int64_t* near_off;
  const float4* src32;       // cell (hi, M), (lo, 0), ...
  const float4* pf;          // (x - com_leaf, m)
  const float4* ph;          // (1/h, 1/h^3, h, (2h)^2)
  PCols tp;                  // float64 tree-order particles
  const double* cx;
  const double *cy, *cz;
  const float* lexp32;
  const double* lexp64;
  const float4* walk;        // cell (com, s) float32
  const float4* walk2;       // cell (h_max, skip, count, 0)
  const int32_t* leaf_sys;   // system of each leaf
  const double* sys_eps;     // Plummer softening length of each system
  double* a;
  double* phi;
  // near lists longer than item_entries(): the first item is the leaf's own, the
  // others (counters[C_SEGS], at most seg_cap) follow the leaves, and
  // k_seg_combine adds their partial sums seg_part in order
  const int32_t* seg_first;
  const int32_t* seg_leaf;
  double* seg_part;
  int64_t seg_cap;
  const int64_t* sys_off;    // float64: first particle of each system; mixed: null
  bool grouped;              // a work item is a group of segments (k_p2p_fp64: GROUPS)
};

// Near entries per segment, by the particles of the leaf's own system alone: an
// eager evaluation, a replayed graph and a batch that holds the system sum
// alike.  Float64 evaluations of few particles take short segments: their leaves
// are too few warps for the GPU's 608 float64 pipes (4096 particles: 367 leaves
// with ~108 near leaves each).  The P2P of a Plummer sphere (theta 0.5) in segments
// of 8, 32, 64 and 256: 7000 particles 0.43, 0.53, 0.61, 1.20 ms; 30000 1.58, 1.61,
// 1.72, 2.23; 90000 5.42, 5.22, 5.36, 6.68; 200000 18.5, 17.5, 17.6, 18.8; 400000 24.1,
// 22.2, 22.1, 23.4.  Where two are close the longer one is taken, whose partial sums
// need less room.  Mixed evaluations keep 256: a shorter segment would move the
// chunks of 256 sources whose float32 sums are folded at once.
//
// A segment's sums start at zero.  Those of a group of 256 entries are added in
// order, then the groups: (first segment + expansion + rest of the first group)
// + (second group + third + ...).  So it makes no difference who adds: with few
// particles in the call each segment is a work item whose sums go to memory
// (1 KB) for k_seg_combine; a work item is a group, its segments added in
// registers, in forests from kFullCall particles on, whose leaves themselves fill
// the GPU (16384 warps and more), and in calls of more than kShortItems segments
// (32768 groups and more; 1 GB), whose near lists are long: segments would take
// 128 bytes a near entry, where groups take 4.  256 systems of 4096, 9.6e6 near
// entries: 47.9 ms a call and 1.2 GB by segments, 48.1 ms and 38 MB by groups; 64 of
// 8191: 27.5 and 28.4 ms.  One system with each leaf near all others: 3000 particles
// 10.8 ms and 1.2 GB, 10.4 and 36 MB; 8000 74.7 and 8.2 GB, 72.8 and 0.25.
constexpr int64_t kFullCall = 262144, kShortItems = int64_t(1) << 20;
constexpr int kSegSteps = 3;
__host__ __device__ __forceinline__ int64_t seg_below(int step) {      // particles, exclusive
  return step == 0 ? 8192 : (step == 1 ? 65536 : 262144);
}
__host__ __device__ __forceinline__ int seg_length(int step) {
  return step == 0 ? 8 : (step == 1 ? 32 : (step == 2 ? 64 : kSegEntries));
}
__host__ __device__ __forceinline__ int seg_step(int64_t n) {
  int step = 0;
  while (step < kSegSteps && n >= seg_below(step)) ++step;
  return step;
}
// Entries per work item.
__device__ __forceinline__ int item_entries(bool grouped, int seglen) {
  return grouped ? kSegEntries : seglen;
}
__device__ __forceinline__ int leaf_segment(const int64_t* __restrict__ sys_off, int sys) {
  return sys_off == nullptr ? kSegEntries : seg_length(seg_step(sys_off[sys + 1] - sys_off[sys]));
}

// M4 cubic spline, q = r/h < 2: F(q)/q^3 and P(q) (qi = 1/q).
__device__ __forceinline__ float m4_fq3(float q, float qi) {
  if (q < 1.0f) return 1.3333333f + q * q * (-1.2f + 0.5f * q);
  return 2.6666667f + q * (-3.0f + q * (1.2f - 0.16666667f * q)) - 0.06666667f * qi * qi * qi;
}
__device__ __forceinline__ float m4_pot(float q, float qi) {
  const float q2 = q * q;
  if (q < 1.0f) return 1.4f + q2 * (-0.6666667f + q2 * (0.3f - 0.1f * q));
  return 1.6f + q2 * (-1.3333333f + q * (1.0f + q * (-0.3f + 0.033333335f * q))) - 0.06666667f * qi;
}
// Interaction of one target with one source, float32, accumulated into f*.
template <int SOFT>
__device__ __forceinline__ void pair32(float rx, float ry, float rz, float mj, const float4& hi,
                                       const float4& hj, float eps2, float& fx, float& fy,
                                       float& fz, float& fp) {
  if (SOFT == KDFMM_SOFT_PLUMMER) {
    const float r2 = rx * rx + ry * ry + rz * rz + eps2;
    const float inv = rsqrt_ftz(r2);
    const float minv = mj * inv;
    const float f = minv * inv * inv;
    fx -= f * rx; fy -= f * ry; fz -= f * rz;
    fp -= minv;
  } else {
    const float r2 = fmaxf(rx * rx + ry * ry + rz * rz, 1e-30f);
    const float inv = rsqrt_ftz(r2);
    const float r = r2 * inv;
    const float qa = r * hi.x, qb = r * hj.x;
    float f, p;
    if (qa < 2.0f || qb < 2.0f) {
      const float inv3 = inv * inv * inv;
      const float fa = qa < 2.0f ? hi.y * m4_fq3(qa, inv * hi.z) : inv3;
      const float fb = qb < 2.0f ? hj.y * m4_fq3(qb, inv * hj.z) : inv3;
      const float pa = qa < 2.0f ? hi.x * m4_pot(qa, inv * hi.z) : inv;
      const float pb = qb < 2.0f ? hj.x * m4_pot(qb, inv * hj.z) : inv;
      f = 0.5f * (fa + fb);
      p = 0.5f * (pa + pb);
    } else {
      f = inv * inv * inv;
      p = inv;
    }
    const float mf = mj * f;
    fx -= mf * rx; fy -= mf * ry; fz -= mf * rz;
    fp -= mj * p;
  }
}

// One side of the symmetrised M4 pair, branch-free: returns g/r (force per
// unit displacement and mass) and psi for smoothing length h (hinv = 1/h,
// hinv3 = 1/h^3), at distance r (inv = 1/r, inv3 = 1/r^3).
//   q < 1     : g/r = h^-3 (4/3 - 6/5 q^2 + 1/2 q^3),
//               psi = h^-1 (7/5 - 2/3 q^2 + 3/10 q^4 - 1/10 q^5)
//   1 <= q < 2: g/r = r^-3 (1 - t^4 (1 - 4/5 t + t^2/6)),  t = 2 - q
//               psi = r^-1 (1 - t^5 (1/10 - t/30))
//   q >= 2    : g/r = r^-3, psi = 1/r  (t clamped to 0)
// The [1,2) force is the enclosed mass 1 - int_q^2 (2-u)^3 u^2 du written in
// t; the [1,2) potential is 1/r + h^-1 R(q) with R = 8/5 - 4/3 q^2 + q^3 -
// 3/10 q^4 + q^5/30 - 16/(15 q), and q R(q) = -t^5 (1/10 - t/30) exactly.
__device__ __forceinline__ void m4_side(float r, float inv, float inv3, float hinv, float hinv3,
                                        float& f, float& p) {
  const float q = r * hinv;
  const float q2 = q * q;
  const float t = fmaxf(2.0f - q, 0.0f);
  const float t2 = t * t;
  const float t4 = t2 * t2;
  const float g = 1.0f + t * (-0.8f + 0.16666667f * t);
  const float f_out = inv3 * fmaf(-t4, g, 1.0f);
  const float f_in = hinv3 * (1.3333334f + q2 * (-1.2f + 0.5f * q));
  f = q < 1.0f ? f_in : f_out;
  const float p_in = hinv * (1.4f + q2 * (-0.6666667f + q2 * (0.3f - 0.1f * q)));
  const float p_out = inv * fmaf(-t4 * t, fmaf(-0.033333335f, t, 0.1f), 1.0f);
  p = q < 1.0f ? p_in : p_out;
}

// Symmetrised M4 pair (Eq. 13), branch-free; hi / hj = (1/h, 1/h^3, h, -).
__device__ __forceinline__ void m4pair32(float rx, float ry, float rz, float mj, const float4& hi,
                                         const float4& hj, float& fx, float& fy, float& fz,
                                         float& fp) {
  const float r2 = fmaxf(rx * rx + ry * ry + rz * rz, 1e-30f);
  const float inv = rsqrt_ftz(r2);
  const float r = r2 * inv;
  const float inv3 = inv * inv * inv;
  float fa, pa, fb, pb;
  m4_side(r, inv, inv3, hi.x, hi.y, fa, pa);
  m4_side(r, inv, inv3, hj.x, hj.y, fb, pb);
  const float mf = 0.5f * mj * (fa + fb);
  fx -= mf * rx; fy -= mf * ry; fz -= mf * rz;
  fp -= 0.5f * mj * (pa + pb);
}

// L2P of the 20 coefficients at x: a = -(C1 + C2 x + C3 x x / 2),
// phi = C0 + C1.x + x.C2.x/2 + C3 x x x / 6.  Returns the parts beyond the
// leading C0 / C1 terms (which the caller adds in higher precision).
template <class T>
__device__ __forceinline__ void l2p_tail(const T* C, T x, T y, T z, T& ax, T& ay, T& az, T& p) {
  const T v0 = C[4] * x + C[5] * y + C[6] * z;
  const T v1 = C[5] * x + C[7] * y + C[8] * z;
  const T v2 = C[6] * x + C[8] * y + C[9] * z;
  const T xx = x * x, yy = y * y, zz = z * z, xy = x * y, xz = x * z, yz = y * z;
  const T w0 = C[10] * xx + C[13] * yy + C[15] * zz + T(2) * (C[11] * xy + C[12] * xz + C[14] * yz);
  const T w1 = C[11] * xx + C[16] * yy + C[18] * zz + T(2) * (C[13] * xy + C[14] * xz + C[17] * yz);
  const T w2 = C[12] * xx + C[17] * yy + C[19] * zz + T(2) * (C[14] * xy + C[15] * xz + C[18] * yz);
  ax = -(v0 + T(0.5) * w0);
  ay = -(v1 + T(0.5) * w1);
  az = -(v2 + T(0.5) * w2);
  p = (C[1] * x + C[2] * y + C[3] * z) + T(0.5) * (x * v0 + y * v1 + z * v2) +
      (x * w0 + y * w1 + z * w2) / T(6);
}

template <int SOFT, bool SELF>
__device__ __forceinline__ void near_leaf32(const P2PArgs& A, int fb, int nb, int sl, int K, int t,
                                            float xs, float ys, float zs, const float4& hi,
                                            float eps2f, float& fx, float& fy, float& fz,
                                            float& fp) {
  for (int j = sl; j < nb; j += K) {
    if (SELF && j == t) continue;
    const float4 s = A.pf[fb + j];
    if (SOFT == KDFMM_SOFT_M4)     // own leaf: nearly every pair is inside a support
      m4pair32(xs - s.x, ys - s.y, zs - s.z, s.w, hi, A.ph[fb + j], fx, fy, fz, fp);
    else
      pair32<SOFT>(xs - s.x, ys - s.y, zs - s.z, s.w, hi, hi, eps2f, fx, fy, fz, fp);
  }
}

// Newtonian pair (no kernel softening, optional Plummer eps^2), float32.
__device__ __forceinline__ void newton32(float rx, float ry, float rz, float mj, float eps2,
                                         float& fx, float& fy, float& fz, float& fp) {
  const float r2 = rx * rx + ry * ry + rz * rz + eps2;
  const float inv = rsqrt_ftz(r2);
  const float minv = mj * inv;
  const float f = minv * inv * inv;
  fx -= f * rx; fy -= f * ry; fz -= f * rz;
  fp -= minv;
}

// Newtonian pair for r2 > 0 outside both kernel supports; contributes
// nothing when `inside` (that pair is evaluated with the kernel instead).
__device__ __forceinline__ void newton32_outside(float rx, float ry, float rz, float r2, float mj,
                                                 bool inside, float& fx, float& fy, float& fz,
                                                 float& fp) {
  const float inv = rsqrt_ftz(r2);              // infinite for coincident pairs: selected away
  const float m1 = mj * inv;
  const float minv = inside ? 0.0f : m1;
  const float f = inside ? 0.0f : m1 * inv * inv;
  fx -= f * rx; fy -= f * ry; fz -= f * rz;
  fp -= minv;
}

constexpr int kStageCap = 256;     // staged sources per warp and chunk
constexpr int kStageRounds = 4;    // staging loads in flight per lane (half with M4 data)
constexpr int kP2PWarps = 4;

// Mixed precision.  Per chunk of near leaves the warp stages their particles
// in shared memory, shifted to the target leaf's centre of mass, and splits
// them into sources that lie outside the kernel support of every target
// (|s| - s_alpha >= 2 max(h_max,alpha, h_j): plain 1/r^2, Eq. 15) and sources
// that may not (full M4 pair).  The split only selects the instruction path:
// the M4 pair reduces to the same 1/r^2 outside the support.  The target's
// own leaf is summed separately so that j = i is skipped exactly.
template <int SOFT>
__global__ void __launch_bounds__(kP2PWarps * 32, 6) k_p2p_mixed(P2PArgs A) {
  constexpr bool M4 = SOFT == KDFMM_SOFT_M4;
  constexpr int R = M4 ? kStageRounds / 2 : kStageRounds;
  __shared__ float4 s_pos[kP2PWarps][kStageCap];
  __shared__ float4 s_ker[M4 ? kP2PWarps : 1][M4 ? kStageCap : 1];
  __shared__ int s_tbeg[kP2PWarps][32];                    // chunk's leaves: first particle - staged start
  __shared__ float4 s_toff[kP2PWarps][32];                 // and offset to the target com
  __shared__ unsigned s_bits[kP2PWarps][kStageCap / 32];   // staged starts
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nleaves = min(A.counters[C_LEAVES], A.max_leaves);
  const int nitems = nleaves + (int)min((int64_t)A.counters[C_SEGS], A.seg_cap);
  for (int item = blockIdx.x * kP2PWarps + warp; item < nitems; item += gridDim.x * kP2PWarps) {
  const bool seg = item >= nleaves;
  const int g = item - nleaves;
  const int k = seg ? A.seg_leaf[g] : item;
  if (k < 0) continue;
  float4* sp = s_pos[warp];
  float4* sk = s_ker[M4 ? warp : 0];
  int* tb = s_tbeg[warp];
  float4* toff = s_toff[warp];
  const int a = A.leaf_cells[k];
  const int fa = A.cfirst[a], nt = A.ccount[a];
  const int K = 32 / nt;
  const int t = lane % nt, sl = lane / nt;
  const bool act = sl < K;
  const float4 xa = A.pf[fa + t];
  float4 hi = make_float4(0.f, 0.f, 0.f, 0.f);
  if (M4) hi = A.ph[fa + t];
  const float4 ca = A.src32[4 * a], cal = A.src32[4 * a + 1];
  const float sa = A.walk[a].w, hmax_a = A.walk2[a].x;
  const double eps = A.sys_eps[A.leaf_sys[k]];
  float eps2f = (float)(eps * eps);
  asm("" : "+f"(eps2f));   // opaque: not recomputed in float64 at every pair
  float axh = 0.f, axl = 0.f, ayh = 0.f, ayl = 0.f, azh = 0.f, azl = 0.f, ph_ = 0.f, pl = 0.f;
  if (!seg) {
    float fx = 0.f, fy = 0.f, fz = 0.f, fp = 0.f;
    if (act)
      near_leaf32<SOFT, true>(A, fa, nt, sl, K, t, xa.x, xa.y, xa.z, hi, eps2f, fx, fy, fz, fp);
    df_add(axh, axl, fx); df_add(ayh, ayl, fy); df_add(azh, azl, fz); df_add(ph_, pl, fp);
  }
  const unsigned full = 0xffffffffu, lt = (1u << lane) - 1u;
  const int64_t nall = min((int64_t)A.near_cnt[k], A.cap_near);
  const int64_t sidx = seg ? (int64_t)(g - A.seg_first[k] + 1) : 0;
  const int seglen = leaf_segment(A.sys_off, A.leaf_sys[k]);
  const int64_t e1 = A.near_off[k] + min(nall, (sidx + 1) * seglen);
  for (int64_t e = A.near_off[k] + sidx * seglen; e < e1;) {
    // up to 32 candidate leaves, one per lane
    const int64_t my = e + lane;
    int cnt = 0, first = 0;
    float dx = 0.f, dy = 0.f, dz = 0.f;
    if (my < e1) {
      const int b = A.near_idx[my];
      if (b != a) {
        cnt = A.ccount[b];
        first = A.cfirst[b];
        const float4 cb = A.src32[4 * b], cbl = A.src32[4 * b + 1];
        dx = (cb.x - ca.x) + (cbl.x - cal.x);
        dy = (cb.y - ca.y) + (cbl.y - cal.y);
        dz = (cb.z - ca.z) + (cbl.z - cal.z);
      }
    }
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int w = __shfl_up_sync(full, incl, o);
      if (lane >= o) incl += w;
    }
    const int L = __popc(__ballot_sync(full, my < e1 && incl <= kStageCap));
    // stage the chunk's sources with flat indexing: a lane takes staged index
    // idx = 32 round + lane; the leaf of idx is the number of leaves that start
    // at or before it, counted on a bitmap of the starts (one word a round, so a
    // population count; a binary search over the starts took a sixth of the
    // kernel on Plummer spheres).  Every load of a batch of R rounds is issued
    // before any is used (the loads are L2 gathers: latency-bound)
    const bool has = lane < L && cnt > 0;
    const unsigned leaves = __ballot_sync(full, has);
    if (lane < kStageCap / 32) s_bits[warp][lane] = 0u;
    __syncwarp();
    if (has) {
      const int slot = __popc(leaves & lt), beg = incl - cnt;
      tb[slot] = first - beg;             // particle = tb + staged index
      toff[slot] = make_float4(dx, dy, dz, 0.0f);
      atomicOr(&s_bits[warp][beg >> 5], 1u << (beg & 31));
    }
    __syncwarp();
    const int total = __shfl_sync(full, incl, L - 1);
    int nN = 0, nK = 0, before = -1;      // leaves that start before the round, minus one
    for (int r0 = 0; r0 < total; r0 += 32 * R) {
      float4 pv[R], hv[R];
      int lv[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int idx = r0 + 32 * r + lane;
        const unsigned starts = r0 + 32 * r < total ? s_bits[warp][(r0 >> 5) + r] : 0u;
        const int l = before + __popc(starts & (lt << 1 | 1u));
        before += __popc(starts);
        lv[r] = l;
        pv[r] = make_float4(0.f, 0.f, 0.f, 0.f);
        hv[r] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (idx < total) {
          const int src = tb[l] + idx;
          pv[r] = A.pf[src];
          if (M4) hv[r] = A.ph[src];
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const bool v = r0 + 32 * r + lane < total;
        const float4 o = toff[lv[r]];
        float4 p = pv[r];
        p.x += o.x; p.y += o.y; p.z += o.z;
        bool need = false;
        if (M4 && v) {
          // d - s_a < X  <=>  d^2 < (s_a + X)^2 (both sides >= 0)
          const float d2 = p.x * p.x + p.y * p.y + p.z * p.z;
          const float reach = sa + 2.0f * fmaxf(hmax_a, hv[r].z) * 1.0001f + 1e-20f;
          need = d2 < reach * reach;
        }
        const unsigned vm = __ballot_sync(full, v), nm = __ballot_sync(full, v && need);
        if (v) {
          if (need) {
            const int pos = kStageCap - 1 - (nK + __popc(nm & lt));
            sp[pos] = p;
            sk[pos] = hv[r];
          } else {
            sp[nN + __popc(vm & ~nm & lt)] = p;
          }
        }
        nK += __popc(nm);
        nN += __popc(vm & ~nm);
      }
    }
    __syncwarp();
    float fx = 0.f, fy = 0.f, fz = 0.f, fp = 0.f;
    if (act) {
#pragma unroll 4
      for (int j = sl; j < nN; j += K) {
        const float4 s = sp[j];
        newton32(xa.x - s.x, xa.y - s.y, xa.z - s.z, s.w, eps2f, fx, fy, fz, fp);
      }
      if (M4) {
        // Two passes over the lane's pairs of the kernel segment, 128 at a
        // time.  Pass 1: every pair as a plain 1/r^2 pair, except those
        // inside either smoothing kernel's support (r < 2 max(h_i, h_j)),
        // which are marked in a bit mask instead; pass 2 visits only the
        // marked pairs with the full symmetrised M4 pair.  Only a sixth of the
        // segment's pairs is inside, and a lane's marked pairs are dense work.
        const float h2i = hi.w;                                   // (2 h_i)^2
        const int j0 = kStageCap - nK + sl;
        const int npair = j0 < kStageCap ? (kStageCap - j0 + K - 1) / K : 0;
        for (int i0 = 0; i0 < npair; i0 += 128) {
          const int nb = min(128, npair - i0);
          const int jb = j0 + K * i0;
          uint32_t in[4] = {0u, 0u, 0u, 0u};
#pragma unroll
          for (int w = 0; w < 4; ++w) {
            const int nbw = min(32, nb - 32 * w);
#pragma unroll 4
            for (int b = 0; b < nbw; ++b) {
              const int j = jb + K * (32 * w + b);
              const float4 s = sp[j];
              const float rx = xa.x - s.x, ry = xa.y - s.y, rz = xa.z - s.z;
              const float r2 = rx * rx + ry * ry + rz * rz;
              const bool inside = r2 < fmaxf(h2i, sk[j].w);        // inside (2 max(h_i, h_j))
              in[w] |= (uint32_t)inside << b;
              newton32_outside(rx, ry, rz, r2, s.w, inside, fx, fy, fz, fp);
            }
          }
#pragma unroll
          for (int w = 0; w < 4; ++w) {
            uint32_t msk = in[w];
            while (msk != 0u) {
              const int b = __ffs(msk) - 1;
              msk &= msk - 1u;
              const int j = jb + K * (32 * w + b);
              const float4 s = sp[j];
              m4pair32(xa.x - s.x, xa.y - s.y, xa.z - s.z, s.w, hi, sk[j], fx, fy, fz, fp);
            }
          }
        }
      }
    }
    df_add(axh, axl, fx); df_add(ayh, ayl, fy); df_add(azh, azl, fz); df_add(ph_, pl, fp);
    __syncwarp();
    e += L;
  }
  // combine the source slices of each target
  for (int s = 1; s < K; ++s) {
    const int src = t + s * nt;
    const float bxh = __shfl_sync(full, axh, src), bxl = __shfl_sync(full, axl, src);
    const float byh = __shfl_sync(full, ayh, src), byl = __shfl_sync(full, ayl, src);
    const float bzh = __shfl_sync(full, azh, src), bzl = __shfl_sync(full, azl, src);
    const float bph = __shfl_sync(full, ph_, src), bpl = __shfl_sync(full, pl, src);
    if (sl == 0) {
      df_add2(axh, axl, bxh, bxl);
      df_add2(ayh, ayl, byh, byl);
      df_add2(azh, azl, bzh, bzl);
      df_add2(ph_, pl, bph, bpl);
    }
  }
  if (sl != 0 || !act) continue;
  if (seg) {
    double* P = A.seg_part + (int64_t)g * 128 + 4 * t;
    P[0] = (double)axh + (double)axl;
    P[1] = (double)ayh + (double)ayl;
    P[2] = (double)azh + (double)azl;
    P[3] = (double)ph_ + (double)pl;
    continue;
  }
  const float* C = A.lexp32 + 24 * (int64_t)k;
  float tx, ty, tz, tp_;
  l2p_tail<float>(C, xa.x, xa.y, xa.z, tx, ty, tz, tp_);
  // a = a_short + a_long (Eq. 3) and phi likewise, summed as (high, low)
  // float pairs and converted to float64 once (the FP64 pipe runs at 1/64 rate)
  df_add2(axh, axl, -C[1], -C[21]);
  df_add2(ayh, ayl, -C[2], -C[22]);
  df_add2(azh, azl, -C[3], -C[23]);
  df_add2(ph_, pl, C[0], C[20]);
  df_add(axh, axl, tx); df_add(ayh, ayl, ty); df_add(azh, azl, tz); df_add(ph_, pl, tp_);
  const int64_t ci = A.tp.idx[fa + t];
  A.a[3 * ci + 0] = (double)axh + (double)axl;
  A.a[3 * ci + 1] = (double)ayh + (double)ayl;
  A.a[3 * ci + 2] = (double)azh + (double)azl;
  if (A.phi) A.phi[ci] = (double)ph_ + (double)pl;
  }
}

constexpr int kStage64 = 192;      // staged sources per warp and chunk (float64 path; at most 256)
constexpr int kQueue64 = 512;      // kernel pairs queued per warp
constexpr int kP2P64Warps = 4;

// One side of the symmetrised M4 pair in float64, added to f (force over
// distance) and p (potential): the polynomials of m4_side, for q < 1 in v = q and
// else in v = 2 - q (0 outside the support), as one evaluation
//   f += (A + w (B + v (C + v D))) h^-3 or r^-3,   w = q^2 or t^4,
// whose constants are selected (integer instructions): 13 float64 operations,
// where a warp whose lanes take both branches runs 20.
__device__ __forceinline__ void m4_side64(double r, double inv, double inv3, double hinv, double h3inv,
                                          double& f, double& p) {
  const double q = r * hinv;
  const bool in = __double2hiint(q) < 0x3ff00000;            // q < 1 (q >= 0)
  const double t = 2.0 - q;
  const double tp = __double2hiint(t) < 0 ? 0.0 : t;
  const double v = in ? q : tp, v2 = v * v, v4 = v2 * v2, w = in ? v2 : v4;
  const double f1 = fma(v, fma(v, in ? 0.0 : -1.0 / 6.0, in ? 0.5 : 0.8), in ? -1.2 : -1.0);
  f = fma(fma(w, f1, in ? 4.0 / 3.0 : 1.0), in ? h3inv : inv3, f);
  const double p1 = fma(v, fma(v, fma(v, in ? -0.1 : 0.0, in ? 0.3 : 1.0 / 30.0), in ? 0.0 : -0.1),
                        in ? -2.0 / 3.0 : 0.0);
  p = fma(fma(w, p1, in ? 1.4 : 1.0), in ? hinv : inv, p);
}

// Float64 mode: lanes = (target, source slice) as K = 32 / n_t slices;
// per chunk of near leaves (at most kStage64 sources) the warp stages the
// sources' float64 positions and masses in shared memory (M4: 1/h, and (2h)^2
// as float32), then every lane sums its slice; the target's own leaf is staged
// by itself (j != i).  The slices are added in slice order.
//
// Bound by the float64 pipe, where an operation costs as much as ~75 float32
// ones: a 1/r^2 pair takes 17 of them (3 differences, 3 for r^2, 4 for 1/r
// (rsqrt64), 4 for m/r and m/r^3, 3 for the force), the tests of the kernel
// supports are float32.  With the library's rsqrt, float64 tests and divisions
// per kernel pair it was ~45 (M4 binary of 2 x 2^20: 133 ms, now 74; Plummer
// sphere of 4096: 1.42 ms in long segments, now 0.23).
template <int SOFT, bool GROUPS>
__global__ void __launch_bounds__(kP2P64Warps * 32, SOFT == KDFMM_SOFT_PLUMMER && !GROUPS ? 8 : 1)
k_p2p_fp64(P2PArgs A) {
  constexpr bool M4 = SOFT == KDFMM_SOFT_M4;
  __shared__ double s_x[kP2P64Warps][kStage64], s_y[kP2P64Warps][kStage64];
  __shared__ double s_z[kP2P64Warps][kStage64], s_m[kP2P64Warps][kStage64];
  __shared__ double s_hinv[M4 ? kP2P64Warps : 1][M4 ? kStage64 : 1];
  __shared__ float s_h2[M4 ? kP2P64Warps : 1][M4 ? kStage64 : 1];
  __shared__ uint8_t s_leaf[kP2P64Warps][kStage64];
  __shared__ int s_tbeg[kP2P64Warps][32], s_tfirst[kP2P64Warps][32];
  constexpr int kW4 = M4 ? kP2P64Warps : 1;
  __shared__ uint16_t s_queue[kW4][M4 ? kQueue64 : 1];    // kernel pairs: owner lane << 8 | source
  __shared__ double s_term[kW4][4][M4 ? 32 : 1];
  __shared__ unsigned s_own[kW4][M4 ? 32 : 1];            // a lane's entries of the batch
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned full = 0xffffffffu;
  const int nleaves = min(A.counters[C_LEAVES], A.max_leaves);
  const int nitems = nleaves + (int)min((int64_t)A.counters[C_SEGS], A.seg_cap);
  double *sx = s_x[warp], *sy = s_y[warp], *sz = s_z[warp], *sm = s_m[warp];
  double* shinv = s_hinv[M4 ? warp : 0];
  float* sh2 = s_h2[M4 ? warp : 0];
  uint8_t* sl_of = s_leaf[warp];
  int* tb = s_tbeg[warp];
  int* tf = s_tfirst[warp];
  for (int item = blockIdx.x * kP2P64Warps + warp; item < nitems; item += gridDim.x * kP2P64Warps) {
  const bool seg = item >= nleaves;
  const int g = item - nleaves;
  const int k = seg ? A.seg_leaf[g] : item;
  if (k < 0) continue;
  const int a = A.leaf_cells[k];
  const int fa = A.cfirst[a], nt = A.ccount[a];
  const int K = 32 / nt;
  const int t = lane % nt, sl = lane / nt;
  const bool act = sl < K;
  const int64_t it = (int64_t)fa + t;
  const double xi = A.tp.x[it], yi = A.tp.y[it], zi = A.tp.z[it];
  const double hinv_i = M4 ? 1.0 / A.tp.h[it] : 0.0;
  const double h3inv_i = hinv_i * hinv_i * hinv_i;
  const float h2i = M4 ? A.ph[it].w : 0.0f;
  const double eps = A.sys_eps[A.leaf_sys[k]];
  const double soft2 = M4 ? 0.0 : eps * eps;      // added to r^2
  double fx = 0.0, fy = 0.0, fz = 0.0, fp = 0.0;
  auto stage = [&](int at, int64_t src) {
    sx[at] = A.tp.x[src];
    sy[at] = A.tp.y[src];
    sz[at] = A.tp.z[src];
    sm[at] = A.tp.m[src];
    if (M4) {
      shinv[at] = 1.0 / A.tp.h[src];
      sh2[at] = A.ph[src].w;
    }
  };
  // the lane's slice of the staged sources but `skip`: pairs outside both
  // supports as 1/r^2.  M4: those that may lie inside are queued by source
  // (ballots), and the warp takes 32 of them at a time, whatever lanes they
  // belong to: the pair's target comes by shuffle, its terms go back through
  // shared memory, each lane adding its own in queue order.  Left to their own
  // lanes the kernel pairs (a twentieth of all) kept a warp busy for as long as
  // its unluckiest lane and took 40 % of the kernel.
  auto kernel_pairs = [&](int nq) {
    __syncwarp();
    for (int i0 = 0; i0 < nq; i0 += 32) {
      const bool v = i0 + lane < nq;
      const int e = v ? s_queue[warp][i0 + lane] : 0, o = e >> 8, j = e & 255;
      const double tx = __shfl_sync(full, xi, o), ty = __shfl_sync(full, yi, o),
                   tz = __shfl_sync(full, zi, o);
      const double hi = __shfl_sync(full, hinv_i, o), h3i = __shfl_sync(full, h3inv_i, o);
      s_own[warp][lane] = 0u;
      const unsigned mine = __match_any_sync(full, v ? o : 32);
      __syncwarp();
      if (v) {
        if ((mine & ((1u << lane) - 1u)) == 0u) s_own[warp][o] = mine;
        const double rx = tx - sx[j], ry = ty - sy[j], rz = tz - sz[j];
        const double r2 = fma(rz, rz, fma(ry, ry, fma(rx, rx, soft2)));
        const double inv = rsqrt64(r2), r = far_sqrt(r2, inv), inv3 = inv * inv * inv;
        const double hj = shinv[j], mh = 0.5 * sm[j];
        double f = 0.0, p = 0.0;
        m4_side64(r, inv, inv3, hi, h3i, f, p);
        m4_side64(r, inv, inv3, hj, hj * hj * hj, f, p);
        f = r2 > 0.0 ? f * mh : 0.0;               // coincident: no force, whatever h^-3 is
        s_term[warp][0][lane] = f * rx;
        s_term[warp][1][lane] = f * ry;
        s_term[warp][2][lane] = f * rz;
        s_term[warp][3][lane] = mh * p;
      }
      __syncwarp();
      for (unsigned m = s_own[warp][lane]; m != 0u; m &= m - 1u) {
        const int k2 = __ffs(m) - 1;
        fx -= s_term[warp][0][k2];
        fy -= s_term[warp][1][k2];
        fz -= s_term[warp][2][k2];
        fp -= s_term[warp][3][k2];
      }
      __syncwarp();
    }
  };
  auto sum_staged = [&](int total, int skip) {
    int nq = 0;
    for (int j0 = 0; j0 < total; j0 += K) {
      const int j = j0 + sl;
      bool in = false;
      if (act && j < total && j != skip) {
        const double rx = xi - sx[j], ry = yi - sy[j], rz = zi - sz[j];
        const double r2 = fma(rz, rz, fma(ry, ry, fma(rx, rx, soft2)));
        in = M4 && maybe_inside(r2, h2i, sh2[j]);
        if (!in) {
          const double inv = rsqrt64(r2);
          const double minv = sm[j] * inv, f = minv * (inv * inv);
          fx = fma(-f, rx, fx); fy = fma(-f, ry, fy); fz = fma(-f, rz, fz);
          fp -= minv;
        }
      }
      if constexpr (M4) {
        const unsigned marks = __ballot_sync(full, in);
        if (marks != 0u) {
          if (in) s_queue[warp][nq + __popc(marks & ((1u << lane) - 1u))] = (uint16_t)(lane << 8 | j);
          nq += __popc(marks);
          if (nq > kQueue64 - 32) {
            kernel_pairs(nq);
            nq = 0;
          }
        }
      }
    }
    if constexpr (M4) {
      if (nq > 0) kernel_pairs(nq);
    }
  };
  const int64_t nall = min((int64_t)A.near_cnt[k], A.cap_near);
  const int seglen = leaf_segment(A.sys_off, A.leaf_sys[k]);
  const int64_t sidx = seg ? (int64_t)(g - A.seg_first[k] + 1) : 0;
  const int64_t entries = item_entries(GROUPS, seglen);
  const int64_t e_end = A.near_off[k] + min(nall, (sidx + 1) * entries);
  double bx = 0.0, by = 0.0, bz = 0.0, bp = 0.0;      // GROUPS, slice 0: sums of the leaf's first
  double rx = 0.0, ry = 0.0, rz = 0.0, rp = 0.0;      // segment, and of the item's others
  bool lead = !seg;
  int64_t e = A.near_off[k] + sidx * entries;
  do {
    if (lead) {
      if (lane < nt) stage(lane, (int64_t)fa + lane);
      __syncwarp();
      sum_staged(nt, t);
      __syncwarp();
    }
    const int64_t e1 = min(e + seglen, e_end);
    while (e < e1) {
      const int64_t my = e + lane;
      int cnt = 0, first = 0;
      if (my < e1) {
        const int b = A.near_idx[my];
        if (b != a) {
          cnt = A.ccount[b];
          first = A.cfirst[b];
        }
      }
      int incl = cnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int w = __shfl_up_sync(full, incl, o);
        if (lane >= o) incl += w;
      }
      const int L = __popc(__ballot_sync(full, my < e1 && incl <= kStage64));
      if (lane < L) {
        const int beg = incl - cnt;
        tb[lane] = beg;
        tf[lane] = first;
        for (int q = 0; q < cnt; ++q) sl_of[beg + q] = (uint8_t)lane;
      }
      __syncwarp();
      const int total = __shfl_sync(full, incl, L - 1);
      for (int idx = lane; idx < total; idx += 32) {
        const int l = sl_of[idx];
        stage(idx, (int64_t)tf[l] + idx - tb[l]);
      }
      __syncwarp();
      sum_staged(total, -1);
      __syncwarp();
      e += L;
    }
    // the segment's slices, in slice order
    for (int s = 1; s < K; ++s) {
      const int src = t + s * nt;
      const double ox = __shfl_sync(full, fx, src), oy = __shfl_sync(full, fy, src);
      const double oz = __shfl_sync(full, fz, src), op = __shfl_sync(full, fp, src);
      if (sl == 0) { fx += ox; fy += oy; fz += oz; fp += op; }
    }
    if constexpr (GROUPS) {
      if (lead) { bx = fx; by = fy; bz = fz; bp = fp; }
      else { rx += fx; ry += fy; rz += fz; rp += fp; }
      fx = fy = fz = fp = 0.0;
      lead = false;
    }
  } while (GROUPS && e < e_end);
  if constexpr (!GROUPS) {                            // one segment an item
    if (seg) { rx = fx; ry = fy; rz = fz; rp = fp; }
    else { bx = fx; by = fy; bz = fz; bp = fp; }
  }
  if (sl != 0 || !act) continue;
  if (seg) {
    double* P = A.seg_part + (int64_t)g * 128 + 4 * t;
    P[0] = rx; P[1] = ry; P[2] = rz; P[3] = rp;
    continue;
  }
  const double* C = A.lexp64 + 20 * (int64_t)k;
  const double x = xi - A.cx[a], y = yi - A.cy[a], z = zi - A.cz[a];
  double tx, ty, tz, tp_;
  l2p_tail<double>(C, x, y, z, tx, ty, tz, tp_);
  const int64_t ci = A.tp.idx[it];
  A.a[3 * ci + 0] = (bx + (tx - C[1])) + rx;
  A.a[3 * ci + 1] = (by + (ty - C[2])) + ry;
  A.a[3 * ci + 2] = (bz + (tz - C[3])) + rz;
  if (A.phi) A.phi[ci] = (bp + (C[0] + tp_)) + rp;
  }
}

// Reserves the extra segments of every leaf (any order: a leaf's segments
// are contiguous and combined in segment order).  More than seg_cap flags
// ST_LISTS and drops the leaf's extra segments (the evaluation is redone);
// their entries below seg_cap are marked -1, which every consumer skips.
__global__ void k_seg_plan(const int32_t* __restrict__ near_cnt, int64_t cap_near,
                           int max_leaves, int32_t* counters, int32_t* seg_first,
                           int32_t* seg_leaf, int64_t seg_cap, const int64_t* __restrict__ sys_off,
                           const int32_t* __restrict__ leaf_sys, bool grouped, int32_t* status) {
  const int nleaves = min(counters[C_LEAVES], max_leaves);
  KD_GRID_STRIDE(k, nleaves) {
    const int x = extra_segments(min((int64_t)near_cnt[k], cap_near),
                                 item_entries(grouped, leaf_segment(sys_off, leaf_sys[k])));
    int first = -1;
    if (x > 0) {
      const int base = atomicAdd(&counters[C_SEGS], x);
      if ((int64_t)base + x <= seg_cap) {
        first = base;
        for (int q = 0; q < x; ++q) seg_leaf[base + q] = k;
      } else {
        atomicOr(status, ST_LISTS);
        for (int q = 0; q < x && (int64_t)base + q < seg_cap; ++q) seg_leaf[base + q] = -1;
      }
    }
    seg_first[k] = first;
  }
}

// Adds the extra items' partial sums to a and phi (caller order): the rest of
// the first group, then the other groups' sums.  Warp per leaf (the warp of its
// first extra item), lane per target.
__global__ void k_seg_combine(P2PArgs A) {
  const int lane = threadIdx.x & 31;
  const int nseg = (int)min((int64_t)A.counters[C_SEGS], A.seg_cap);
  for (int g = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); g < nseg;
       g += (int)((gridDim.x * blockDim.x) >> 5)) {
    const int k = A.seg_leaf[g];
    if (k < 0) continue;
    const int f = A.seg_first[k];
    if (g != f) continue;
    const int a = A.leaf_cells[k];
    if (lane >= A.ccount[a]) continue;
    const int entries = item_entries(A.grouped, leaf_segment(A.sys_off, A.leaf_sys[k]));
    const int x = extra_segments(min((int64_t)A.near_cnt[k], A.cap_near), entries);
    const int group = kSegEntries / entries;              // items of a group (a power of two)
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;        // of the group
    double r0 = 0.0, r1 = 0.0, r2 = 0.0, r3 = 0.0;        // of the first group
    double t0 = 0.0, t1 = 0.0, t2 = 0.0, t3 = 0.0;        // of the others
    // (a heavy leaf has hundreds of items: eight pieces' loads in flight)
#pragma unroll 8
    for (int q = 1; q <= x; ++q) {
      const double2* P = reinterpret_cast<const double2*>(A.seg_part + (int64_t)(f + q - 1) * 128 + 4 * lane);
      const double2 p01 = P[0], p23 = P[1];
      if ((q & (group - 1)) == 0) {
        if (q == group) { r0 = s0; r1 = s1; r2 = s2; r3 = s3; }
        else { t0 += s0; t1 += s1; t2 += s2; t3 += s3; }
        s0 = s1 = s2 = s3 = 0.0;
      }
      s0 += p01.x; s1 += p01.y; s2 += p23.x; s3 += p23.y;
    }
    if (x < group) { r0 = s0; r1 = s1; r2 = s2; r3 = s3; }
    else { t0 += s0; t1 += s1; t2 += s2; t3 += s3; }
    const int64_t ci = A.tp.idx[A.cfirst[a] + lane];
    A.a[3 * ci + 0] = (A.a[3 * ci + 0] + r0) + t0;
    A.a[3 * ci + 1] = (A.a[3 * ci + 1] + r1) + t1;
    A.a[3 * ci + 2] = (A.a[3 * ci + 2] + r2) + t2;
    if (A.phi) A.phi[ci] = (A.phi[ci] + r3) + t3;
  }
}

inline unsigned blocks_for(int64_t n, int threads) { return (unsigned)((n + threads - 1) / threads); }

}  // namespace

// Near entries of the last walk (exact lists: those allocated).
static int64_t near_entries(const kdfmm_tree_s* t) {
  return t->L.exact ? t->L.near_cap : t->host_stats[KDFMM_STAT_NNEAR];
}

// At most so many extra items if each segment is one: of each length class the
// entries of its systems (no more than all, no more than their particles
// squared) over the length.  *shorter: those of short segments.
static int64_t segment_items(const kdfmm_tree_s* t, int64_t* shorter) {
  const int64_t entries = near_entries(t);
  *shorter = 0;
  if (t->p.precision != KDFMM_FP64) return entries / kSegEntries + 64;
  double own[kSegSteps + 1] = {};
  for (int k = 0; k < t->n_sys; ++k) {
    const double n = (double)(t->host_sys_off[k + 1] - t->host_sys_off[k]);
    own[seg_step((int64_t)n)] += n * n;
  }
  int64_t items = 64;
  for (int q = 0; q <= kSegSteps; ++q) {
    items += (int64_t)std::min((double)entries, own[q]) / seg_length(q);
    if (q < kSegSteps) *shorter = items;
  }
  return items;
}

// What the extra items of the evaluation are (L.seg_grouped), with room for them
// and, for later evaluations of other particles, `spare` of that more.
int ensure_segments(kdfmm_tree_s* t, double spare) {
  Lists& L = t->L;
  int64_t shorter;
  int64_t need = segment_items(t, &shorter);
  // (Mixed segments and those of one large system are of 256 entries by themselves.)
  L.seg_grouped = t->p.precision == KDFMM_FP64 &&
                  ((t->n_sys > 1 && t->n >= kFullCall) || shorter > kShortItems);
  if (L.seg_grouped) need = near_entries(t) / kSegEntries + 64;
  need += (int64_t)(spare * (double)need);
  if (L.seg_cap >= need && L.seg_leaf != nullptr) return KDFMM_OK;
  const int64_t cap = std::max<int64_t>(need, 64);
  int32_t* leaf = nullptr;
  double* part = nullptr;
  if (cudaMalloc(&leaf, (size_t)cap * sizeof(int32_t)) != cudaSuccess ||
      cudaMalloc(&part, (size_t)cap * 128 * sizeof(double)) != cudaSuccess) {
    cudaFree(leaf);
    cudaGetLastError();
    return set_error(KDFMM_ERR_OOM, "P2P segments (%lld)", (long long)cap);
  }
  cudaFree(L.seg_leaf);
  cudaFree(L.seg_part);
  L.seg_leaf = leaf;
  L.seg_part = part;
  L.seg_cap = cap;
  return KDFMM_OK;
}

int plan_segments(kdfmm_tree_s* t, cudaStream_t s) {
  const int gl = std::max(t->grid_leaves, 1);
  cudaMemsetAsync(t->counters + C_SEGS, 0, sizeof(int32_t), s);
  k_seg_plan<<<std::min<unsigned>(blocks_for(gl, 256), grid_blocks()), 256, 0, s>>>(
      t->L.near_cnt, t->L.exact ? INT64_MAX : t->L.cap_near, gl, t->counters, t->L.seg_first,
      t->L.seg_leaf, t->L.seg_cap, t->p.precision == KDFMM_FP64 ? t->sys_off : nullptr, t->leaf_sys,
      t->L.seg_grouped, t->status);
  t->launches += 1;
  return check_cuda(cudaGetLastError(), "segment plan");
}

int run_p2p(kdfmm_tree_s* t, double* a, double* phi, cudaStream_t s) {
  P2PArgs A{};
  A.leaf_cells = t->leaf_cells;
  A.counters = t->counters;
  A.cap_near = t->L.exact ? INT64_MAX : t->L.cap_near;
  A.max_leaves = std::max(t->grid_leaves, 1);
  A.cfirst = t->c.first;
  A.ccount = t->c.count;
  A.near_cnt = t->L.near_cnt;
  A.near_off = t->L.near_off;
  A.near_idx = t->L.near_idx;
  A.src32 = t->c.src32;
  A.pf = t->pf;
  A.ph = t->ph;
  A.tp = t->tp;
  A.cx = t->c.cx; A.cy = t->c.cy; A.cz = t->c.cz;
  A.lexp32 = t->lexp32;
  A.lexp64 = t->lexp64;
  A.walk = t->c.walk;
  A.walk2 = t->c.walk2;
  A.leaf_sys = t->leaf_sys;
  A.sys_eps = t->sys_eps;
  A.a = a;
  A.phi = phi;
  A.seg_first = t->L.seg_first;
  A.seg_leaf = t->L.seg_leaf;
  A.seg_part = t->L.seg_part;
  A.seg_cap = t->L.seg_cap;
  int rc = plan_segments(t, s);
  if (rc) return rc;
  A.sys_off = t->p.precision == KDFMM_FP64 ? t->sys_off : nullptr;
  A.grouped = t->L.seg_grouped;
  const int gl = std::max(t->grid_leaves, 1);
  const bool m4 = t->p.soft_kind == KDFMM_SOFT_M4;
  if (t->p.precision == KDFMM_MIXED) {
    const unsigned gm = blocks_for(gl, kP2PWarps);
    if (m4) k_p2p_mixed<KDFMM_SOFT_M4><<<gm, kP2PWarps * 32, 0, s>>>(A);
    else k_p2p_mixed<KDFMM_SOFT_PLUMMER><<<gm, kP2PWarps * 32, 0, s>>>(A);
  } else {
    // a warp per leaf and per segment that there may be
    const unsigned g64 = blocks_for(gl + t->L.seg_cap, kP2P64Warps);
    if (A.grouped) {
      if (m4) k_p2p_fp64<KDFMM_SOFT_M4, true><<<g64, kP2P64Warps * 32, 0, s>>>(A);
      else k_p2p_fp64<KDFMM_SOFT_PLUMMER, true><<<g64, kP2P64Warps * 32, 0, s>>>(A);
    } else {
      if (m4) k_p2p_fp64<KDFMM_SOFT_M4, false><<<g64, kP2P64Warps * 32, 0, s>>>(A);
      else k_p2p_fp64<KDFMM_SOFT_PLUMMER, false><<<g64, kP2P64Warps * 32, 0, s>>>(A);
    }
  }
  k_seg_combine<<<grid_blocks(2), 256, 0, s>>>(A);
  t->launches += 2;
  return check_cuda(cudaGetLastError(), "p2p launch");
}

}  // namespace kdfmm
