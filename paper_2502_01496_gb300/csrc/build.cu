// kd-tree construction and cell moments (Sec. 2; Eq. 7).
//
// Each cell is cut through its centre of mass across the longest side of its
// bounding box; a cell with more than n_leaf particles is split.  The centre
// of mass is the pairwise (perfect binary tree) sum of m and m x over the
// cell's particles in ascending caller index, zero-padded to a power of two,
// divided by the pairwise sum of m -- every float64 operation that decides a
// cut is correctly rounded and uncontracted, so the tree is reproducible bit
// for bit on any device and on the host.
//
// Phase A: cells larger than kSubtreeMax are split level by level in global
//          memory, each cell tiled into chunks of 2048 (or 512) elements aligned
//          to the cell's first particle (chunk sums are the subtrees of the pairwise
//          tree, so the tiling does not change the result).
// Phase B: a cell of at most kSubtreeMax particles is finished by one CTA with
//          its particles held in shared memory, all cells of a level together.
// Then the cells are renumbered in pre-order from their particle ranges, the
// quadrupoles and h_max are accumulated bottom-up, and float32 views for the
// walk, the M2L and the P2P are derived.
#include <algorithm>
#include <climits>
#include <type_traits>

#include "kdfmm_internal.cuh"

namespace kdfmm {

namespace {

struct BuildArgs {
  TmpCells tmp;
  int32_t* counters;
  int32_t* status;
  const int64_t* sys_off;          // forest: particle offsets of the systems
  const int32_t* sys_nleaf;        // forest: leaf size of each system
  int32_t n_sys;
  int64_t capA, capB, capL, cap_cells;
};

__device__ __forceinline__ int nleaf_at(const BuildArgs& A, int64_t first) {
  return A.sys_nleaf[system_of(A.sys_off, A.n_sys, first)];
}

__device__ __forceinline__ double coord(const PCols& p, int axis, int64_t i) {
  return axis == 0 ? p.x[i] : (axis == 1 ? p.y[i] : p.z[i]);
}

__device__ __forceinline__ void set_status(int32_t* status, int bits) { atomicOr(status, bits); }

// ---------------------------------------------------------------------------
// initial gather: caller order -> SoA buffer 0, with validation
// ---------------------------------------------------------------------------
__global__ void k_init(const double* __restrict__ x, const double* __restrict__ m,
                       const double* __restrict__ h, int64_t n, const int64_t* __restrict__ sys_off,
                       int n_sys, const double* __restrict__ sys_eps, int soft_kind, PCols b,
                       int32_t* status) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double xi = x[3 * i], yi = x[3 * i + 1], zi = x[3 * i + 2], mi = m[i];
  double hi = (h != nullptr && soft_kind == KDFMM_SOFT_M4) ? h[i]
                                                           : sys_eps[system_of(sys_off, n_sys, i)];
  bool ok = isfinite(xi) && isfinite(yi) && isfinite(zi) && isfinite(mi) && isfinite(hi) &&
            mi > 0.0 && (soft_kind == KDFMM_SOFT_M4 ? hi > 0.0 : hi >= 0.0);
  if (!ok) set_status(status, ST_NONFINITE);
  b.x[i] = xi; b.y[i] = yi; b.z[i] = zi; b.m[i] = mi;      // (h joins at the leaves)
  b.idx[i] = (int32_t)i;
}

// One root segment per system (build-order cell k for system k).
__global__ void k_roots(BuildArgs A, Seg* segA, Seg* segB, Seg* segL) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k == 0) atomicAdd(&A.counters[0], A.n_sys);
  if (k >= A.n_sys) return;
  const int64_t f = A.sys_off[k], cnt = A.sys_off[k + 1] - f;
  const Seg g{(int32_t)f, (int32_t)cnt, k, 0};
  if (cnt > kSubtreeMax) {
    const int i = atomicAdd(&A.counters[1], 1);
    if (i < A.capA) segA[i] = g; else set_status(A.status, ST_CAPACITY);
  } else if (cnt > A.sys_nleaf[k]) {
    const int i = atomicAdd(&A.counters[2], 1);
    if (i < A.capB) segB[i] = g; else set_status(A.status, ST_CAPACITY);
  } else {
    const int i = atomicAdd(&A.counters[3], 1);
    if (i < A.capL) segL[i] = g; else set_status(A.status, ST_CAPACITY);
  }
}

// Pushes a new segment onto the list that will process it.
__device__ void push_child(const BuildArgs& A, Seg c, Seg* nextA, Seg* segB, Seg* segL) {
  if (c.count > kSubtreeMax) {
    int k = atomicAdd(&A.counters[1], 1);
    if (k < A.capA) nextA[k] = c; else set_status(A.status, ST_CAPACITY);
  } else if (c.count > nleaf_at(A, c.first)) {
    int k = atomicAdd(&A.counters[2], 1);
    if (k < A.capB) segB[k] = c; else set_status(A.status, ST_CAPACITY);
  } else {
    int k = atomicAdd(&A.counters[3], 1);
    if (k < A.capL) segL[k] = c; else set_status(A.status, ST_CAPACITY);
  }
}

// ---------------------------------------------------------------------------
// phase A: four launches a level.  The chunk kernels run one block per chunk;
// the last block of a segment to finish (a counter per segment) goes on with
// the segment's own step -- the cut after the sums, the split after the counts --
// on all its threads, instead of a launch of one warp per segment (a top cell
// of 2^24 particles has 8192 chunks).  T threads make chunks of 8 T elements:
// 64 while large chunks would not reach every SM (small evaluations wait on the
// float64 pipes of the few SMs that hold a chunk), else 256.  Eight launches a
// level before: 2^24 clumped particles, all levels, 7.2 ms for the sums, cuts, counts,
// splits and maps, now 6.3; a 60013-particle sphere, with the scatter, 0.43 ms, now
// 0.29.
// ---------------------------------------------------------------------------
template <int T>
__device__ __forceinline__ int nchunks_of(int count) { return (count + 8 * T - 1) / (8 * T); }

// After the last phase-A level: segments still waiting for a split mean the
// fixed number of levels was too small.
__global__ void k_levels_done(const int32_t* counters, int32_t* status) {
  if (counters[C_NEXT_A] > 0) set_status(status, ST_UNFINISHED);
}

// Start of a phase-A level (single block): the segments pushed by the previous
// level are this level's (counters[C_NA]), the push counter restarts; chunk
// offsets of the segments, the chunk -> segment map, the segments' counters.
template <int T>
__global__ void k_level_map(const Seg* __restrict__ segs, int32_t* __restrict__ seg_off,
                            int32_t* __restrict__ chunk_seg, int32_t* __restrict__ seg_done,
                            int32_t* counters, int64_t capA, int32_t* status) {
  __shared__ int32_t warp_tot[32];
  __shared__ int32_t carry;
  int nA = counters[C_NEXT_A];
  if (nA > capA) {
    set_status(status, ST_CAPACITY);
    nA = (int)capA;
  }
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  if (threadIdx.x == 0) {
    counters[C_NA] = nA;
    counters[C_NEXT_A] = 0;
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int base = 0; base < nA; base += blockDim.x) {
    int s = base + threadIdx.x;
    int e = s < nA ? nchunks_of<T>(segs[s].count) : 0;
    int incl = e;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    if (lane == 31) warp_tot[w] = incl;
    __syncthreads();
    if (w == 0) {
      int t = lane < (int)(blockDim.x >> 5) ? warp_tot[lane] : 0;
      int ti = t;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        int v = __shfl_up_sync(0xffffffffu, ti, o);
        if (lane >= o) ti += v;
      }
      warp_tot[lane] = ti - t;
    }
    __syncthreads();
    int excl = carry + warp_tot[w] + incl - e;
    __syncthreads();
    if (s < nA) {
      seg_off[s] = excl;
      seg_done[2 * s] = seg_done[2 * s + 1] = 0;
    }
    if (threadIdx.x == blockDim.x - 1) carry = excl + e;
    // the map: a long segment's chunks by the whole block, the others' by their threads
    if (s < nA && e <= 32)
      for (int c = 0; c < e; ++c) chunk_seg[excl + c] = s;
    unsigned big = __ballot_sync(0xffffffffu, e > 32);
    while (big != 0u) {
      const int l = __ffs(big) - 1;
      big &= big - 1u;
      const int be = __shfl_sync(0xffffffffu, e, l), bx = __shfl_sync(0xffffffffu, excl, l),
                bs = __shfl_sync(0xffffffffu, s, l);
      for (int c = lane; c < be; c += 32) chunk_seg[bx + c] = bs;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) counters[C_CHUNKS] = carry;
}

// True in every thread of the last of `of` blocks to come here (what the
// others wrote before is visible then).
__device__ __forceinline__ bool last_block(int32_t* counter, int of) {
  __shared__ int s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(counter, 1) == of - 1;
  __syncthreads();
  if (!s_last) return false;
  __threadfence();
  return true;
}

// Chunk partial sums (pairwise subtree of 8 T elements) and bounding box keys;
// then, once per segment, the pairwise tree over its chunk sums, centre of
// mass, axis, cut.
template <int T>
__global__ void __launch_bounds__(T)
k_chunk_reduce(const Seg* __restrict__ segs, const int32_t* __restrict__ chunk_seg,
               const int32_t* __restrict__ seg_off, const int32_t* __restrict__ counters,
               PCols p, double* csum, long long* ckey, int32_t* seg_done, TmpCells tmp,
               int32_t* __restrict__ seg_axis, double* __restrict__ seg_cut, float* __restrict__ seg_xb) {
  constexpr int kW = T / 32;
  const int b = blockIdx.x;
  if (b >= counters[C_CHUNKS]) return;
  const int s = chunk_seg[b];
  const Seg g = segs[s];
  const int off = seg_off[s];
  const int rel0 = (b - off) * 8 * T;
  const int cnt = g.count - rel0;               // valid elements from the chunk start
  const int64_t base = (int64_t)g.first + rel0;
  __shared__ double ws[kW][4];
  __shared__ long long wk[kW][6];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  // block sums and boxes: the perfect tree over the lanes as a reduce-scatter
  // (two components, then one: 6 float64 additions a warp instead of 20, same
  // bits: the pairs are those of the butterfly), then the tree over the warps.
  // lane 0 .. 3 of warp 0 end with components m, y, x, z of the total, thread 0
  // with the keys.
  auto block_reduce = [&](const Sum4& v, long long lo[3], long long hi[3], double& total, long long key[6]) {
    const unsigned full = 0xffffffffu;
    const bool odd = lane & 1, second = lane & 2;
    const double a0 = (odd ? v.y : v.m) + __shfl_xor_sync(full, odd ? v.m : v.y, 1);
    const double a1 = (odd ? v.z : v.x) + __shfl_xor_sync(full, odd ? v.x : v.z, 1);
    double s = (second ? a1 : a0) + __shfl_xor_sync(full, second ? a0 : a1, 2);
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) s = __dadd_rn(s, __shfl_xor_sync(full, s, o));
#pragma unroll
    for (int d = 0; d < 3; ++d) { lo[d] = warp_min_ll(lo[d]); hi[d] = warp_max_ll(hi[d]); }
    __syncthreads();
    if (lane < 4) ws[w][lane] = s;
    if (lane == 0)
      for (int d = 0; d < 3; ++d) { wk[w][d] = lo[d]; wk[w][3 + d] = hi[d]; }
    __syncthreads();
    if (threadIdx.x >= 4) return;
    double t4[kW];
#pragma unroll
    for (int q = 0; q < kW; ++q) t4[q] = ws[q][lane];
#pragma unroll
    for (int width = kW; width > 1; width >>= 1)
#pragma unroll
      for (int q = 0; q < width / 2; ++q) t4[q] = __dadd_rn(t4[2 * q], t4[2 * q + 1]);
    total = t4[0];
    if (threadIdx.x != 0) return;
    for (int d = 0; d < 6; ++d) {
      long long r = wk[0][d];
      for (int q = 1; q < kW; ++q) r = d < 3 ? min(r, wk[q][d]) : max(r, wk[q][d]);
      key[d] = r;
    }
  };
  {
    // the bounding-box keys come with the same loads (get runs once per element)
    long long lo[3] = {LLONG_MAX, LLONG_MAX, LLONG_MAX}, hi[3] = {LLONG_MIN, LLONG_MIN, LLONG_MIN};
    auto get = [&](int k) {
      int64_t i = base + k;
      const double x = p.x[i], y = p.y[i], z = p.z[i];
      const long long kx = dkey(x), ky = dkey(y), kz = dkey(z);
      lo[0] = min(lo[0], kx); hi[0] = max(hi[0], kx);
      lo[1] = min(lo[1], ky); hi[1] = max(hi[1], ky);
      lo[2] = min(lo[2], kz); hi[2] = max(hi[2], kz);
      return elem4(p.m[i], x, y, z);
    };
    const Sum4 v = block_tree<3>(8 * threadIdx.x, cnt, get);
    double t;
    long long key[6];
    block_reduce(v, lo, hi, t, key);
    if (threadIdx.x < 4) csum[4 * (int64_t)b + ((lane & 1) << 1 | lane >> 1)] = t;
    if (threadIdx.x == 0)
      for (int d = 0; d < 6; ++d) ckey[6 * (int64_t)b + d] = key[d];
  }
  const int C = nchunks_of<T>(g.count);
  if (!last_block(&seg_done[2 * s], C)) return;
  // the segment: thread t sums its aligned block of B chunks (carry stack)
  int P = 1;
  while (P < C) P <<= 1;
  const int B = P > T ? P / T : 1;
  auto chunk = [&](int c) {
    if (c >= C) return zero4();
    const double* q = csum + 4 * (int64_t)(off + c);
    return Sum4{__ldcg(q), __ldcg(q + 1), __ldcg(q + 2), __ldcg(q + 3)};
  };
  Sum4 v;
  if (B == 1) {
    v = chunk(threadIdx.x);
  } else {
    Sum4 st[16];
    int top = 0;
    for (int k = 0; k < B; ++k) {
      Sum4 e = chunk(threadIdx.x * B + k);
      for (int kk = k; kk & 1; kk >>= 1) e = add4(st[--top], e);
      st[top++] = e;
    }
    v = st[0];
  }
  long long lo[3] = {LLONG_MAX, LLONG_MAX, LLONG_MAX}, hi[3] = {LLONG_MIN, LLONG_MIN, LLONG_MIN};
  for (int c = threadIdx.x; c < C; c += T)
    for (int d = 0; d < 3; ++d) {
      lo[d] = min(lo[d], __ldcg(&ckey[6 * (int64_t)(off + c) + d]));
      hi[d] = max(hi[d], __ldcg(&ckey[6 * (int64_t)(off + c) + 3 + d]));
    }
  double t = 0.0;
  long long key[6] = {0, 0, 0, 0, 0, 0};
  block_reduce(v, lo, hi, t, key);
  if (w != 0) return;
  // the three divisions run once, on lanes 0, 1, 2
  const double M = __shfl_sync(0xffffffffu, t, 0);
  const double sx = __shfl_sync(0xffffffffu, t, 2), sy = __shfl_sync(0xffffffffu, t, 1),
               sz = __shfl_sync(0xffffffffu, t, 3);
  const double quo = __ddiv_rn(lane == 1 ? sy : (lane == 2 ? sz : sx), M);
  const double cx = __shfl_sync(0xffffffffu, quo, 0), cy = __shfl_sync(0xffffffffu, quo, 1),
               cz = __shfl_sync(0xffffffffu, quo, 2);
  if (lane == 0) {
    double dlo[3], dhi[3];
    for (int d = 0; d < 3; ++d) {
      dlo[d] = dunkey(key[d]);
      dhi[d] = dunkey(key[3 + d]);
    }
    const int axis = longest_axis(dlo, dhi);
    const int c = g.cell;
    tmp.first[c] = g.first; tmp.count[c] = g.count; tmp.depth[c] = g.dbuf >> 1;
    tmp.M[c] = M; tmp.cx[c] = cx; tmp.cy[c] = cy; tmp.cz[c] = cz;
    tmp.s[c] = 0.0;
    seg_axis[s] = axis;
    seg_cut[s] = axis == 0 ? cx : (axis == 1 ? cy : cz);
    double X = 0.0;
    for (int d = 0; d < 3; ++d) X = fmax(X, fmax(fabs(dlo[d]), fabs(dhi[d])));
    seg_xb[s] = (float)X * 1.000001f;
  }
}

// Per chunk: particles left of the cut (one coordinate read).  Then, once per
// segment: offsets of the left particles per chunk, the split point and the two
// children.
template <int T>
__global__ void __launch_bounds__(T)
k_chunk_count(const Seg* __restrict__ segs, const int32_t* __restrict__ chunk_seg,
              const int32_t* __restrict__ seg_off, const int32_t* __restrict__ counters, PCols p,
              const int32_t* __restrict__ seg_axis, const double* __restrict__ seg_cut,
              int32_t* cleft, int32_t* seg_done, int32_t* __restrict__ cloff,
              int32_t* __restrict__ seg_nl, BuildArgs A, Seg* nextA, Seg* segB, Seg* segL, int dst_buf) {
  constexpr int kW = T / 32;
  const int b = blockIdx.x;
  if (b >= counters[C_CHUNKS]) return;
  const int s = chunk_seg[b];
  const Seg g = segs[s];
  const int off = seg_off[s];
  const int rel0 = (b - off) * 8 * T;
  const int cnt = min(8 * T, g.count - rel0);
  const int64_t base = (int64_t)g.first + rel0;
  const int axis = seg_axis[s];
  const double* const x = axis == 0 ? p.x : (axis == 1 ? p.y : p.z);
  const long long ckey = dkey(seg_cut[s]);
  int nl = 0;
#pragma unroll
  for (int pass = 0; pass < 8; ++pass) {   // all loads in flight
    const int k = pass * T + threadIdx.x;
    if (k < cnt) nl += dkey(x[base + k]) < ckey;
  }
  __shared__ int wn[kW];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  nl = __reduce_add_sync(0xffffffffu, nl);
  if (lane == 0) wn[w] = nl;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int q = 0; q < kW; ++q) t += wn[q];
    cleft[b] = t;
  }
  const int C = nchunks_of<T>(g.count);
  if (!last_block(&seg_done[2 * s + 1], C)) return;
  int run = 0;
  for (int c0 = 0; c0 < C; c0 += T) {
    const int c = c0 + threadIdx.x;
    const int v = c < C ? __ldcg(&cleft[off + c]) : 0;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int u = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += u;
    }
    __syncthreads();
    if (lane == 31) wn[w] = incl;
    __syncthreads();
    int before = 0, tot = 0;
#pragma unroll
    for (int q = 0; q < kW; ++q) {
      const int u = wn[q];
      before += q < w ? u : 0;
      tot += u;
    }
    if (c < C) cloff[off + c] = run + before + incl - v;
    run += tot;
  }
  if (threadIdx.x != 0) return;
  nl = run;
  const bool fallback = (nl == 0 || nl == g.count);
  if (fallback) {
    nl = g.count / 2;
    atomicAdd(&A.counters[C_FALLBACK], 1);
  }
  seg_nl[s] = fallback ? -nl - 1 : nl;
  const int c = g.cell;
  int cid = atomicAdd(&A.counters[C_CELLS], 2);
  if (cid + 2 > A.cap_cells) { set_status(A.status, ST_CAPACITY); return; }
  A.tmp.left[c] = cid;
  A.tmp.right[c] = cid + 1;
  const int depth = (g.dbuf >> 1) + 1;
  atomicMax(&A.counters[C_DEPTH], depth);
  push_child(A, Seg{g.first, nl, cid, depth << 1 | dst_buf}, nextA, segB, segL);
  push_child(A, Seg{g.first + nl, g.count - nl, cid + 1, depth << 1 | dst_buf}, nextA, segB, segL);
}

// Stable scatter of one chunk into the other buffer.  Element k of the chunk
// (pass k / T, thread k % T) goes to the left child at
// its rank among the segment's left elements, else to the right child.  The
// flags of all the chunk's elements are taken first (their coordinate loads in
// flight together), one block barrier publishes the passes' warp counts, and
// the moves follow with kMoveBatch elements' loads in flight per thread.  Pass
// by pass, with two barriers each, the kernel waited on one load at a time:
// this form took the benchmark's build 3.72 -> 3.56 ms (batches of 1, 2 or 4
// elements, rolled or unrolled, measured within 1 % of each other).
constexpr int kScatterPasses = 8;
template <int T>
__global__ void __launch_bounds__(T)
k_chunk_scatter(const Seg* __restrict__ segs, const int32_t* __restrict__ chunk_seg,
                const int32_t* __restrict__ seg_off, const int32_t* __restrict__ counters, PCols src,
                PCols dst, const int32_t* __restrict__ seg_axis, const double* __restrict__ seg_cut,
                const int32_t* __restrict__ cloff, const int32_t* __restrict__ seg_nl,
                TmpCells tmp, const float* __restrict__ seg_xb) {
  const int b = blockIdx.x;
  if (b >= counters[C_CHUNKS]) return;
  const int s = chunk_seg[b];
  const Seg g = segs[s];
  const int rel0 = (b - seg_off[s]) * 8 * T;
  const int code = seg_nl[s];
  const bool fallback = code < 0;
  const int nl = fallback ? -code - 1 : code;
  const int axis = seg_axis[s];
  // small evaluations wait on latency: all the moves of a thread in flight
  constexpr int kMoveBatch = T == 64 ? 8 : 2;
  const long long ckey = dkey(seg_cut[s]);
  __shared__ int wcount[kScatterPasses][T / 32];
  __shared__ long long ws2[T / 32];
  __shared__ int wd2[T / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  bool flag[kScatterPasses];
  int rank[kScatterPasses];
#pragma unroll
  for (int pass = 0; pass < kScatterPasses; ++pass) {
    const int k = rel0 + pass * T + threadIdx.x;   // position within the segment
    flag[pass] = false;
    if (k < g.count)
      flag[pass] = fallback ? (k < nl) : (dkey(coord(src, axis, (int64_t)g.first + k)) < ckey);
  }
#pragma unroll
  for (int pass = 0; pass < kScatterPasses; ++pass) {
    const unsigned mask = __ballot_sync(0xffffffffu, flag[pass]);
    rank[pass] = __popc(mask & lt);
    if (lane == 0) wcount[pass][w] = __popc(mask);
  }
  __syncthreads();
  int before = fallback ? min(rel0, nl) : cloff[b];          // left elements before the pass
#pragma unroll
  for (int pass = 0; pass < kScatterPasses; ++pass) {
    int woff = 0, tot = 0;
#pragma unroll
    for (int q = 0; q < T / 32; ++q) {
      const int c = wcount[pass][q];
      woff += q < w ? c : 0;
      tot += c;
    }
    rank[pass] += before + woff;                               // left elements before this one
    before += tot;
  }
  const double cx = tmp.cx[g.cell], cy = tmp.cy[g.cell], cz = tmp.cz[g.cell];
  const float cxf = trunc_to_float(cx), cyf = trunc_to_float(cy), czf = trunc_to_float(cz);
  float dmax = 0.0f;                  // largest float32 squared distance to the centre of mass
#pragma unroll 1
  for (int p0 = 0; p0 < kScatterPasses; p0 += kMoveBatch) {
    double px[kMoveBatch], py[kMoveBatch], pz[kMoveBatch], pm[kMoveBatch];
    int32_t pi[kMoveBatch];
#pragma unroll
    for (int u = 0; u < kMoveBatch; ++u) {
      const int k = rel0 + (p0 + u) * T + threadIdx.x;
      px[u] = py[u] = pz[u] = pm[u] = 0.0;
      pi[u] = 0;
      if (k < g.count) {
        const int64_t i = (int64_t)g.first + k;
        px[u] = src.x[i]; py[u] = src.y[i]; pz[u] = src.z[i];
        pm[u] = src.m[i]; pi[u] = src.idx[i];
      }
    }
#pragma unroll
    for (int u = 0; u < kMoveBatch; ++u) {
      const int k = rel0 + (p0 + u) * T + threadIdx.x;
      if (k >= g.count) continue;
      const int lb = rank[p0 + u];
      const int64_t d = flag[p0 + u] ? (int64_t)g.first + lb : (int64_t)g.first + nl + (k - lb);
      dst.x[d] = px[u]; dst.y[d] = py[u]; dst.z[d] = pz[u];
      dst.m[d] = pm[u]; dst.idx[d] = pi[u];
      const float ex = trunc_to_float(px[u]) - cxf, ey = trunc_to_float(py[u]) - cyf,
                  ez = trunc_to_float(pz[u]) - czf;
      dmax = fmaxf(dmax, ex * ex + ey * ey + ez * ez);
    }
  }
  // the chunk's largest exact distance, from the elements whose float32 distance
  // is within its error of the chunk's largest (the segment's largest is the
  // largest of its chunks').  The few threads that hold one read theirs again:
  // distances kept for all passes unrolled the moves, 4.9 ms against 3.3 of the
  // build of 2^24 particles.
  const int dm = __reduce_max_sync(0xffffffffu, __float_as_int(dmax));
  if (lane == 0) wd2[w] = dm;
  __syncthreads();
  int db = 0;
#pragma unroll
  for (int q = 0; q < T / 32; ++q) db = max(db, wd2[q]);
  const float Dm = sqrtf(__int_as_float(db));
  const float thr = Dm - 2.0f * dist_err_bound(seg_xb[s], Dm);
  const float thr2 = thr > 0.0f ? thr * thr * (1.0f - 1e-6f) : -1.0f;
  long long s2 = 0;
  if (dmax >= thr2) {
#pragma unroll 4
    for (int pass = 0; pass < kScatterPasses; ++pass) {
      const int k = rel0 + pass * T + threadIdx.x;
      if (k >= g.count) continue;
      const int64_t i = (int64_t)g.first + k;
      const double px = src.x[i], py = src.y[i], pz = src.z[i];
      const float ex = trunc_to_float(px) - cxf, ey = trunc_to_float(py) - cyf,
                  ez = trunc_to_float(pz) - czf;
      if (ex * ex + ey * ey + ez * ez >= thr2)
        s2 = max(s2, __double_as_longlong(dist2_rn(px, py, pz, cx, cy, cz)));
    }
  }
  s2 = warp_max_ll(s2);
  if (lane == 0) ws2[w] = s2;
  __syncthreads();
  if (threadIdx.x == 0) {
    long long m2 = 0;
    for (int q = 0; q < T / 32; ++q) m2 = max(m2, ws2[q]);
    if (m2 > 0)
      atomicMax(reinterpret_cast<unsigned long long*>(&tmp.s[g.cell]), (unsigned long long)m2);
  }
}

// ---------------------------------------------------------------------------
// phase B: one CTA finishes a subtree in shared memory
// ---------------------------------------------------------------------------
struct SubArgs {
  BuildArgs A;
  PCols buf0, buf1, out;
  const Seg* segB;
  int qcap;
  const double* h;                     // caller's smoothing lengths, or NULL: the systems' softening
  const double* sys_eps;
};

// All cells of a tree level are processed together, in batches of up to
// kBatchCells: a cell's particles are cut into octets (8 consecutive
// positions, an aligned block of its pairwise tree), a thread takes an octet
// whatever the size of its cell, and the octets' sums are folded cell by cell
// as the rest of the perfect binary tree.  So every level keeps the CTA's
// threads equally busy, and takes a dozen barriers.  Splitting large cells by
// the CTA one after the other, medium ones by a warp and small ones by a
// thread left most warps idle behind one: 1009 particles on one CTA took 323 us
// (now 87), a 60013-particle sphere 450 us (134), 2^24 clumped particles 10.4 ms
// (4.0).  While the subtrees leave SMs idle (E = 4) an octet is four particles
// and the CTA has 512 threads: half the instructions a thread and level (1009
// particles 101 -> 87 us, 60013 175 -> 134 us).
// Bound: the float64 pipe (1/64 rate; 3 products and 4 sums a particle and
// level) once the SMs are full, barriers and shared-memory latency before.
constexpr int kBatchCells = 128;
template <int E>
struct SubShape {
  static constexpr int kThreads = kSubtreeMax / E, kOctets = kSubtreeMax / E + kBatchCells, kPerThread = 2,
                       kLog = E == 8 ? 3 : 2;
  static_assert(E == 8 || E == 4, "particles of an octet");
  static_assert(kOctets <= kPerThread * kThreads, "octets of a batch per thread");
  static_assert(kBatchCells * 2 <= kThreads && kBatchCells % 32 == 0, "cells of a batch per thread");
};

// Shared-memory views of one subtree.
struct SubSmem {
  double *x, *y, *z, *m;               // float64 particles (phase-A order)
  Sum4* osum;                          // per octet: its sum, then folded into the cell's first
  long long* key;                      // (same memory) per cell: exact bounding-box keys, if needed
  double* com;                         // per cell: centre of mass
  unsigned long long* s2;              // per cell: exact squared size (bits)
  int* bb;                             // per cell: float32 bounding box keys, min xyz, max xyz
  int *d2m, *axis, *irank;             // per cell: float32 squared size, cut axis, rank among the split
  float* thr2;                         // per cell: candidates for the exact size
  int* oct0;                           // per cell: its first octet (kBatchCells + 1)
  int* opre;                           // per octet: left particles before it (octets + 1)
  uint16_t *idx0, *idx1, *fin;         // particle order of a level (two buffers) and of finished leaves
  int2 *q0, *q1;                       // cells of a level (two buffers): (first | count << 16, cell id)
};

template <int E>
__host__ __device__ __forceinline__ size_t sub_carve(unsigned char* base, int qcap, SubSmem* L) {
  size_t at = 0;
  auto take = [&](size_t bytes) {
    const size_t was = at;
    at += (bytes + 15) / 16 * 16;
    return base + was;
  };
  double* x = reinterpret_cast<double*>(take(4 * kSubtreeMax * sizeof(double)));
  L->x = x; L->y = x + kSubtreeMax; L->z = x + 2 * kSubtreeMax; L->m = x + 3 * kSubtreeMax;
  L->osum = reinterpret_cast<Sum4*>(take(SubShape<E>::kOctets * sizeof(Sum4)));
  L->key = reinterpret_cast<long long*>(L->osum);
  L->com = reinterpret_cast<double*>(take(3 * kBatchCells * sizeof(double)));
  L->s2 = reinterpret_cast<unsigned long long*>(take(kBatchCells * sizeof(unsigned long long)));
  L->bb = reinterpret_cast<int*>(take(6 * kBatchCells * sizeof(int)));
  L->d2m = reinterpret_cast<int*>(take(kBatchCells * sizeof(int)));
  L->axis = reinterpret_cast<int*>(take(kBatchCells * sizeof(int)));
  L->irank = reinterpret_cast<int*>(take(kBatchCells * sizeof(int)));
  L->thr2 = reinterpret_cast<float*>(take(kBatchCells * sizeof(float)));
  L->oct0 = reinterpret_cast<int*>(take((kBatchCells + 1) * sizeof(int)));
  L->opre = reinterpret_cast<int*>(take((SubShape<E>::kOctets + 1) * sizeof(int)));
  uint16_t* ix = reinterpret_cast<uint16_t*>(take(3 * kSubtreeMax * sizeof(uint16_t)));
  L->idx0 = ix; L->idx1 = ix + kSubtreeMax; L->fin = ix + 2 * kSubtreeMax;
  L->q0 = reinterpret_cast<int2*>(take(2 * (size_t)qcap * sizeof(int2)));
  L->q1 = L->q0 + qcap;
  return at;
}

// Order-preserving int32 key of a float.
__device__ __forceinline__ int fkey(float v) {
  const int b = __float_as_int(v);
  return b ^ ((b >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float funkey(int k) { return __int_as_float(k ^ ((k >> 31) & 0x7fffffff)); }

template <int E>
__global__ void __launch_bounds__(SubShape<E>::kThreads, 512 / SubShape<E>::kThreads)
k_subtree(SubArgs S) {
  constexpr int kThreads = SubShape<E>::kThreads, kPerThread = SubShape<E>::kPerThread;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_seg, s_base, s_tot[3][kBatchCells / 32];
  SubSmem L;
  sub_carve<E>(smem_raw, S.qcap, &L);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned full = 0xffffffffu;
  const BuildArgs& A = S.A;
  const TmpCells& T = A.tmp;

  // persistent: the CTA takes segments from a work counter until none is left
  const int nB = min(A.counters[C_NB], (int)A.capB);
  for (;;) {
  __syncthreads();
  if (tid == 0) s_seg = atomicAdd(&A.counters[C_WORK], 1);
  __syncthreads();
  if (s_seg >= nB) break;
  const Seg g = S.segB[s_seg];
  const PCols in = (g.dbuf & 1) ? S.buf1 : S.buf0;
  const int n = g.count, gfirst = g.first;
  const int sys = system_of(A.sys_off, A.n_sys, gfirst);
  const int n_leaf = A.sys_nleaf[sys];
  for (int k = tid; k < n; k += kThreads) {
    L.x[k] = in.x[gfirst + k]; L.y[k] = in.y[gfirst + k]; L.z[k] = in.z[gfirst + k];
    L.m[k] = in.m[gfirst + k];
    L.idx0[k] = (uint16_t)k;
  }
  if (tid == 0) L.q0[0] = make_int2(n << 16, g.cell);
  int cur = 0, nq = 1, depth = g.dbuf >> 1;
  bool overflow = false;
  __syncthreads();
  while (nq > 0 && !overflow) {
    const uint16_t* const ix = cur ? L.idx1 : L.idx0;
    uint16_t* const ox = cur ? L.idx0 : L.idx1;
    const int2* const q_in = cur ? L.q1 : L.q0;
    int2* const q_out = cur ? L.q0 : L.q1;
    int nq_next = 0;
    for (int b0 = 0; b0 < nq && !overflow; b0 += kBatchCells) {
      const int ncb = min(kBatchCells, nq - b0);
      const int2* const q = q_in + b0;
      // octets and split cells before each cell (packed in one scan)
      int cnt_c = 0, pack = 0, incl = 0;
      if (tid < kBatchCells) {
        cnt_c = tid < ncb ? q[tid].x >> 16 : 0;
        incl = pack = ((cnt_c + E - 1) / E) | (cnt_c > n_leaf) << 16;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_up_sync(full, incl, o);
          if (lane >= o) incl += v;
        }
        const int mx = __reduce_max_sync(full, pack & 0xffff);
        if (lane == 31) { s_tot[0][warp] = incl; s_tot[1][warp] = mx; }
      }
      __syncthreads();
      int noct = 0, nsplit = 0, maxoct = 0;
#pragma unroll
      for (int w = 0; w < kBatchCells / 32; ++w) {
        const int v = s_tot[0][w];
        if (w < warp) incl += v;
        noct += v & 0xffff;
        nsplit += v >> 16;
        maxoct = max(maxoct, s_tot[1][w]);
      }
      int base = 0;                       // (thread 0) first id of the children
      if (tid < kBatchCells) {
        const int ex = incl - pack;
        L.oct0[tid] = ex & 0xffff;
        L.irank[tid] = ex >> 16;
        L.s2[tid] = 0ull;
        L.d2m[tid] = 0;
#pragma unroll
        for (int d = 0; d < 3; ++d) { L.bb[6 * tid + d] = INT_MAX; L.bb[6 * tid + 3 + d] = INT_MIN; }
        if (tid == 0) {
          L.oct0[kBatchCells] = noct;
          if (nsplit > 0) base = atomicAdd(&A.counters[C_CELLS], 2 * nsplit);
        }
      }
      __syncthreads();
      // the thread's octets: cell, first element in the cell, elements
      int oc[kPerThread], rel[kPerThread], val[kPerThread];
      int lf[kPerThread], cn[kPerThread];
#pragma unroll
      for (int u = 0; u < kPerThread; ++u) {
        const int o = tid + u * kThreads;
        oc[u] = -1; rel[u] = val[u] = lf[u] = cn[u] = 0;
        if (o < noct) {
          int c = 0;
#pragma unroll
          for (int step = kBatchCells / 2; step > 0; step >>= 1)
            if (c + step < ncb && L.oct0[c + step] <= o) c += step;
          const int e = q[c].x;
          oc[u] = c;
          lf[u] = e & 0xffff;
          cn[u] = e >> 16;
          rel[u] = E * (o - L.oct0[c]);
          val[u] = min(E, cn[u] - rel[u]);
        }
      }
      // octet sums, float32 bounding boxes (coordinates truncated: monotone)
#pragma unroll
      for (int u = 0; u < kPerThread; ++u) {
        if (u * kThreads + (tid & ~31) >= noct) continue;    // the whole warp has none
        int lo[3] = {INT_MAX, INT_MAX, INT_MAX}, hi[3] = {INT_MIN, INT_MIN, INT_MIN};
        if (oc[u] >= 0) {
          const uint16_t* p = ix + lf[u] + rel[u];
          auto get = [&](int k) {
            const int i = p[k];
            const double x = L.x[i], y = L.y[i], z = L.z[i];
            const int kx = fkey(trunc_to_float(x)), ky = fkey(trunc_to_float(y)),
                      kz = fkey(trunc_to_float(z));
            lo[0] = min(lo[0], kx); hi[0] = max(hi[0], kx);
            lo[1] = min(lo[1], ky); hi[1] = max(hi[1], ky);
            lo[2] = min(lo[2], kz); hi[2] = max(hi[2], kz);
            return elem4(L.m[i], x, y, z);
          };
          L.osum[tid + u * kThreads] = block_tree<SubShape<E>::kLog>(0, val[u], get);
        }
        if (__all_sync(full, oc[u] == __shfl_sync(full, oc[u], 0))) {   // one cell: one set of atomics
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const int l = __reduce_min_sync(full, lo[d]), h = __reduce_max_sync(full, hi[d]);
            if (lane == 0) { atomicMin(&L.bb[6 * oc[u] + d], l); atomicMax(&L.bb[6 * oc[u] + 3 + d], h); }
          }
        } else if (oc[u] >= 0) {
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            atomicMin(&L.bb[6 * oc[u] + d], lo[d]);
            atomicMax(&L.bb[6 * oc[u] + 3 + d], hi[d]);
          }
        }
      }
      // the rest of the pairwise tree: octets 2s apart take the one s after
      for (int s = 1; s < maxoct; s <<= 1) {
        __syncthreads();
#pragma unroll
        for (int u = 0; u < kPerThread; ++u) {
          const int r = rel[u] / E;
          if (oc[u] >= 0 && (r & (2 * s - 1)) == 0 && E * (r + s) < cn[u]) {
            Sum4* p = L.osum + tid + u * kThreads;
            p[0] = add4(p[0], p[s]);
          }
        }
      }
      if (tid == 0) s_base = nsplit > 0 && base + 2 * nsplit > A.cap_cells ? -1 : base;
      __syncthreads();
      // centres of mass, cut axes; an axis whose lead is within the error of
      // the float32 box is decided from the exact box
      bool unclear = false;
      for (int t = tid; t < 4 * ncb; t += kThreads) {
        const int c = t >> 2, d = t & 3, cell = q[c].y;
        const Sum4& v = L.osum[L.oct0[c]];
        if (d < 3) {
          const double quo = __ddiv_rn(d == 0 ? v.x : (d == 1 ? v.y : v.z), v.m);
          L.com[3 * c + d] = quo;
          (d == 0 ? T.cx : (d == 1 ? T.cy : T.cz))[cell] = quo;
        } else {
          T.M[cell] = v.m;
          T.first[cell] = gfirst + (q[c].x & 0xffff);
          T.count[cell] = q[c].x >> 16;
          T.depth[cell] = depth;
          float ext[3], X = 0.0f;
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            const float l = funkey(L.bb[6 * c + k]), h = funkey(L.bb[6 * c + 3 + k]);
            ext[k] = h - l;
            X = fmaxf(X, fmaxf(fabsf(l), fabsf(h)));
          }
          int ax = 0;
          float best = ext[0];
          if (ext[1] > best) { ax = 1; best = ext[1]; }
          if (ext[2] > best) { ax = 2; best = ext[2]; }
          // an extent is off by less than 3 x 2^-23 X (two truncations, one
          // rounding); NaN and infinite boxes are unclear too
          const float margin = X * 1e-6f + 1e-37f;
          bool clear = true;
#pragma unroll
          for (int k = 0; k < 3; ++k) clear = clear && (k == ax || best - ext[k] > margin);
          if (q[c].x >> 16 <= n_leaf) clear = true;               // a leaf is not cut
          L.axis[c] = clear ? ax : -1;
          unclear = unclear || !clear;
        }
      }
      const bool exact = __syncthreads_or(unclear);
      if (s_base < 0) {
        if (tid == 0) set_status(A.status, ST_CAPACITY);
        overflow = true;
        continue;
      }
      if (exact) {
        for (int t = tid; t < 6 * ncb; t += kThreads) L.key[t] = t % 6 < 3 ? LLONG_MAX : LLONG_MIN;
        __syncthreads();
#pragma unroll
        for (int u = 0; u < kPerThread; ++u) {
          if (oc[u] < 0 || L.axis[oc[u]] >= 0) continue;
          for (int k = 0; k < val[u]; ++k) {
            const int i = ix[lf[u] + rel[u] + k];
            long long* key = L.key + 6 * oc[u];
            const long long kk[3] = {dkey(L.x[i]), dkey(L.y[i]), dkey(L.z[i])};
            for (int d = 0; d < 3; ++d) { atomicMin(&key[d], kk[d]); atomicMax(&key[3 + d], kk[d]); }
          }
        }
        __syncthreads();
        if (tid < ncb && L.axis[tid] < 0) {
          double dlo[3], dhi[3];
          for (int d = 0; d < 3; ++d) {
            dlo[d] = dunkey(L.key[6 * tid + d]);
            dhi[d] = dunkey(L.key[6 * tid + 3 + d]);
          }
          L.axis[tid] = longest_axis(dlo, dhi);
        }
        __syncthreads();
      }
      // left flags (bits of the octet) and float32 squared distances
      unsigned left[kPerThread];
      float d2[kPerThread][E];
#pragma unroll
      for (int u = 0; u < kPerThread; ++u) {
        left[u] = 0u;
        if (u * kThreads + (tid & ~31) >= noct) continue;
        float mx = 0.0f;
        if (oc[u] >= 0) {
          const double* com = L.com + 3 * oc[u];
          const float cx = trunc_to_float(com[0]), cy = trunc_to_float(com[1]), cz = trunc_to_float(com[2]);
          const bool cut = cn[u] > n_leaf;
          const int ax = L.axis[oc[u]];
          const long long ckey = dkey(com[ax]);
#pragma unroll
          for (int k = 0; k < E; ++k) {
            d2[u][k] = -2.0f;
            if (k < val[u]) {
              const int i = ix[lf[u] + rel[u] + k];
              const double x = L.x[i], y = L.y[i], z = L.z[i];
              const float dx = trunc_to_float(x) - cx, dy = trunc_to_float(y) - cy, dz = trunc_to_float(z) - cz;
              d2[u][k] = dx * dx + dy * dy + dz * dz;
              mx = fmaxf(mx, d2[u][k]);
              const double a = ax == 0 ? x : (ax == 1 ? y : z);
              if (cut && dkey(a) < ckey) left[u] |= 1u << k;
            }
          }
          L.opre[tid + u * kThreads] = __popc(left[u]);
        }
        if (__all_sync(full, oc[u] == __shfl_sync(full, oc[u], 0))) {
          const int m = __reduce_max_sync(full, __float_as_int(mx));
          if (lane == 0) atomicMax(&L.d2m[oc[u]], m);
        } else if (oc[u] >= 0) {
          atomicMax(&L.d2m[oc[u]], __float_as_int(mx));
        }
      }
      __syncthreads();
      if (warp == 0) {                    // left particles before each octet of the batch
        constexpr int kPer = SubShape<E>::kOctets / 32;
        int v[kPer], run = 0;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
          const int o = lane * kPer + k;
          v[k] = run;
          run += o < noct ? L.opre[o] : 0;
        }
        int in2 = run;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int w = __shfl_up_sync(full, in2, o);
          if (lane >= o) in2 += w;
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
          const int o = lane * kPer + k;
          if (o < noct) L.opre[o] = in2 - run + v[k];
        }
        if (lane == 31) L.opre[noct] = in2;
      } else if (tid >= kBatchCells && tid - kBatchCells < ncb) {
        const int c = tid - kBatchCells;
        float X = 0.0f;
#pragma unroll
        for (int k = 0; k < 6; ++k) X = fmaxf(X, fabsf(funkey(L.bb[6 * c + k])));
        const float Dm = sqrtf(__int_as_float(L.d2m[c]));
        const float thr = Dm - 2.0f * dist_err_bound(X * 1.000001f, Dm);
        L.thr2[c] = thr > 0.0f ? thr * thr * (1.0f - 1e-6f) : -1.0f;
      }
      __syncthreads();
      // exact size from the candidates; the stable partition of cut cells
#pragma unroll
      for (int u = 0; u < kPerThread; ++u) {
        const int c = oc[u];
        if (c < 0) continue;
        const float thr2 = L.thr2[c];
        unsigned cand = 0u;
#pragma unroll
        for (int k = 0; k < E; ++k)
          if (k < val[u] && d2[u][k] >= thr2) cand |= 1u << k;
        const uint16_t* p = ix + lf[u] + rel[u];
        long long s2 = 0;
        while (cand != 0u) {
          const int i = p[__ffs(cand) - 1];
          cand &= cand - 1u;
          s2 = max(s2, __double_as_longlong(dist2_rn(L.x[i], L.y[i], L.z[i], L.com[3 * c],
                                                     L.com[3 * c + 1], L.com[3 * c + 2])));
        }
        if (s2 > 0) atomicMax(&L.s2[c], (unsigned long long)s2);
        if (cn[u] <= n_leaf) {
          for (int k = 0; k < val[u]; ++k) L.fin[lf[u] + rel[u] + k] = p[k];
        } else {
          const int before = L.opre[L.oct0[c]], nl = L.opre[c + 1 < ncb ? L.oct0[c + 1] : noct] - before;
          if (nl == 0 || nl == cn[u]) {                            // split by position: order kept
            for (int k = 0; k < val[u]; ++k) ox[lf[u] + rel[u] + k] = p[k];
          } else {
            int l = L.opre[tid + u * kThreads] - before, r = nl + rel[u] - l;
            for (int k = 0; k < val[u]; ++k)
              ox[lf[u] + ((left[u] >> k & 1u) ? l++ : r++)] = p[k];
          }
        }
      }
      __syncthreads();
      // sizes, children
      if (tid < ncb) {
        const int cell = q[tid].y, first = q[tid].x & 0xffff, cnt = q[tid].x >> 16;
        T.s[cell] = __longlong_as_double((long long)L.s2[tid]);
        if (cnt > n_leaf) {
          int nl = L.opre[tid + 1 < ncb ? L.oct0[tid + 1] : noct] - L.opre[L.oct0[tid]];
          if (nl == 0 || nl == cnt) {
            nl = cnt / 2;
            atomicAdd(&A.counters[C_FALLBACK], 1);
          }
          const int cid = s_base + 2 * L.irank[tid];
          T.left[cell] = cid;
          T.right[cell] = cid + 1;
          int2* out = q_out + nq_next + 2 * L.irank[tid];
          out[0] = make_int2(nl << 16 | first, cid);
          out[1] = make_int2((cnt - nl) << 16 | (first + nl), cid + 1);
        } else {
          T.left[cell] = -1;
          T.right[cell] = -1;
        }
      }
      nq_next += 2 * nsplit;
      __syncthreads();
    }
    cur ^= 1;
    nq = nq_next;
    if (nq > 0) ++depth;
  }
  if (overflow) continue;
  if (tid == 0) atomicMax(&A.counters[C_DEPTH], depth);
  for (int k = tid; k < n; k += kThreads) {
    const int src = L.fin[k];
    const int64_t p = (int64_t)gfirst + k;
    S.out.x[p] = L.x[src]; S.out.y[p] = L.y[src]; S.out.z[p] = L.z[src]; S.out.m[p] = L.m[src];
    const int32_t i = in.idx[gfirst + src];
    S.out.h[p] = S.h ? S.h[i] : S.sys_eps[sys];
    S.out.idx[p] = i;
  }
  }
}

// Leaves produced directly by phase A (or a root that is already a leaf): one
// thread per leaf, pairwise sums by a carry stack.
__global__ void k_leaf_segs(SubArgs S, const Seg* __restrict__ segL) {
  const int nL = min(S.A.counters[C_NL], (int)S.A.capL);
  KD_GRID_STRIDE(sidx, nL) {
  const Seg g = segL[sidx];
  const PCols in = (g.dbuf & 1) ? S.buf1 : S.buf0;
  const int cnt = g.count;
  int P = 1;
  while (P < cnt) P <<= 1;
  Sum4 st[8];
  int top = 0;
  for (int k = 0; k < P; ++k) {
    Sum4 e = zero4();
    if (k < cnt) {
      const int64_t i = (int64_t)g.first + k;
      e = elem4(in.m[i], in.x[i], in.y[i], in.z[i]);
    }
    for (int kk = k; kk & 1; kk >>= 1) e = add4(st[--top], e);
    st[top++] = e;
  }
  const Sum4 v = st[0];
  const double M = v.m;
  const double cx = __ddiv_rn(v.x, M), cy = __ddiv_rn(v.y, M), cz = __ddiv_rn(v.z, M);
  long long s2 = 0;
  for (int k = 0; k < cnt; ++k) {
    const int64_t i = (int64_t)g.first + k;
    s2 = max(s2, __double_as_longlong(dist2_rn(in.x[i], in.y[i], in.z[i], cx, cy, cz)));
    S.out.x[i] = in.x[i]; S.out.y[i] = in.y[i]; S.out.z[i] = in.z[i];
    S.out.m[i] = in.m[i]; S.out.idx[i] = in.idx[i];
    S.out.h[i] = S.h ? S.h[in.idx[i]] : S.sys_eps[system_of(S.A.sys_off, S.A.n_sys, g.first)];
  }
  TmpCells t = S.A.tmp;
  const int c = g.cell;
  t.first[c] = g.first; t.count[c] = cnt; t.depth[c] = g.dbuf >> 1;
  t.M[c] = M; t.cx[c] = cx; t.cy[c] = cy; t.cz[c] = cz;
  t.s[c] = __longlong_as_double(s2);
  t.left[c] = -1; t.right[c] = -1;
  }
}

// ---------------------------------------------------------------------------
// pre-order numbering: a cell's id is the number of cells starting before its
// first particle plus its depth below the topmost cell starting there; a
// leaf's ordinal the number of leaves starting before it.  One scan over the
// particle positions counts both (cells in the low, leaves in the high half
// of a 64-bit word).
// ---------------------------------------------------------------------------
typedef unsigned long long Starts;
__device__ __forceinline__ int cells_before(const Starts* off, int64_t p) { return (int)(unsigned)off[p]; }
__device__ __forceinline__ int leaves_before(const Starts* off, int64_t p) { return (int)(off[p] >> 32); }

__global__ void k_number_init(Starts* starts, int32_t* min_depth, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) { starts[i] = 0; min_depth[i] = INT_MAX; }
}

// Cells to number.  A build that did not come to its end (too few phase-A levels,
// a full list, refused input) leaves cells whose links are those of an earlier
// tree: it counts as without cells, so that the numbering finds none, k_remap
// leaves no cells and no leaves in the counters, and neither the kernels after it
// nor the walk, M2L and P2P of a captured evaluation touch that tree.  The status
// word tells the host.
__device__ __forceinline__ int cells_to_number(const int32_t* counters) {
  const int ncells = counters[C_CELLS];
  return counters[C_STATUS] & (ST_UNFINISHED | ST_CAPACITY | ST_NONFINITE) ? 0 : ncells;
}

__global__ void k_count_starts(TmpCells tmp, const int32_t* __restrict__ counters, Starts* cnt,
                               int32_t* min_depth) {
  const int ncells = cells_to_number(counters);
  KD_GRID_STRIDE(c, ncells) {
    const int f = tmp.first[c];
    atomicAdd(&cnt[f], tmp.left[c] < 0 ? (Starts(1) << 32 | 1) : Starts(1));
    atomicMin(&min_depth[f], tmp.depth[c]);
  }
}

__device__ __forceinline__ int preorder_id(const Starts* off, const int32_t* min_depth, int first,
                                           int depth) {
  return cells_before(off, first) + depth - min_depth[first];
}

// Cells in pre-order, their sizes (the square root of the squared size), the
// leaves with their systems, the systems' roots; the leaf count goes to
// counters[C_LEAVES].
__global__ void k_remap(TmpCells tmp, int32_t* counters, const Starts* __restrict__ off,
                        const int32_t* __restrict__ min_depth, Cells c, int32_t* status, int64_t n,
                        int32_t* leaf_rank, int32_t* leaf_cells, int32_t* leaf_sys,
                        const int64_t* __restrict__ sys_off, int n_sys, int32_t* sys_root) {
  const int t_n = cells_to_number(counters);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    counters[C_LEAVES] = leaves_before(off, n);
    if (t_n == 0) counters[C_CELLS] = 0;         // (other blocks go by the status alone then)
  }
  KD_GRID_STRIDE(k, n_sys + 1) sys_root[k] = cells_before(off, sys_off[k]);
  KD_GRID_STRIDE(t, t_n) {
  const int f = tmp.first[t], cnt = tmp.count[t], d = tmp.depth[t];
  const int id = preorder_id(off, min_depth, f, d);
  c.first[id] = f; c.count[id] = cnt; c.depth[id] = d;
  c.skip[id] = cells_before(off, f + cnt);
  c.M[id] = tmp.M[t]; c.cx[id] = tmp.cx[t]; c.cy[id] = tmp.cy[t]; c.cz[id] = tmp.cz[t];
  c.s[id] = sqrt(tmp.s[t]);
  c.ready[id] = 0;
  const int lt = tmp.left[t];
  if (lt >= 0) {
    const int rt = tmp.right[t];
    const int idl = preorder_id(off, min_depth, tmp.first[lt], tmp.depth[lt]);
    const int idr = preorder_id(off, min_depth, tmp.first[rt], tmp.depth[rt]);
    if (idl != id + 1) atomicOr(status, ST_INTERNAL);
    c.left[id] = idl; c.right[id] = idr;
    c.parent[idl] = id; c.parent[idr] = id;
    leaf_rank[id] = -1;
  } else {
    c.left[id] = -1; c.right[id] = -1;
    const int r = leaves_before(off, f);
    leaf_rank[id] = r;
    leaf_cells[r] = id;
    leaf_sys[r] = system_of(sys_off, n_sys, f);
  }
  if (d == 0) c.parent[id] = -1;               // a system's root
  }
}

// Component q of a symmetric tensor xx xy xz yy yz zz.
__device__ __forceinline__ int comp_i(int q) { return q < 3 ? 0 : (q < 5 ? 1 : 2); }
__device__ __forceinline__ int comp_j(int q) { return q < 3 ? q : (q < 5 ? q - 2 : 2); }
__device__ __forceinline__ double pick3(int i, double x, double y, double z) {
  return i == 0 ? x : (i == 1 ? y : z);
}

// Upward pass: 8 lanes per leaf.  The lanes take the leaf's particles (their
// float32 records on the way), sum S_jk = sum m y_j y_k (9 float64 operations a
// particle) and scatter the sums over the lanes, lane q < 6 holding component
// q: Q = 3 S - tr(S) I (Eq. 7).  Then the group climbs: the second child of a
// cell to finish adds both children's Q, shifted to the parent's centre of mass
// (parallel axes: + M (3 d d - |d|^2 I)), a component a lane.  Every sum runs in a
// fixed order.  Bound by the float64 pipe and, in small trees, by the chain of
// the climb (an atomic and a moment load a level): a thread per leaf did all six
// components itself, 46 operations a level for 13 here, and read its particles
// one after the other.  With the particle records and the cells' views: 1009
// particles 58 us, now 34; 2^24 clumped particles 1.71 ms, now 1.37 (1.92 with the
// views written by the climb, their conversions on a few lanes).
__global__ void __launch_bounds__(128)
k_upward(Cells c, const int32_t* __restrict__ leaf_cells, const int32_t* __restrict__ counters, PCols tp,
         float4* pf, float4* ph) {
  const int lane = threadIdx.x & 31, q = lane & 7, g0 = lane & ~7;
  const unsigned group = 0xffu << g0;
  const int nleaves = counters[C_LEAVES];
  const int qi = comp_i(min(q, 5)), qj = comp_j(min(q, 5));
  const bool diag = qi == qj;
  for (int k = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 3); k < nleaves;
       k += (int)((gridDim.x * blockDim.x) >> 3)) {
    int cur = leaf_cells[k];
    double Q;
    long long hm = 0;                           // largest h, as the bits of a non-negative double
    {
      const int f = c.first[cur], cnt = c.count[cur];
      const double cx = c.cx[cur], cy = c.cy[cur], cz = c.cz[cur];
      double S[8] = {0, 0, 0, 0, 0, 0, 0, 0};
      for (int j = q; j < cnt; j += 8) {
        const int64_t i = (int64_t)f + j;
        const double m = tp.m[i], h = tp.h[i];
        const double y0 = tp.x[i] - cx, y1 = tp.y[i] - cy, y2 = tp.z[i] - cz;
        const double my0 = m * y0, my1 = m * y1, my2 = m * y2;
        S[0] = fma(my0, y0, S[0]); S[1] = fma(my0, y1, S[1]); S[2] = fma(my0, y2, S[2]);
        S[3] = fma(my1, y1, S[3]); S[4] = fma(my1, y2, S[4]); S[5] = fma(my2, y2, S[5]);
        hm = max(hm, __double_as_longlong(h));
        pf[i] = make_float4(rn_to_float(y0), rn_to_float(y1), rn_to_float(y2), rn_to_float(m));
        const float hf = rn_to_float(h);
        const float hi = hf > 0.0f ? 1.0f / hf : 0.0f;
        ph[i] = make_float4(hi, hi * hi * hi, hf, 4.0f * hf * hf);   // 1/h, 1/h^3, h, (2h)^2
      }
      // reduce-scatter: after the exchange over lane bit o, a lane keeps the
      // half of the sums whose index bit equals its own
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        const bool up = (q & o) != 0;
#pragma unroll
        for (int i = 0; i < o; ++i) {
          const double send = up ? S[i] : S[i + o], keep = up ? S[i + o] : S[i];
          S[i] = keep + __shfl_xor_sync(group, send, o);
        }
        hm = max(hm, __shfl_xor_sync(group, hm, o));
      }
      const double tr = __shfl_sync(group, S[0], g0) + __shfl_sync(group, S[0], g0 + 3) +
                        __shfl_sync(group, S[0], g0 + 5);
      Q = diag ? 3.0 * S[0] - tr : 3.0 * S[0];
    }
    for (;;) {
      const double x = c.cx[cur], y = c.cy[cur], z = c.cz[cur], M = c.M[cur];
      if (q < 6) c.Q[6 * (int64_t)cur + q] = Q;
      else if (q == 6) c.hmax[cur] = __longlong_as_double(hm);
      const int p = c.parent[cur];
      if (p < 0) break;
      const int L = p + 1, R = c.right[p], sib = cur == L ? R : L;
      // the parent's and the children's static moments, ahead of the atomic
      const double px = c.cx[p], py = c.cy[p], pz = c.cz[p];
      const double sx = c.cx[sib], sy = c.cy[sib], sz = c.cz[sib], sM = c.M[sib];
      __threadfence();
      __syncwarp(group);
      int arrived = 0;
      if (q == 0) arrived = atomicAdd(&c.ready[p], 1);
      if (__shfl_sync(group, arrived, g0) == 0) break;      // the sibling finishes the parent
      __threadfence();
      const double sQ = q < 6 ? __ldcg(&c.Q[6 * (int64_t)sib + q]) : 0.0;
      const long long sh = __double_as_longlong(__ldcg(&c.hmax[sib]));
      // offsets from the parent's centre of mass: lanes 0-2 this cell's, 3-5
      // the sibling's; |d|^2 M of each child on the lanes' halves
      const double d = q < 3 ? pick3(q, x, y, z) - pick3(q, px, py, pz)
                             : pick3(q - 3, sx, sy, sz) - pick3(q - 3, px, py, pz);
      const double d0 = __shfl_sync(group, d, g0), d1 = __shfl_sync(group, d, g0 + 1),
                   d2 = __shfl_sync(group, d, g0 + 2);
      const double e0 = __shfl_sync(group, d, g0 + 3), e1 = __shfl_sync(group, d, g0 + 4),
                   e2 = __shfl_sync(group, d, g0 + 5);
      const bool half = q >= 4;
      const double u0 = half ? e0 : d0, u1 = half ? e1 : d1, u2 = half ? e2 : d2;
      const double mdd = (half ? sM : M) * (u0 * u0 + u1 * u1 + u2 * u2);
      const double mdd_c = __shfl_sync(group, mdd, g0), mdd_s = __shfl_sync(group, mdd, g0 + 4);
      const double tc = 3.0 * M * pick3(qi, d0, d1, d2), ts = 3.0 * sM * pick3(qi, e0, e1, e2);
      const double vc = Q + fma(tc, pick3(qj, d0, d1, d2), diag ? -mdd_c : 0.0);
      const double vs = sQ + fma(ts, pick3(qj, e0, e1, e2), diag ? -mdd_s : 0.0);
      Q = cur == L ? vc + vs : vs + vc;
      hm = max(hm, sh);
      cur = p;
    }
    __syncwarp(group);
  }
}

// float32 views of the cells.
__global__ void k_derive_cells(Cells c, const int32_t* __restrict__ counters, float* com_bound) {
  const int t_n = counters[C_CELLS];
  KD_GRID_STRIDE(t, t_n) {
  const double cx = c.cx[t], cy = c.cy[t], cz = c.cz[t], M = c.M[t];
  const float hx = rn_to_float(cx), hy = rn_to_float(cy), hz = rn_to_float(cz);
  double Q[6];
  for (int k = 0; k < 6; ++k) Q[k] = c.Q[6 * (int64_t)t + k];
  c.walk[t] = make_float4(hx, hy, hz, rn_to_float(c.s[t]));
  c.walk2[t] = make_float4(rn_to_float(c.hmax[t]), __int_as_float(c.skip[t]),
                           __int_as_float(c.count[t]), 0.0f);
  c.src32[4 * (int64_t)t + 0] = make_float4(hx, hy, hz, rn_to_float(M));
  c.src32[4 * (int64_t)t + 1] =
      make_float4(rn_to_float(cx - float_to_double(hx)), rn_to_float(cy - float_to_double(hy)),
                  rn_to_float(cz - float_to_double(hz)), 0.0f);
  c.src32[4 * (int64_t)t + 2] =
      make_float4(rn_to_float(Q[0]), rn_to_float(Q[1]), rn_to_float(Q[2]), rn_to_float(Q[3]));
  c.src32[4 * (int64_t)t + 3] = make_float4(rn_to_float(Q[4]), rn_to_float(Q[5]), 0.0f, 0.0f);
  double* s64 = c.src64 + 10 * (int64_t)t;
  s64[0] = cx; s64[1] = cy; s64[2] = cz; s64[3] = M;
  for (int k = 0; k < 6; ++k) s64[4 + k] = Q[k];
  const int b = __float_as_int(fmaxf(fabsf(hx), fmaxf(fabsf(hy), fabsf(hz))));
  if (b > *(volatile int*)com_bound) atomicMax(reinterpret_cast<int*>(com_bound), b);
  }
}

// Per-particle float32 data relative to the centre of mass of its leaf.
__global__ void k_particles32(const Cells c, const int32_t* __restrict__ leaf_cells,
                              const int32_t* __restrict__ counters, PCols tp, float4* pf,
                              float4* ph) {
  const int nleaves = counters[C_LEAVES];
  const int lane = threadIdx.x & 31;
  const int w0 = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int nw = (int)((gridDim.x * blockDim.x) >> 5);
  for (int k = w0; k < nleaves; k += nw) {
    const int cell = leaf_cells[k];
    const int f = c.first[cell], cnt = c.count[cell];
    if (lane >= cnt) continue;
    const int64_t i = (int64_t)f + lane;
    pf[i] = make_float4(rn_to_float(tp.x[i] - c.cx[cell]), rn_to_float(tp.y[i] - c.cy[cell]),
                        rn_to_float(tp.z[i] - c.cz[cell]), rn_to_float(tp.m[i]));
    const float h = rn_to_float(tp.h[i]);
    const float hi = h > 0.0f ? 1.0f / h : 0.0f;
    ph[i] = make_float4(hi, hi * hi * hi, h, 4.0f * h * h);   // 1/h, 1/h^3, h, (2h)^2
  }
}

inline unsigned blocks_for(int64_t n, int threads) { return (unsigned)((n + threads - 1) / threads); }

}  // namespace

// ---------------------------------------------------------------------------
// host orchestration
// ---------------------------------------------------------------------------
static int alloc_cols(PCols* c, int64_t n, bool with_h) {
  if (cudaMalloc(&c->x, n * sizeof(double)) != cudaSuccess) return -1;
  if (cudaMalloc(&c->y, n * sizeof(double)) != cudaSuccess) return -1;
  if (cudaMalloc(&c->z, n * sizeof(double)) != cudaSuccess) return -1;
  if (cudaMalloc(&c->m, n * sizeof(double)) != cudaSuccess) return -1;
  if (with_h && cudaMalloc(&c->h, n * sizeof(double)) != cudaSuccess) return -1;
  if (cudaMalloc(&c->idx, n * sizeof(int32_t)) != cudaSuccess) return -1;
  return 0;
}
static void free_cols(PCols* c) {
  cudaFree(c->x); cudaFree(c->y); cudaFree(c->z); cudaFree(c->m); cudaFree(c->h); cudaFree(c->idx);
  *c = PCols{};
}

void free_build_buffers(kdfmm_tree_s* t) {
  for (int k = 0; k < 2; ++k) { free_cols(&t->buf[k]); cudaFree(t->segA[k]); t->segA[k] = nullptr; }
  free_cols(&t->tp);
  void* ptrs[] = {t->segB, t->segL, t->chunk_seg, t->seg_chunk_off, t->chunk_sum, t->chunk_key,
                  t->chunk_left, t->chunk_loff, t->seg_done, t->seg_axis, t->seg_cut, t->seg_nl,
                  t->seg_xb,
                  t->tmp.first, t->tmp.count, t->tmp.left, t->tmp.right, t->tmp.depth, t->tmp.M,
                  t->tmp.cx, t->tmp.cy, t->tmp.cz, t->tmp.s, t->starts, t->min_depth,
                  t->scan_tmp, t->pf, t->ph, t->c.first, t->c.count, t->c.left,
                  t->c.right, t->c.parent, t->c.skip, t->c.depth, t->c.M, t->c.cx, t->c.cy,
                  t->c.cz, t->c.s, t->c.hmax, t->c.Q, t->c.walk, t->c.walk2, t->c.src32,
                  t->c.src64, t->c.ready, t->leaf_cells, t->leaf_rank, t->leaf_sys, t->lexp64,
                  t->lexp32};
  for (void* p : ptrs) cudaFree(p);
  t->segB = t->segL = nullptr;
  t->chunk_seg = t->seg_chunk_off = t->chunk_left = t->chunk_loff = t->seg_axis = t->seg_nl = t->seg_done = nullptr;
  t->chunk_sum = t->seg_cut = nullptr;
  t->chunk_key = nullptr;
  t->seg_xb = nullptr;
  t->tmp = TmpCells{};
  t->starts = nullptr;
  t->min_depth = t->scan_tmp = nullptr;
  t->pf = t->ph = nullptr;
  t->c = Cells{};
  t->leaf_cells = t->leaf_rank = t->leaf_sys = nullptr;
  t->lexp64 = nullptr;
  t->lexp32 = nullptr;
  t->cap_n = 0;
}

#define KD_ALLOC(ptr, count)                                                        \
  do {                                                                              \
    if (cudaMalloc((void**)&(ptr), (size_t)(count) * sizeof(*(ptr))) != cudaSuccess) \
      return set_error(KDFMM_ERR_OOM, "device allocation of %s failed", #ptr);      \
  } while (0)

static int ensure_build_buffers(kdfmm_tree_s* t, int64_t n) {
  if (t->cap_n >= n) return KDFMM_OK;
  cudaDeviceSynchronize();
  free_build_buffers(t);
  cudaGetLastError();
  for (int k = 0; k < 2; ++k)
    if (alloc_cols(&t->buf[k], n, false)) return set_error(KDFMM_ERR_OOM, "particle buffers");
  if (alloc_cols(&t->tp, n, true)) return set_error(KDFMM_ERR_OOM, "tree-order particles");
  t->capA = n / kSubtreeMax + 4;
  t->capB = n / 2 + 4;
  t->capL = n / 4 + 64;
  KD_ALLOC(t->segA[0], t->capA);
  KD_ALLOC(t->segA[1], t->capA);
  KD_ALLOC(t->segB, t->capB);
  KD_ALLOC(t->segL, t->capL);
  // (a later build of fewer particles may take the small chunks)
  t->cap_chunks = std::max<int64_t>(n / kChunk, std::min<int64_t>(n, small_chunk_max()) / (8 * 64)) + t->capA + 4;
  KD_ALLOC(t->chunk_seg, t->cap_chunks);
  KD_ALLOC(t->chunk_sum, 4 * t->cap_chunks);
  KD_ALLOC(t->chunk_key, 6 * t->cap_chunks);
  KD_ALLOC(t->chunk_left, t->cap_chunks);
  KD_ALLOC(t->chunk_loff, t->cap_chunks);
  KD_ALLOC(t->seg_chunk_off, t->capA);
  KD_ALLOC(t->seg_done, 2 * t->capA);
  KD_ALLOC(t->seg_axis, t->capA);
  KD_ALLOC(t->seg_cut, t->capA);
  KD_ALLOC(t->seg_nl, t->capA);
  KD_ALLOC(t->seg_xb, t->capA);
  t->cap_cells = 2 * n + 2;
  const int64_t nc = t->cap_cells;
  KD_ALLOC(t->tmp.first, nc); KD_ALLOC(t->tmp.count, nc); KD_ALLOC(t->tmp.left, nc);
  KD_ALLOC(t->tmp.right, nc); KD_ALLOC(t->tmp.depth, nc); KD_ALLOC(t->tmp.M, nc);
  KD_ALLOC(t->tmp.cx, nc); KD_ALLOC(t->tmp.cy, nc); KD_ALLOC(t->tmp.cz, nc); KD_ALLOC(t->tmp.s, nc);
  KD_ALLOC(t->starts, n + 2);
  KD_ALLOC(t->min_depth, n + 2);
  t->cap_scan = scan_tmp_elems(nc > n + 2 ? nc : n + 2) * 2 + 16;
  KD_ALLOC(t->scan_tmp, t->cap_scan);
  KD_ALLOC(t->pf, n);
  KD_ALLOC(t->ph, n);
  Cells& c = t->c;
  KD_ALLOC(c.first, nc); KD_ALLOC(c.count, nc); KD_ALLOC(c.left, nc); KD_ALLOC(c.right, nc);
  KD_ALLOC(c.parent, nc); KD_ALLOC(c.skip, nc); KD_ALLOC(c.depth, nc);
  KD_ALLOC(c.M, nc); KD_ALLOC(c.cx, nc); KD_ALLOC(c.cy, nc); KD_ALLOC(c.cz, nc);
  KD_ALLOC(c.s, nc); KD_ALLOC(c.hmax, nc); KD_ALLOC(c.Q, 6 * nc);
  KD_ALLOC(c.walk, nc); KD_ALLOC(c.walk2, nc); KD_ALLOC(c.src32, 4 * nc); KD_ALLOC(c.src64, 10 * nc);
  KD_ALLOC(c.ready, nc);
  KD_ALLOC(t->leaf_cells, nc);
  KD_ALLOC(t->leaf_rank, nc + 1);
  KD_ALLOC(t->leaf_sys, nc);
  KD_ALLOC(t->lexp64, 20 * (n + 1));
  KD_ALLOC(t->lexp32, 24 * (n + 1));
  t->cap_n = n;
  return KDFMM_OK;
}

// Queue entries (the cells a level can hold: twice the cells that a level can
// split) and dynamic shared memory of the subtree kernel for trees of the
// given leaf size.
static int subtree_qcap(int n_leaf) { return 2 * (kSubtreeMax / (n_leaf + 1)) + 2; }
static size_t subtree_smem_for(bool fine, int qcap) {
  SubSmem L;
  return fine ? sub_carve<4>(nullptr, qcap, &L) : sub_carve<8>(nullptr, qcap, &L);
}

// Octets of four particles while a CTA of 512 threads an SM takes all subtrees at
// once (a subtree has some 1024 to 2048 particles, and a system at least one);
// beyond that two CTAs of 256 threads an SM overlap each other's barriers (a
// binary of 262146 particles, some 250 subtrees: 165 us against 180).
static bool subtree_fine(const kdfmm_tree_s* t) {
  return std::max<int64_t>(t->n / 1024, t->n_sys) <= sm_count();
}

// Launch sizes of the persistent subtree kernel (host calls only; made once
// per handle and shared-memory size, outside any stream capture).  The
// kernel's shared-memory limit is one value for all handles of the process,
// so it is set to the size of the smallest leaves (1), which no handle
// exceeds: a limit set to this handle's own size would fail the next launch
// of a handle with smaller leaves.
static int subtree_setup(kdfmm_tree_s* t, bool fine, size_t smem) {
  if (t->subtree_smem == smem && t->subtree_fine == fine) return KDFMM_OK;
  void (*const kernel)(SubArgs) = fine ? k_subtree<4> : k_subtree<8>;
  int rc = check_cuda(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)subtree_smem_for(fine, subtree_qcap(1))),
                      "subtree smem attribute");
  if (rc) return rc;
  int per_sm = 0, sms = 0;
  rc = check_cuda(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                      &per_sm, kernel, fine ? SubShape<4>::kThreads : SubShape<8>::kThreads, smem),
                  "subtree occupancy");
  if (rc) return rc;
  rc = check_cuda(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, t->device), "SMs");
  if (rc) return rc;
  t->subtree_grid = std::max(1, per_sm) * std::max(1, sms);
  t->subtree_smem = smem;
  t->subtree_fine = fine;
  return KDFMM_OK;
}

// Builds the tree (or forest).  fixed_levels < 0: the host follows the
// device counters (a synchronisation after the first step, each phase-A
// level, the subtrees and the numbering) and records the number of phase-A
// levels in t->levels_used.  fixed_levels >= 0: the same launches with no
// synchronisation -- exactly that many phase-A levels, every launch sized
// from capacities and reading its count on the device -- so the sequence can
// be captured in a CUDA graph; a phase A that needed more levels, or any
// capacity overflow, is left in the status word for the caller to check (the
// tree then has no cells: cells_to_number).
int build_tree(kdfmm_tree_s* t, const double* x, const double* m, const double* h, cudaStream_t s,
               int fixed_levels) {
  const int64_t n = t->n;
  const bool deferred = fixed_levels >= 0;
  int rc = ensure_build_buffers(t, n);
  if (rc) return rc;
  const kdfmm_params& P = t->p;
  cudaMemsetAsync(t->counters, 0, C_BUILD_END * sizeof(int32_t), s);
  BuildArgs A{};
  A.tmp = t->tmp;
  A.counters = t->counters;
  A.status = t->status;
  A.sys_off = t->sys_off;
  A.sys_nleaf = t->sys_nleaf;
  A.n_sys = t->n_sys;
  A.capA = t->capA; A.capB = t->capB; A.capL = t->capL; A.cap_cells = t->cap_cells;
  k_init<<<blocks_for(n, 256), 256, 0, s>>>(x, m, h, n, t->sys_off, t->n_sys, t->sys_eps,
                                            P.soft_kind, t->buf[0], t->status);
  k_roots<<<blocks_for(t->n_sys, 128), 128, 0, s>>>(A, t->segA[0], t->segB, t->segL);
  t->launches += 2;

  int32_t* hc = t->host_counters;
  auto read_back = [&](const char* what) {
    cudaMemcpyAsync(hc, t->counters, C_BUILD_END * sizeof(int32_t), cudaMemcpyDeviceToHost, s);
    return check_cuda(cudaStreamSynchronize(s), what);
  };
  if (!deferred) {
    if ((rc = read_back("build init"))) return rc;
    if (hc[C_STATUS] & ST_NONFINITE)
      return set_error(KDFMM_ERR_NONFINITE, "non-finite position or non-positive mass / h");
  }
  // phase A: cells above kSubtreeMax, one level per pass
  const bool small = n <= small_chunk_max();
  const unsigned maxc = (unsigned)(n / (small ? 8 * 64 : kChunk) + t->capA + 1);
  int cur = 0, level = 0;
  auto run_level = [&](auto threads, const Seg* segs, Seg* next, int src, int dst) {
    constexpr int T = decltype(threads)::value;
    k_level_map<T><<<1, 1024, 0, s>>>(segs, t->seg_chunk_off, t->chunk_seg, t->seg_done, t->counters,
                                      t->capA, t->status);
    k_chunk_reduce<T><<<maxc, T, 0, s>>>(segs, t->chunk_seg, t->seg_chunk_off, t->counters, t->buf[src],
                                         t->chunk_sum, t->chunk_key, t->seg_done, t->tmp, t->seg_axis,
                                         t->seg_cut, t->seg_xb);
    k_chunk_count<T><<<maxc, T, 0, s>>>(segs, t->chunk_seg, t->seg_chunk_off, t->counters, t->buf[src],
                                        t->seg_axis, t->seg_cut, t->chunk_left, t->seg_done,
                                        t->chunk_loff, t->seg_nl, A, next, t->segB, t->segL, dst);
    k_chunk_scatter<T><<<maxc, T, 0, s>>>(segs, t->chunk_seg, t->seg_chunk_off, t->counters, t->buf[src],
                                          t->buf[dst], t->seg_axis, t->seg_cut, t->chunk_loff, t->seg_nl,
                                          t->tmp, t->seg_xb);
  };
  while (deferred ? level < fixed_levels : hc[C_NEXT_A] > 0) {
    const int src = level & 1, dst = src ^ 1;
    if (small) run_level(std::integral_constant<int, 64>{}, t->segA[cur], t->segA[cur ^ 1], src, dst);
    else run_level(std::integral_constant<int, kChunkThreads>{}, t->segA[cur], t->segA[cur ^ 1], src, dst);
    t->launches += 4;
    cur ^= 1;
    ++level;
    if (!deferred) {
      if ((rc = read_back("build level"))) return rc;
      if (hc[C_STATUS] & ST_CAPACITY) return set_error(KDFMM_ERR_CAPACITY, "segment lists overflow");
      if (level > 200) return set_error(KDFMM_ERR_INTERNAL, "phase A did not terminate");
    }
  }
  if (deferred) {
    if (fixed_levels > 0) {             // (none: no system needs phase A)
      k_levels_done<<<1, 1, 0, s>>>(t->counters, t->status);
      t->launches += 1;
    }
  } else {
    t->levels_used = level;
  }

  // phase B: the remaining cells in shared memory, persistent CTAs
  SubArgs S{};
  S.A = A;
  S.buf0 = t->buf[0];
  S.buf1 = t->buf[1];
  S.out = t->tp;
  S.segB = t->segB;
  S.h = P.soft_kind == KDFMM_SOFT_M4 ? h : nullptr;
  S.sys_eps = t->sys_eps;
  S.qcap = subtree_qcap(t->min_nleaf);
  const bool fine = subtree_fine(t);
  const size_t smem = subtree_smem_for(fine, S.qcap);
  if ((rc = subtree_setup(t, fine, smem))) return rc;
  const int gsub = deferred ? t->subtree_grid : std::max(1, std::min(t->subtree_grid, hc[C_NB]));
  if (fine) k_subtree<4><<<gsub, SubShape<4>::kThreads, smem, s>>>(S);
  else k_subtree<8><<<gsub, SubShape<8>::kThreads, smem, s>>>(S);
  k_leaf_segs<<<grid_blocks(2), 128, 0, s>>>(S, t->segL);
  t->launches += 2;
  if (!deferred) {
    if ((rc = read_back("build subtrees"))) return rc;
    if (hc[C_STATUS] & ST_NONFINITE)
      return set_error(KDFMM_ERR_NONFINITE, "non-finite position or non-positive mass / h");
    if (hc[C_STATUS] & ST_CAPACITY) return set_error(KDFMM_ERR_CAPACITY, "build capacity exceeded");
    t->ncells = hc[C_CELLS];
    t->nfallback = hc[C_FALLBACK];
    t->depth = hc[C_DEPTH];
  }

  // pre-order numbering, counts read on the device
  k_number_init<<<blocks_for(n + 1, 256), 256, 0, s>>>(t->starts, t->min_depth, n + 1);
  k_count_starts<<<grid_blocks(), 256, 0, s>>>(t->tmp, t->counters, t->starts, t->min_depth);
  scan_u64(t->starts, n, reinterpret_cast<unsigned long long*>(t->scan_tmp), s);
  k_remap<<<grid_blocks(), 256, 0, s>>>(t->tmp, t->counters, t->starts, t->min_depth, t->c, t->status, n,
                                      t->leaf_rank, t->leaf_cells, t->leaf_sys, t->sys_off, t->n_sys,
                                      t->sys_root);
  if (!deferred) {
    if ((rc = read_back("build finalise"))) return rc;
    t->nleaves = hc[C_LEAVES];
    if (hc[C_STATUS] & ST_INTERNAL) return set_error(KDFMM_ERR_INTERNAL, "pre-order numbering inconsistent");
  }
  // the grid follows the last known leaf count with a margin; more leaves than
  // groups of 8 lanes loop
  const int64_t up_groups = std::max<int64_t>(t->nleaves, 1) + t->nleaves / 4 + 128;
  k_upward<<<blocks_for(8 * up_groups, 128), 128, 0, s>>>(t->c, t->leaf_cells, t->counters, t->tp, t->pf,
                                                       t->ph);
  k_derive_cells<<<grid_blocks(), 256, 0, s>>>(t->c, t->counters, t->com_bound);
  t->launches += 5 + scan_launches(n);
  return check_cuda(cudaGetLastError(), "build launch");
}

// ---------------------------------------------------------------------------
// Frozen topology: new positions / masses / smoothing lengths for the same
// particles, the tree's cells and the last interaction lists kept.  Leaf sums
// are pairwise over the leaf's particles (tree order = ascending caller index
// within a leaf); a parent's M and sum m x are its left child's plus its right
// child's; s is the exact maximum distance; Q the parallel-axis shift.
// ---------------------------------------------------------------------------
namespace {

__global__ void k_gather_frozen(const double* __restrict__ x, const double* __restrict__ m,
                                const double* __restrict__ h, int64_t n,
                                const int64_t* __restrict__ sys_off, int n_sys,
                                const double* __restrict__ sys_eps, int soft_kind, PCols tp,
                                int32_t* status) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const int64_t i = tp.idx[p];
  const double xi = x[3 * i], yi = x[3 * i + 1], zi = x[3 * i + 2], mi = m[i];
  const double hi = (h != nullptr && soft_kind == KDFMM_SOFT_M4)
                        ? h[i]
                        : sys_eps[system_of(sys_off, n_sys, i)];
  const bool ok = isfinite(xi) && isfinite(yi) && isfinite(zi) && isfinite(mi) && isfinite(hi) &&
                  mi > 0.0 && (soft_kind == KDFMM_SOFT_M4 ? hi > 0.0 : hi >= 0.0);
  if (!ok) atomicOr(status, ST_NONFINITE);
  tp.x[p] = xi; tp.y[p] = yi; tp.z[p] = zi; tp.m[p] = mi; tp.h[p] = hi;
}

// Leaves: pairwise sums (carry stack), centre of mass, exact size, h_max, Q.
__global__ void k_leaf_frozen(Cells c, const int32_t* __restrict__ leaf_cells, int nleaves, PCols tp,
                              double* Sx, double* Sy, double* Sz) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nleaves) return;
  const int t = leaf_cells[k];
  const int f = c.first[t], cnt = c.count[t];
  Sum4 st[8];
  int top = 0;
  for (int j = 0; j < cnt; ++j) {
    const int64_t i = (int64_t)f + j;
    Sum4 e = elem4(tp.m[i], tp.x[i], tp.y[i], tp.z[i]);
    for (int kk = j; kk & 1; kk >>= 1) e = add4(st[--top], e);
    st[top++] = e;
  }
  Sum4 v = st[top - 1];
  for (int i = top - 2; i >= 0; --i) v = add4(st[i], v);
  const double cx = __ddiv_rn(v.x, v.m), cy = __ddiv_rn(v.y, v.m), cz = __ddiv_rn(v.z, v.m);
  long long s2 = 0;
  double q[6] = {0, 0, 0, 0, 0, 0}, hm = 0.0;
  for (int j = 0; j < cnt; ++j) {
    const int64_t i = (int64_t)f + j;
    s2 = max(s2, __double_as_longlong(dist2_rn(tp.x[i], tp.y[i], tp.z[i], cx, cy, cz)));
    const double mi = tp.m[i];
    const double y0 = tp.x[i] - cx, y1 = tp.y[i] - cy, y2 = tp.z[i] - cz;
    const double y2s = y0 * y0 + y1 * y1 + y2 * y2;
    q[0] += mi * (3.0 * y0 * y0 - y2s);
    q[1] += mi * (3.0 * y0 * y1);
    q[2] += mi * (3.0 * y0 * y2);
    q[3] += mi * (3.0 * y1 * y1 - y2s);
    q[4] += mi * (3.0 * y1 * y2);
    q[5] += mi * (3.0 * y2 * y2 - y2s);
    hm = fmax(hm, tp.h[i]);
  }
  c.M[t] = v.m; c.cx[t] = cx; c.cy[t] = cy; c.cz[t] = cz;
  Sx[t] = v.x; Sy[t] = v.y; Sz[t] = v.z;
  c.s[t] = sqrt(__longlong_as_double(s2));
  c.hmax[t] = hm;
  for (int j = 0; j < 6; ++j) c.Q[6 * t + j] = q[j];
}

// Parents from their children, bottom-up (the second child to finish goes on).
__global__ void k_upward_frozen(Cells c, const int32_t* __restrict__ leaf_cells, int nleaves,
                                double* Sx, double* Sy, double* Sz) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nleaves) return;
  int cur = leaf_cells[k];
  while (true) {
    const int p = c.parent[cur];
    if (p < 0) break;
    __threadfence();
    if (atomicAdd(&c.ready[p], 1) == 0) break;
    __threadfence();
    const int L = c.left[p], R = c.right[p];
    const double M = __dadd_rn(__ldcg(&c.M[L]), __ldcg(&c.M[R]));
    const double sx = __dadd_rn(__ldcg(&Sx[L]), __ldcg(&Sx[R]));
    const double sy = __dadd_rn(__ldcg(&Sy[L]), __ldcg(&Sy[R]));
    const double sz = __dadd_rn(__ldcg(&Sz[L]), __ldcg(&Sz[R]));
    const double px = __ddiv_rn(sx, M), py = __ddiv_rn(sy, M), pz = __ddiv_rn(sz, M);
    double q[6] = {0, 0, 0, 0, 0, 0}, hm = 0.0;
    const int ch[2] = {L, R};
    for (int side = 0; side < 2; ++side) {
      const int kc = ch[side];
      const double mk = __ldcg(&c.M[kc]);
      const double d0 = __ldcg(&c.cx[kc]) - px, d1 = __ldcg(&c.cy[kc]) - py, d2 = __ldcg(&c.cz[kc]) - pz;
      const double dd = d0 * d0 + d1 * d1 + d2 * d2;
      q[0] += __ldcg(&c.Q[6 * kc + 0]) + mk * (3.0 * d0 * d0 - dd);
      q[1] += __ldcg(&c.Q[6 * kc + 1]) + mk * (3.0 * d0 * d1);
      q[2] += __ldcg(&c.Q[6 * kc + 2]) + mk * (3.0 * d0 * d2);
      q[3] += __ldcg(&c.Q[6 * kc + 3]) + mk * (3.0 * d1 * d1 - dd);
      q[4] += __ldcg(&c.Q[6 * kc + 4]) + mk * (3.0 * d1 * d2);
      q[5] += __ldcg(&c.Q[6 * kc + 5]) + mk * (3.0 * d2 * d2 - dd);
      hm = fmax(hm, __ldcg(&c.hmax[kc]));
    }
    c.M[p] = M; c.cx[p] = px; c.cy[p] = py; c.cz[p] = pz;
    Sx[p] = sx; Sy[p] = sy; Sz[p] = sz;
    for (int j = 0; j < 6; ++j) c.Q[6 * p + j] = q[j];
    c.hmax[p] = hm;
    cur = p;
  }
}

// Exact size of every super-cell: one warp per cell, float32 filter over
// truncated coordinates, float64 for the candidates.
__global__ void k_size_frozen(Cells c, int ncells, PCols tp) {
  const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (t >= ncells || c.left[t] < 0) return;
  const int64_t f = c.first[t];
  const int cnt = c.count[t];
  const double cx = c.cx[t], cy = c.cy[t], cz = c.cz[t];
  const float cxf = trunc_to_float(cx), cyf = trunc_to_float(cy), czf = trunc_to_float(cz);
  float d2m = 0.0f, X = fmaxf(fabsf(cxf), fmaxf(fabsf(cyf), fabsf(czf)));
  for (int j = lane; j < cnt; j += 32) {
    const float dx = trunc_to_float(tp.x[f + j]) - cxf, dy = trunc_to_float(tp.y[f + j]) - cyf,
                dz = trunc_to_float(tp.z[f + j]) - czf;
    d2m = fmaxf(d2m, dx * dx + dy * dy + dz * dz);
    X = fmaxf(X, fmaxf(fabsf(trunc_to_float(tp.x[f + j])),
                       fmaxf(fabsf(trunc_to_float(tp.y[f + j])), fabsf(trunc_to_float(tp.z[f + j])))));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    d2m = fmaxf(d2m, __shfl_xor_sync(0xffffffffu, d2m, o));
    X = fmaxf(X, __shfl_xor_sync(0xffffffffu, X, o));
  }
  const float Dm = sqrtf(d2m);
  const float thr = Dm - 2.0f * dist_err_bound(X * 1.000001f, Dm);
  const float thr2 = thr > 0.0f ? thr * thr * (1.0f - 1e-6f) : -1.0f;
  long long s2 = 0;
  for (int j = lane; j < cnt; j += 32) {
    const double px = tp.x[f + j], py = tp.y[f + j], pz = tp.z[f + j];
    const float dx = trunc_to_float(px) - cxf, dy = trunc_to_float(py) - cyf,
                dz = trunc_to_float(pz) - czf;
    if (dx * dx + dy * dy + dz * dz >= thr2)
      s2 = max(s2, __double_as_longlong(dist2_rn(px, py, pz, cx, cy, cz)));
  }
  s2 = warp_max_ll(s2);
  if (lane == 0) c.s[t] = sqrt(__longlong_as_double(s2));
}

}  // namespace

int recompute_moments(kdfmm_tree_s* t, const double* x, const double* m, const double* h,
                      cudaStream_t s) {
  const int64_t n = t->n;
  const int ncells = t->ncells, nl = t->nleaves;
  cudaMemsetAsync(t->status, 0, sizeof(int32_t), s);
  cudaMemsetAsync(t->com_bound, 0, sizeof(float), s);
  k_gather_frozen<<<blocks_for(n, 256), 256, 0, s>>>(x, m, h, n, t->sys_off, t->n_sys, t->sys_eps,
                                                     t->p.soft_kind, t->tp, t->status);
  double *Sx = t->tmp.cx, *Sy = t->tmp.cy, *Sz = t->tmp.cz;     // free after the build
  k_leaf_frozen<<<blocks_for(nl, 128), 128, 0, s>>>(t->c, t->leaf_cells, nl, t->tp, Sx, Sy, Sz);
  cudaMemsetAsync(t->c.ready, 0, (size_t)ncells * sizeof(int32_t), s);
  k_upward_frozen<<<blocks_for(nl, 128), 128, 0, s>>>(t->c, t->leaf_cells, nl, Sx, Sy, Sz);
  k_size_frozen<<<blocks_for((int64_t)ncells * 32, 256), 256, 0, s>>>(t->c, ncells, t->tp);
  k_derive_cells<<<grid_blocks(), 256, 0, s>>>(t->c, t->counters, t->com_bound);
  k_particles32<<<grid_blocks(), 256, 0, s>>>(t->c, t->leaf_cells, t->counters, t->tp,
                                                                  t->pf, t->ph);
  t->launches += 6;
  cudaMemcpyAsync(&t->host_counters[16], t->status, sizeof(int32_t), cudaMemcpyDeviceToHost, s);
  int rc = check_cuda(cudaStreamSynchronize(s), "frozen moments");
  if (rc) return rc;
  if (t->host_counters[16] & ST_NONFINITE)
    return set_error(KDFMM_ERR_NONFINITE, "non-finite position or non-positive mass / h");
  return check_cuda(cudaGetLastError(), "frozen moments launch");
}

}  // namespace kdfmm
