// Device-wide exclusive scans (build finalisation, list offsets) and the total
// momentum reduction sum_i m_i v_i (Sec. 4, Eq. 30: the total force the
// leaf-only walk fails to cancel).
#include "kdfmm_internal.cuh"

namespace kdfmm {

namespace {

constexpr int kScanThreads = 256;
constexpr int kScanPer = 8;
constexpr int kScanTile = kScanThreads * kScanPer;

template <class T>
__device__ __forceinline__ T warp_incl_scan(T v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    T w = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += w;
  }
  return v;
}

// Exclusive scan of one tile per block (in place when out is in); the block
// total goes to tot[block].
template <class TI, class TO>
__global__ void k_scan_tile(const TI* in, TO* out, int64_t n, TO* __restrict__ tot) {
  __shared__ TO warp_tot[kScanThreads / 32];
  const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanPer;
  TO v[kScanPer];
  TO run = 0;
#pragma unroll
  for (int k = 0; k < kScanPer; ++k) {
    int64_t i = base + k;
    TO e = i < n ? (TO)in[i] : (TO)0;
    v[k] = run;
    run += e;
  }
  TO incl = warp_incl_scan<TO>(run);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 31) warp_tot[w] = incl;
  __syncthreads();
  if (w == 0) {
    TO t = lane < kScanThreads / 32 ? warp_tot[lane] : (TO)0;
    TO ti = warp_incl_scan<TO>(t);
    if (lane < kScanThreads / 32) warp_tot[lane] = ti - t;
    if (lane == kScanThreads / 32 - 1) tot[blockIdx.x] = ti;
  }
  __syncthreads();
  TO off = warp_tot[w] + incl - run;
#pragma unroll
  for (int k = 0; k < kScanPer; ++k) {
    int64_t i = base + k;
    if (i < n) out[i] = off + v[k];
  }
}

// Exclusive scan of the nb block totals in place, tot[nb] = grand total.
template <class TO>
__global__ void k_scan_top(TO* tot, int64_t nb) {
  __shared__ TO warp_tot[32];
  __shared__ TO carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int64_t base = 0; base < nb; base += blockDim.x) {
    int64_t i = base + threadIdx.x;
    TO e = i < nb ? tot[i] : (TO)0;
    TO incl = warp_incl_scan<TO>(e);
    if (lane == 31) warp_tot[w] = incl;
    __syncthreads();
    if (w == 0) {
      TO t = lane < (int)(blockDim.x / 32) ? warp_tot[lane] : (TO)0;
      TO ti = warp_incl_scan<TO>(t);
      warp_tot[lane] = ti - t;
    }
    __syncthreads();
    TO excl = carry + warp_tot[w] + incl - e;
    __syncthreads();
    if (i < nb) tot[i] = excl;
    if (threadIdx.x == blockDim.x - 1) carry = excl + e;
    __syncthreads();
  }
  if (threadIdx.x == 0) tot[nb] = carry;
}

template <class TO>
__global__ void k_scan_add(TO* __restrict__ out, int64_t n, const TO* __restrict__ tot, int64_t nb) {
  const int64_t base = (int64_t)blockIdx.x * kScanTile;
  const TO off = tot[blockIdx.x];
  for (int k = threadIdx.x; k < kScanTile; k += blockDim.x) {
    int64_t i = base + k;
    if (i < n) out[i] += off;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) out[n] = tot[nb];
}

// The whole scan by one block, tile after tile (8 values a thread).
constexpr int kScanSmall = 32768;
template <class TI, class TO>
__global__ void __launch_bounds__(1024) k_scan_small(const TI* in, TO* out, int n) {
  __shared__ TO warp_tot[2][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  TO carry = 0;
  int buf = 0;
  for (int t0 = 0; t0 < n; t0 += 8 * 1024, buf ^= 1) {
    const int base = t0 + 8 * (int)threadIdx.x;
    TO v[8], run = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const TO e = base + k < n ? (TO)in[base + k] : (TO)0;
      v[k] = run;
      run += e;
    }
    const TO incl = warp_incl_scan<TO>(run);
    if (lane == 31) warp_tot[buf][w] = incl;
    __syncthreads();
    const TO t = warp_tot[buf][lane], ti = warp_incl_scan<TO>(t);
    const TO before = __shfl_sync(0xffffffffu, ti - t, w), total = __shfl_sync(0xffffffffu, ti, 31);
    const TO off = carry + before + incl - run;
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (base + k < n) out[base + k] = off + v[k];
    carry += total;
  }
  if (threadIdx.x == 0) out[n] = carry;
}

// Up to kScanSmall values one block's tiles cost less than two more launches
// (1009 values: 3 us for 10; 16386: 5 for 10).
template <class TI, class TO>
void scan_impl(const TI* in, TO* out, int64_t n, TO* tmp, cudaStream_t s) {
  int64_t nb = (n + kScanTile - 1) / kScanTile;
  if (nb == 0) {
    cudaMemsetAsync(out, 0, sizeof(TO), s);
    return;
  }
  if (n <= kScanSmall) {
    k_scan_small<TI, TO><<<1, 1024, 0, s>>>(in, out, (int)n);
    return;
  }
  k_scan_tile<TI, TO><<<(unsigned)nb, kScanThreads, 0, s>>>(in, out, n, tmp);
  k_scan_top<TO><<<1, 1024, 0, s>>>(tmp, nb);
  k_scan_add<TO><<<(unsigned)nb, kScanThreads, 0, s>>>(out, n, tmp, nb);
}

// ---------------------------------------------------------------------------
// total momentum
// ---------------------------------------------------------------------------
constexpr int kMomThreads = 256;

// Two-sum tree over the rows of sh (sum, error; three components), row r of a
// round taking row r + stride.  A thread does one component of a row (7 float64
// operations a round instead of 21: the rounds are a chain on the 1/64-rate
// pipe); rounds whose partners are all zero, beyond `rows`, change nothing and
// are left out.
__device__ __forceinline__ void momentum_tree(double (*sh)[6], int rows) {
  int stride = kMomThreads / 2;
  while (stride >= rows && stride > 0) stride >>= 1;
  for (; stride > 0; stride >>= 1) {
    for (int t = threadIdx.x; t < 3 * stride; t += kMomThreads) {
      const int c = t / stride, r = t - c * stride;
      double s, e;
      two_sum_d(sh[r][2 * c], sh[r + stride][2 * c], s, e);
      sh[r][2 * c] = s;
      sh[r][2 * c + 1] = __dadd_rn(__dadd_rn(sh[r][2 * c + 1], sh[r + stride][2 * c + 1]), e);
    }
    __syncthreads();
  }
}

// Each block sums its contiguous range in plain float64 per thread, then
// combines its threads with two-sum in a fixed order: partial = (hi, lo) x 3.
// A single block (n <= 4096) writes the result.
__global__ void k_momentum_blocks(const double* __restrict__ m, const double* __restrict__ v,
                                  int64_t n, int64_t per_block, double* __restrict__ part,
                                  double* __restrict__ out) {
  __shared__ double sh[kMomThreads][6];
  const int64_t lo = (int64_t)blockIdx.x * per_block;
  const int64_t hi = min(n, lo + per_block);
  double ax = 0.0, ay = 0.0, az = 0.0;
  for (int64_t i = lo + threadIdx.x; i < hi; i += kMomThreads) {
    double mi = m[i];
    ax = __dadd_rn(ax, __dmul_rn(mi, v[3 * i + 0]));
    ay = __dadd_rn(ay, __dmul_rn(mi, v[3 * i + 1]));
    az = __dadd_rn(az, __dmul_rn(mi, v[3 * i + 2]));
  }
  sh[threadIdx.x][0] = ax; sh[threadIdx.x][1] = 0.0;
  sh[threadIdx.x][2] = ay; sh[threadIdx.x][3] = 0.0;
  sh[threadIdx.x][4] = az; sh[threadIdx.x][5] = 0.0;
  __syncthreads();
  momentum_tree(sh, (int)min((int64_t)kMomThreads, max(hi - lo, (int64_t)0)));
  if (gridDim.x == 1) {
    if (threadIdx.x < 3)
      out[threadIdx.x] = __dadd_rn(sh[0][2 * threadIdx.x], sh[0][2 * threadIdx.x + 1]);
  } else if (threadIdx.x < 6) {
    part[6 * blockIdx.x + threadIdx.x] = sh[0][threadIdx.x];
  }
}

// Combines the partials: thread t folds partials t, t + 256, ... with two-sum,
// then a fixed-order tree over the threads.  Deterministic for a given count.
__global__ void k_momentum_final(const double* __restrict__ part, int nb, double* __restrict__ out) {
  __shared__ double sh[kMomThreads][6];
  double v[6] = {0, 0, 0, 0, 0, 0};
  for (int b = threadIdx.x; b < nb; b += kMomThreads) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      double s, e;
      two_sum_d(v[2 * c], part[6 * b + 2 * c], s, e);
      v[2 * c] = s;
      v[2 * c + 1] = __dadd_rn(__dadd_rn(v[2 * c + 1], part[6 * b + 2 * c + 1]), e);
    }
  }
  for (int j = 0; j < 6; ++j) sh[threadIdx.x][j] = v[j];
  __syncthreads();
  momentum_tree(sh, min(nb, kMomThreads));
  if (threadIdx.x < 3) out[threadIdx.x] = __dadd_rn(sh[0][2 * threadIdx.x], sh[0][2 * threadIdx.x + 1]);
}

}  // namespace

int scan_launches(int64_t n) { return n <= kScanSmall ? 1 : 3; }

int64_t scan_tmp_elems(int64_t n) { return (n + kScanTile - 1) / kScanTile + 2; }

void scan_u64(unsigned long long* v, int64_t n, unsigned long long* tmp, cudaStream_t s) {
  scan_impl<unsigned long long, unsigned long long>(v, v, n, tmp, s);
}

void scan_i32_to_i64(const int32_t* in, int64_t* out, int64_t n, int64_t* tmp, cudaStream_t s) {
  scan_impl<int32_t, int64_t>(in, out, n, tmp, s);
}

int64_t momentum_blocks(int64_t n) {
  int64_t nb = (n + 4095) / 4096;
  if (nb > 1024) nb = 1024;
  if (nb < 1) nb = 1;
  return nb;
}

int momentum(const double* m, const double* v, int64_t n, double* out, double* scratch,
             cudaStream_t s) {
  int64_t nb = momentum_blocks(n);
  int64_t per = (n + nb - 1) / nb;
  k_momentum_blocks<<<(unsigned)nb, kMomThreads, 0, s>>>(m, v, n, per, scratch, out);
  if (nb > 1) k_momentum_final<<<1, kMomThreads, 0, s>>>(scratch, (int)nb, out);
  return check_cuda(cudaGetLastError(), "momentum launch");
}

}  // namespace kdfmm
