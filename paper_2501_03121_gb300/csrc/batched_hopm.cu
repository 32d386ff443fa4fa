// Power methods over many independent FP32 tensors of uneven order and
// shape in one persistent launch: one thread-block cluster runs every sweep
// of one tensor (small tensors: one block, batched_hopm_block.cu) (largest tensors first, pulled from an atomic counter), its
// blocks meeting at the hardware cluster barrier.
//
// A sweep reads A twice and meets d cluster barriers:
//   pass 0     z_0[i] = sum_{j,l} A[i,j,l] x_1[j] w[l], w = x_2 (x) ... (x) x_{d-1}:
//              every block streams a contiguous range of the n_0*n_1 rows of
//              A; a thread owns a column l, so x_1 is applied per element and
//              w once per column sum, and T = A x_1 x_1 is never written.
//   level j    W_j = W_{j-1} x_{j-1} x_{j-1} (W_0 = A), every block a contiguous
//   (1..d-1)   range of the columns; before the barrier the block contracts
//              its own columns with x_{j+1} (x) ... (x) x_{d-1} into its part of z_j.
// After each barrier every block adds the blocks' parts of z_j in rank order
// and normalises for itself (identical inputs and order, hence identical
// vectors and the same status in every block), so no further barrier is
// needed: the vectors live in each block's shared memory.  Parts and W
// buffers alternate, so a block that runs ahead by one phase never writes
// what a slower one still reads.
//
// Bound: the two passes over A, latency (bytes in flight per SM) before HBM:
// 512 threads of 64 registers, two blocks per SM, hold 64-128 bytes of A per
// thread in flight.  512 tensors of 8..192 per mode (2.1e9 elements), 10
// sweeps: 32.8 ms = 5.2 TB/s of the passes, 283 tensors 22 ms, 73 tensors and
// 5 sweeps 4.2 ms; 4096 tensors 265 ms (of another draw 305).  One block per
// tensor, the layout before this one, took 117, 105, 52 and 287 ms (307): a
// single block streams about 10 GB/s, and the launch ended with the largest
// tensors alone on the GPU.
// Streaming (evict-first) loads measured 5-8% faster than plain ones; 256
// threads per block, or three blocks per SM, slower.
#include <algorithm>
#include <mutex>
#include <set>
#include <vector>

#include "common.cuh"
#include "internal.h"

namespace tvcg {
namespace {

constexpr int kHT = 512;              // threads per block
constexpr int kHW = kHT / kWarp;      // warps per block
constexpr int kHSlots = kHW;           // thread partials held per reduction (one warp reduces each)
constexpr int kHXCap = 3072;          // vector entries held in shared memory

using HItem = HopmItem;

// Column tiling of one pass for one block: m chunks of w columns, P rows at a time.
struct HTile {
  int64_t m;
  int w, P;
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

__device__ __forceinline__ uint32_t cluster_id() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
  return r;
}

// Barrier of the cluster's blocks; global writes before it are visible after it.
__device__ __forceinline__ void cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The chunk count with the fewest loads per thread for `rows` rows of
// `cols` columns: chunks of whole warps, the spare warps taking further rows.
__device__ HTile pick_tile(int64_t cols, int64_t rows) {
  HTile best{1, 32, kHW};
  if (cols < 1) return best;
  int64_t cost = INT64_MAX;
  const int64_t m0 = (cols + kHT - 1) / kHT;
  for (int64_t m = m0; m < m0 + 12; m++) {
    const int w = (int)(((cols + m - 1) / m + 31) / 32) * 32;
    const int P = kHT / w;
    const int64_t c = m * ((rows + P - 1) / P);
    if (c < cost) {
      cost = c;
      best = HTile{m, w, P};
    }
    if (w == 32) break;
  }
  return best;
}

// Rows [r0, r1) of phase ph (multiples of four rows, so that x is read in
// 16-byte pieces).
__device__ __forceinline__ void phase_rows(int64_t rows, int P, int ph, int64_t& r0, int64_t& r1) {
  const int64_t rp = ((rows + P - 1) / P + 3) / 4 * 4;
  r0 = min(rows, ph * rp);
  r1 = ph < P ? min(rows, r0 + rp) : r0;
}

template <int VEC>
__device__ __forceinline__ void ld_row(const float* p, float (&v)[VEC]) {
  if constexpr (VEC == 4) {
    const float4 f = __ldcs(reinterpret_cast<const float4*>(p));
    v[0] = f.x;
    v[1] = f.y;
    v[2] = f.z;
    v[3] = f.w;
  } else if constexpr (VEC == 2) {
    const float2 f = __ldcs(reinterpret_cast<const float2*>(p));
    v[0] = f.x;
    v[1] = f.y;
  } else {
    v[0] = __ldcs(p);
  }
}

// Rows in flight per thread (64 to 128 bytes).  Fewer (4 rows of 16 bytes)
// or more (32 rows of 4, which spills) measured 8-15% slower.
template <int VEC>
inline constexpr int kHRows = VEC == 1 ? 16 : 8;

// a[e] = sum_q p[q * stride + e] x[q], q < n, e < VEC, x 16-byte aligned.
template <int VEC>
__device__ __forceinline__ void col_dot(const float* __restrict__ p, int64_t stride, const float* x, int n,
                                        float (&a)[VEC]) {
  constexpr int RB = kHRows<VEC>;
  float b[VEC];
#pragma unroll
  for (int g = 0; g < VEC; g++) a[g] = b[g] = 0.0f;
  int q = 0;
  for (; q + RB <= n; q += RB, x += RB) {
    float v[RB][VEC];
#pragma unroll
    for (int e = 0; e < RB; e++, p += stride) ld_row<VEC>(p, v[e]);
#pragma unroll
    for (int e = 0; e < RB; e += 4) {
      const float4 xv = *reinterpret_cast<const float4*>(x + e);
#pragma unroll
      for (int g = 0; g < VEC; g++) {
        a[g] = __fmaf_rn(v[e][g], xv.x, a[g]);
        b[g] = __fmaf_rn(v[e + 1][g], xv.y, b[g]);
        a[g] = __fmaf_rn(v[e + 2][g], xv.z, a[g]);
        b[g] = __fmaf_rn(v[e + 3][g], xv.w, b[g]);
      }
    }
  }
  if (q < n) {
    const int left = n - q;
    float v[RB - 1][VEC];
#pragma unroll
    for (int e = 0; e < RB - 1; e++, p += stride)
      if (e < left) ld_row<VEC>(p, v[e]);
#pragma unroll
    for (int e = 0; e < RB - 1; e++)
      if (e < left) {
        const float xv = x[e];
#pragma unroll
        for (int g = 0; g < VEC; g++) a[g] = __fmaf_rn(v[e][g], xv, a[g]);
      }
  }
#pragma unroll
  for (int g = 0; g < VEC; g++) a[g] += b[g];
}

__device__ __forceinline__ float warp_add(float v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
  return v;
}

struct HShared {
  int cl;   // blocks per cluster
  int vec;  // columns per load of A
  HItem it;
  HTile tile[TVC_MAX_ORDER];
  float* xs[TVC_MAX_ORDER];
  double red64[kHW + 2];
  alignas(16) float x[kHXCap];
  float red[kHSlots][kHT];
};

// prod_{m = from}^{d-1} x_m[digit_m(l)]
__device__ __forceinline__ float outer_at(const HShared& s, int from, int64_t l) {
  const int d = s.it.d;
  if (from >= d) return 1.0f;
  if (from == d - 1) return s.xs[from][l];
  float r = 1.0f;
  if (l <= 0xFFFFFFFFll) {
    uint32_t rem = (uint32_t)l;
    for (int m = d - 1; m > from; m--) {
      const uint32_t n = (uint32_t)s.it.dims[m];
      const uint32_t q = rem / n;
      r *= s.xs[m][rem - q * n];
      rem = q;
    }
    return r * s.xs[from][rem];
  }
  int64_t rem = l;
  for (int m = d - 1; m > from; m--) {
    const int64_t n = s.it.dims[m], q = rem / n;
    r *= s.xs[m][rem - q * n];
    rem = q;
  }
  return r * s.xs[from][rem];
}

// red[q][*], q < nb, summed by warp q into out[q].
__device__ __forceinline__ void reduce_slots(HShared& s, int nb, float* out) {
  __syncthreads();
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (wid < nb) {
    float a = 0.0f;
#pragma unroll
    for (int e = 0; e < kHT / 32; e++) a += s.red[wid][e * 32 + lane];
    a = warp_add(a);
    if (lane == 0) out[wid] = a;
  }
  __syncthreads();
}

// The sums over the warp's lanes of a[0..M-1], the kept values halved per
// exchange (M = 16: 16 shuffles instead of 80): lane L returns the sum of
// a[L / (32 / M)].
template <int M>
__device__ __forceinline__ float warp_add_many(float (&a)[M]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int h = M / 2, bit = 16; h >= 1; h >>= 1, bit >>= 1) {
    const bool up = lane & bit;
#pragma unroll
    for (int e = 0; e < h; e++) {
      const float mine = up ? a[e + h] : a[e], other = up ? a[e] : a[e + h];
      a[e] = mine + __shfl_xor_sync(0xFFFFFFFFu, other, bit);
    }
  }
  float r = a[0];
#pragma unroll
  for (int bit = 16 / M; bit >= 1; bit >>= 1) r += __shfl_xor_sync(0xFFFFFFFFu, r, bit);
  return r;
}

// The columns of rank's block, a range that starts on a multiple of VEC.
template <int VEC>
__device__ __forceinline__ void own_columns(int64_t cols, int rank, int cl, int64_t& ca, int64_t& cb) {
  ca = cols / VEC * rank / cl * VEC;
  cb = cols / VEC * (rank + 1) / cl * VEC;
}

// This block's part of z_0: its columns q of the n_0 x (n_1 ... n_{d-1}) view
// against x_1 (x) ... (x) x_{d-1}, formed once per thread for four of its
// columns and held in registers while the rows stream by.
template <int VEC>
__device__ void pass0(HShared& s, int rank, float* zp) {
  constexpr int RB = kHRows<VEC>;
  constexpr int NQ = 4 / VEC;  // chunks per thread held in registers
  const int t = threadIdx.x, wid = t >> 5, lane = t & 31;
  const int64_t n0 = s.it.dims[0];
  int64_t cols = 1, ca, cb;
  for (int m = 1; m < s.it.d; m++) cols *= s.it.dims[m];
  own_columns<VEC>(cols, rank, s.cl, ca, cb);
  if (ca >= cb) {
    for (int64_t i = t; i < n0; i += kHT) zp[i] = 0.0f;
    return;
  }
  const HTile tl = s.tile[1];
  const int ww = tl.w >> 5, ph = wid / ww, wc = wid - ph * ww;
  const int step = tl.w * VEC;  // columns per chunk
  float* const zw = &s.red[0][0];  // [wc][row] of a range of rows
  const int64_t span = kHSlots * kHT / ww / 4 * 4;
  for (int64_t R0 = 0; R0 < n0; R0 += span) {
    const int rows = (int)min(span, n0 - R0);
    int64_t r0, r1;
    phase_rows(rows, tl.P, ph, r0, r1);
    const int nr = (int)(r1 - r0), nbat = (nr + RB - 1) / RB, per = nbat > 0 ? (nr + nbat - 1) / nbat : 1;
    for (int64_t c0 = 0; c0 < tl.m && nr > 0; c0 += NQ) {
      const int64_t col0 = ca + c0 * step + (wc * 32 + lane) * VEC;
      const int nq = (int)min((int64_t)NQ, tl.m - c0);
      float coef[NQ][VEC];
#pragma unroll
      for (int q = 0; q < NQ; q++)
#pragma unroll
        for (int g = 0; g < VEC; g++) {
          const int64_t col = col0 + q * step + g;
          coef[q][g] = (q < nq && col < cb) ? outer_at(s, 1, col) : 0.0f;
        }
      for (int b = (int)r0; b < (int)r1; b += per) {
        const int nb = min(per, (int)r1 - b);
        const float* const p0 = s.it.A + (R0 + b) * cols + col0;
        float acc[RB];
#pragma unroll
        for (int e = 0; e < RB; e++) acc[e] = 0.0f;
#pragma unroll
        for (int q = 0; q < NQ; q++) {
          if (q < nq) {
            const float* p = p0 + q * step;
            const bool ok = col0 + q * step < cb;
            float v[RB][VEC];
#pragma unroll
            for (int e = 0; e < RB; e++, p += cols) {
#pragma unroll
              for (int g = 0; g < VEC; g++) v[e][g] = 0.0f;
              if (e < nb && ok) ld_row<VEC>(p, v[e]);
            }
#pragma unroll
            for (int e = 0; e < RB; e++)
#pragma unroll
              for (int g = 0; g < VEC; g++) acc[e] = __fmaf_rn(v[e][g], coef[q][g], acc[e]);
          }
        }
        const float sum = warp_add_many<RB>(acc);
        const int row = lane / (32 / RB);
        if (lane % (32 / RB) == 0 && row < nb) {
          float* o = zw + wc * rows + b + row;
          *o = c0 == 0 ? sum : *o + sum;
        }
      }
    }
    __syncthreads();
    for (int i = t; i < rows; i += kHT) {
      float z = zw[i];
      for (int q = 1; q < ww; q++) z += zw[q * rows + i];
      zp[R0 + i] = z;
    }
    __syncthreads();
  }
}

// Level j: this block's columns of W_j = src x_0 x_{j-1} (src: n_{j-1} rows
// of n_j * rest columns) into dst and its part of z_j into zp; at the last
// level W_j is z_j and goes to zp.  The chunks are walked from the last to
// the first: pass 0 and level 1 read the same columns, so level 1 starts with
// what the caches still hold.
template <int VEC>
__device__ void level(HShared& s, int j, int rank, const float* src, float* dst, float* zp) {
  const int t = threadIdx.x, wid = t >> 5, lane = t & 31;
  int64_t rest = 1, ca, cb;
  for (int m = j + 1; m < s.it.d; m++) rest *= s.it.dims[m];
  const int64_t nj = s.it.dims[j], cols = nj * rest;
  own_columns<VEC>(cols, rank, s.cl, ca, cb);
  const bool last = j == s.it.d - 1;
  if (!last)
    for (int64_t i = t; i < nj; i += kHT)
      if (ca >= cb || i < ca / rest || i * rest >= cb) zp[i] = 0.0f;
  if (ca >= cb) return;
  const HTile tl = s.tile[j];
  const int ww = tl.w >> 5, ph = wid / ww, ll = (wid - ph * ww) * 32 + lane;
  int64_t r0, r1;
  phase_rows(s.it.dims[j - 1], tl.P, ph, r0, r1);
  const float* const xc = s.xs[j - 1] + r0;
  float* out = last ? zp : dst;
  for (int64_t c = tl.m - 1; c >= 0; c--) {
    const int64_t cc = ca + (c * tl.w + ll) * VEC;
    const bool ok = cc < cb;
    float a[VEC] = {};
    if (ok) col_dot<VEC>(src + r0 * cols + cc, cols, xc, (int)(r1 - r0), a);
    if (tl.P > 1) {
      float* red = &s.red[0][0];
#pragma unroll
      for (int g = 0; g < VEC; g++) red[g * kHT + t] = a[g];
      __syncthreads();
      if (ph == 0)
        for (int q = 1; q < tl.P; q++)
#pragma unroll
          for (int g = 0; g < VEC; g++) a[g] += red[g * kHT + q * tl.w + t];
      __syncthreads();
    }
    if (ok && ph == 0) {
#pragma unroll
      for (int g = 0; g < VEC; g++) out[cc + g] = a[g];
    }
  }
  if (last) return;
  __syncthreads();  // the block's columns are written
  const int64_t ja = ca / rest, je = (cb - 1) / rest + 1;
  if (je - ja >= kHW) {  // short pieces: a warp each
    for (int64_t jj = ja + wid; jj < je; jj += kHW) {
      const int64_t la = max(ca - jj * rest, (int64_t)0), lb = min(cb - jj * rest, rest);
      float a = 0.0f;
      for (int64_t l = la + lane; l < lb; l += 32) a = __fmaf_rn(__ldcg(dst + jj * rest + l), outer_at(s, j + 1, l), a);
      a = warp_add(a);
      if (lane == 0) zp[jj] = a;
    }
  } else {
    for (int64_t jj = ja; jj < je; jj++) {
      const int64_t la = max(ca - jj * rest, (int64_t)0), lb = min(cb - jj * rest, rest);
      float a = 0.0f;
#pragma unroll 4
      for (int64_t l = la + t; l < lb; l += kHT) a = __fmaf_rn(__ldcg(dst + jj * rest + l), outer_at(s, j + 1, l), a);
      s.red[jj - ja][t] = a;
    }
    reduce_slots(s, (int)(je - ja), zp + ja);
  }
}

// x_j = z / ||z|| (FP64 norm) in this block's copy, z[i] the sum of the
// `parts` parts zp[r * n + i]; returns the norm.  A zero or non-finite norm
// leaves x_j as it was.
__device__ double normalize(HShared& s, int j, const float* zp, int parts) {
  const int t = threadIdx.x, wid = t >> 5;
  const int64_t n = s.it.dims[j];
  float* x = s.xs[j];
  float z0 = 0.0f;  // this thread's first entry (all of them when n <= kHT)
  double ss = 0.0;
  for (int64_t i = t; i < n; i += kHT) {
    float z = __ldcg(zp + i);
    for (int r = 1; r < parts; r++) z += __ldcg(zp + r * n + i);
    if (i < kHT) z0 = z;
    ss = fma((double)z, (double)z, ss);
  }
  const int nw = (int)min((int64_t)kHW, (n + 31) / 32);  // warps that hold entries
  if (wid < nw) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) ss += __shfl_xor_sync(0xFFFFFFFFu, ss, off);
    if ((t & 31) == 0) s.red64[wid] = ss;
  }
  __syncthreads();
  if (t == 0) {
    double sum = s.red64[0];
    for (int w = 1; w < nw; w++) sum += s.red64[w];
    const double sigma = sqrt(sum);
    s.red64[kHW] = sigma;
    s.red64[kHW + 1] = 1.0 / sigma;
  }
  __syncthreads();
  const double sigma = s.red64[kHW], inv = s.red64[kHW + 1];
  if (isfinite(sigma) && sigma > 0.0) {
    if (t < n) x[t] = (float)((double)z0 * inv);
    for (int64_t i = t + kHT; i < n; i += kHT) {
      float z = __ldcg(zp + i);
      for (int r = 1; r < parts; r++) z += __ldcg(zp + r * n + i);
      x[i] = (float)((double)z * inv);
    }
  }
  __syncthreads();
  return sigma;
}

struct HScratch {
  float* base;
  int64_t slen, zlen, xlen;  // per cluster of cl blocks: 2 W buffers, 2 * cl parts, cl blocks' vectors
  int cl;
};

__global__ void __launch_bounds__(kHT, 2) hopm_batched_kernel(const HItem* __restrict__ items, int count, int iters,
                                                            int* counter, int* slots, HScratch sc) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  HShared& s = *reinterpret_cast<HShared*>(smem_raw);
  const int rank = (int)cluster_rank();
  const int64_t cid = cluster_id();
  float* W[2];
  float* Z[2];
  const int cl = sc.cl;
  W[0] = sc.base + cid * (2 * sc.slen + cl * (2 * sc.zlen + sc.xlen));
  W[1] = W[0] + sc.slen;
  Z[0] = W[1] + sc.slen;
  Z[1] = Z[0] + cl * sc.zlen;
  float* xpriv = Z[1] + cl * sc.zlen + rank * sc.xlen;
  int* slot = slots + 2 * cid;
  int zb = 0;
  if (threadIdx.x == 0) s.cl = cl;
  for (int g = 0;; g ^= 1) {
    if (rank == 0 && threadIdx.x == 0) slot[g] = atomicAdd(counter, 1);
    cluster_sync();
    const int b = __ldcg(slot + g);
    if (b >= count) break;
    if (threadIdx.x < sizeof(HItem) / sizeof(int))
      reinterpret_cast<int*>(&s.it)[threadIdx.x] = reinterpret_cast<const int*>(items + b)[threadIdx.x];
    __syncthreads();
    const int d = s.it.d;
    if (threadIdx.x < d) {
      const int j = threadIdx.x;
      int64_t cols = 1, at = 0, all = 0;
      for (int m = j; m < d; m++) cols *= s.it.dims[m];
      for (int m = 0; m < d; m++) {
        const int64_t len = (s.it.dims[m] + 3) / 4 * 4;  // 16-byte aligned vectors
        if (m < j) at += len;
        all += len;
      }
      if (j == 1) {
        // widest loads that every row start of A allows
        const uintptr_t a = reinterpret_cast<uintptr_t>(s.it.A);
        s.vec = (cols % 4 == 0 && a % 16 == 0) ? 4 : (cols % 2 == 0 && a % 8 == 0) ? 2 : 1;
        cols /= s.vec;
      }
      if (j > 0) s.tile[j] = pick_tile(cols * (rank + 1) / s.cl - cols * rank / s.cl, s.it.dims[j - 1]);
      s.xs[j] = (all <= kHXCap ? s.x : xpriv) + at;
    }
    __syncthreads();
    for (int m = 0; m < d; m++)
      for (int64_t i = threadIdx.x; i < s.it.dims[m]; i += kHT) s.xs[m][i] = s.it.x[m][i];
    __syncthreads();
    int status = TVC_OK;
    double sigma = 0.0;
    for (int it = 0; it < iters && status == TVC_OK; it++) {
      const float* src = s.it.A;
      for (int j = 0; j < d && status == TVC_OK; j++) {
        const int64_t nj = s.it.dims[j];
        float* const zp = j == d - 1 ? Z[zb] : Z[zb] + rank * nj;
        if (j == 0) {
          if (s.vec == 4)
            pass0<4>(s, rank, zp);
          else if (s.vec == 2)
            pass0<2>(s, rank, zp);
          else
            pass0<1>(s, rank, zp);
        } else {
          float* const dst = W[j & 1];
          if (j > 1 || s.vec == 1)
            level<1>(s, j, rank, src, dst, zp);
          else if (s.vec == 4)
            level<4>(s, j, rank, src, dst, zp);
          else
            level<2>(s, j, rank, src, dst, zp);
          src = dst;
        }
        cluster_sync();
        sigma = normalize(s, j, Z[zb], j == d - 1 ? 1 : cl);
        zb ^= 1;
        if (!isfinite(sigma)) status = TVC_ERR_NONFINITE;
        else if (sigma == 0.0) status = TVC_ERR_ZERO_NORM;
      }
    }
    if (rank == 0 && iters > 0) {
      for (int m = 0; m < d; m++)
        for (int64_t i = threadIdx.x; i < s.it.dims[m]; i += kHT) s.it.x[m][i] = s.xs[m][i];
    }
    if (rank == 0 && threadIdx.x == 0) {
      if (s.it.lam) *s.it.lam = sigma;
      if (s.it.status) *s.it.status = status;
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------ host --

struct HLayout {
  size_t off_counter = 0, off_slots = 0, off_items = 0, off_scratch = 0, total = 0;
  HScratch sc{};
  int clusters = 0;
  bool block = false;             // one block per tensor
  int64_t slen = 0, zlen = 0;     // its scratch
};

// Batches of small tensors run one block per tensor (batched_hopm_block.cu): all
// tensors of at most 65536 elements, or 64 or more of at most 220000; matrices of
// at most 10000, or 32 or more of at most 40000.  ms of 5 sweeps, blocks /
// clusters: 4096 of 3..6 per mode 0.86 / 2.9, 512 of 8..32 0.19 / 0.92, 4096 of 30..60
// 3.3 / 6.7, 64 of 30..60 0.29 / 0.34; beyond the line one of 48^3 0.16 / 0.13, 64 of
// 64^3 0.60 / 0.33, 8 matrices of 20..200 0.12 / 0.09 (64 of them 0.19 / 0.43), 304 of
// 100..500 1.0 / 0.57.
bool block_wanted(const hopm_batch_desc* d, int count) {
  for (int b = 0; b < count; b++) {
    int64_t N = 1;
    for (int m = 0; m < d[b].order; m++) N *= d[b].dims[m];
    const bool matrix = d[b].order == 2;
    if (N > (matrix ? 10000 : 65536) && (count < (matrix ? 32 : 64) || N > (matrix ? 40000 : 220000))) return false;
  }
  return true;
}

HLayout layout_hopm(const hopm_batch_desc* d, int count) {
  HLayout L;
  L.off_slots = 256;
  if (block_wanted(d, count)) {
    L.block = true;
    for (int b = 0; b < count; b++) {
      int64_t N = 1, least = d[b].dims[0];
      for (int m = 0; m < d[b].order; m++) {
        N *= d[b].dims[m];
        least = std::min(least, d[b].dims[m]);
        L.zlen = std::max(L.zlen, d[b].dims[m]);
      }
      L.slen = std::max(L.slen, N / least);
    }
    L.slen = (int64_t)align_up((size_t)L.slen, 64);
    L.zlen = (int64_t)align_up((size_t)L.zlen, 64);
    L.off_items = L.off_slots;
    L.off_scratch = L.off_items + align_up((size_t)std::max(1, count) * sizeof(HItem), 256);
    L.total = L.off_scratch + hopm_block_ws_bytes(L.slen, L.zlen);
    return L;
  }
  int64_t slen = 1, zlen = 1, xlen = 0, total = 0, largest = 1;
  for (int b = 0; b < count; b++) {
    int64_t N = 1, sum = 0;
    for (int m = 0; m < d[b].order; m++) {
      N *= d[b].dims[m];
      sum += (d[b].dims[m] + 3) / 4 * 4;
      zlen = std::max(zlen, d[b].dims[m]);
    }
    total += N;
    largest = std::max(largest, N);
    slen = std::max(slen, N / d[b].dims[0]);
    if (sum > kHXCap) xlen = std::max(xlen, sum);
  }
  L.sc.slen = (int64_t)align_up((size_t)slen, 64);
  L.sc.zlen = (int64_t)align_up((size_t)zlen, 64);
  L.sc.xlen = (int64_t)align_up((size_t)xlen, 64);
  // Blocks per cluster: the widest clusters finish one tensor soonest (each
  // block streams about 15 GB/s of it), narrower ones meet at fewer and
  // cheaper barriers.  Halve while the clusters resident at once would still
  // share the whole batch more evenly than its largest tensor: 10 sweeps of
  // 512 tensors with 16 / 8 / 4 / 2 blocks 51 / 36 / 33 / 49 ms (rule: 4),
  // 283 tensors 32 / 22 / 26 / 46 ms (8), 5 sweeps of 73 tensors 4.1 / 5.2 /
  // 9.5 / 18 ms (16).
  const int blocks = 2 * device_sms();
  int cl = 16;
  while (cl > 2 && 1.25 * (double)largest * (blocks / (cl / 2)) < (double)total) cl /= 2;
  L.sc.cl = cl;
  L.clusters = std::max(1, std::min(count, blocks / cl));
  L.off_items = L.off_slots + align_up((size_t)L.clusters * 2 * sizeof(int), 256);
  L.off_scratch = L.off_items + align_up((size_t)std::max(1, count) * sizeof(HItem), 256);
  L.total = L.off_scratch + (size_t)L.clusters *
                                (2 * L.sc.slen + cl * (2 * L.sc.zlen + L.sc.xlen)) * sizeof(float) + 16;
  return L;
}

// Attributes of the cluster kernel, once per device.
cudaError_t prepare_kernel() {
  static std::mutex mu;
  static std::set<int> done;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lk(mu);
  if (done.count(dev)) return cudaSuccess;
  e = cudaFuncSetAttribute(hopm_batched_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(HShared));
  if (e == cudaSuccess)  // clusters of 16
    e = cudaFuncSetAttribute(hopm_batched_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess) done.insert(dev);
  return e;
}

}  // namespace
}  // namespace tvcg

using namespace tvcg;

extern "C" size_t hopm_batched_workspace_size(const hopm_batch_desc* descs, int count) {
  if (count < 0 || (count > 0 && !descs)) return 0;
  for (int b = 0; b < count; b++)
    if (descs[b].order < 2 || check_dims(descs[b].order, descs[b].dims, nullptr) != TVC_OK) return 0;
  return layout_hopm(descs, count).total;
}

extern "C" tvc_status hopm_batched(const hopm_batch_desc* descs, int count, int iters, int flags, void* workspace,
                                   size_t ws_bytes, tvc_stream_t stream) {
  if (count < 0 || iters < 0 || !descs) return TVC_ERR_INVALID_ARG;
  if (count == 0) return TVC_OK;
  for (int b = 0; b < count; b++) {
    if (descs[b].order < 2 || !descs[b].A || check_dims(descs[b].order, descs[b].dims, nullptr) != TVC_OK)
      return TVC_ERR_INVALID_ARG;
    for (int m = 0; m < descs[b].order; m++)
      if (!descs[b].x[m]) return TVC_ERR_INVALID_ARG;
  }
  const HLayout L = layout_hopm(descs, count);
  if (!workspace || ws_bytes < L.total) return TVC_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  char* w = static_cast<char*>(workspace);
  if (!(flags & TVC_BATCH_PREUPLOADED)) {
    std::vector<std::pair<int64_t, int>> order;
    for (int b = 0; b < count; b++) {
      int64_t N = 1;
      for (int m = 0; m < descs[b].order; m++) N *= descs[b].dims[m];
      order.push_back({N, b});
    }
    std::stable_sort(order.begin(), order.end(), [](auto& a, auto& b) { return a.first > b.first; });
    std::vector<HItem> items;
    for (auto& pr : order) {
      const hopm_batch_desc& e = descs[pr.second];
      HItem it{};
      it.A = e.A;
      it.d = e.order;
      for (int m = 0; m < e.order; m++) {
        it.dims[m] = e.dims[m];
        it.x[m] = e.x[m];
      }
      it.lam = e.lambda_out;
      it.status = e.status_out;
      items.push_back(it);
    }
    if (cudaMemcpyAsync(w + L.off_items, items.data(), items.size() * sizeof(HItem), cudaMemcpyHostToDevice, st) !=
        cudaSuccess)
      return TVC_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return TVC_ERR_CUDA;
  }
  if (L.block) {
    cudaMemsetAsync(w + L.off_counter, 0, sizeof(int), st);
    count_launches(1);
    return cuda_status(hopm_block_launch(reinterpret_cast<const HItem*>(w + L.off_items), count, iters,
                                         reinterpret_cast<int*>(w + L.off_counter),
                                         reinterpret_cast<float*>(w + L.off_scratch), L.slen, L.zlen, st));
  }
  if (prepare_kernel() != cudaSuccess) return cuda_status(cudaGetLastError());
  cudaMemsetAsync(w + L.off_counter, 0, sizeof(int), st);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(L.clusters * L.sc.cl));
  cfg.blockDim = dim3(kHT);
  cfg.dynamicSmemBytes = sizeof(HShared);
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = L.sc.cl;
  at.val.clusterDim.y = 1;
  at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  HScratch sc = L.sc;
  // vectors in memory are read in 16-byte pieces, whatever the workspace's own alignment
  sc.base = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(w + L.off_scratch) + 15) & ~(uintptr_t)15);
  const cudaError_t e =
      cudaLaunchKernelEx(&cfg, hopm_batched_kernel, reinterpret_cast<const HItem*>(w + L.off_items), count, iters,
                         reinterpret_cast<int*>(w + L.off_counter), reinterpret_cast<int*>(w + L.off_slots), sc);
  count_launches(1);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return cuda_status(e);
  }
  return cuda_status(cudaGetLastError());
}
