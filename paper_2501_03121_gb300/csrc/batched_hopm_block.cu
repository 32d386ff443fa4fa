// Power methods of many small FP32 tensors in one persistent launch, one block
// per tensor (largest first, pulled from an atomic counter); larger ones run in
// clusters (batched_hopm.cu, which says where the line lies).
//
// A sweep has the schedule of the single power method, every step a block-wide
// contraction behind a block barrier.  Bound: latency, hidden by six tensors per
// SM (clusters of blocks of 512 threads hold two blocks per SM and pay for the
// cluster barrier and their column tiling on every phase).
#include "common.cuh"
#include "internal.h"

namespace tvcg {
namespace {

constexpr int kT = 256;           // threads per block
constexpr int kBlocksPerSM = 6;

// y[o] = sum_j A[(i*nk + j)*v + l] x[j], o = i*v + l < u*v; G lanes per output.
__device__ void blk_tvc(const float* __restrict__ A, int64_t u, int64_t nk, int64_t v, const float* __restrict__ x,
                        float* __restrict__ y, int G) {
  const int64_t uv = u * v;
  if (v >= 2) {
    // One thread per output o = (i, l): the pair is found by one division
    // and then advanced by the block stride; sixteen rows of n_k in flight
    // through pointer increments (one block streams at the rate its bytes in
    // flight allow), only the last (< 8) rows predicated.
    int64_t o = threadIdx.x;
    if (o >= uv) return;
    int64_t i = o / v, l = o - i * v;
    const int64_t stride = kT;
    const int64_t di = stride / v, dl = stride - di * v;
    for (; o < uv; o += stride) {
      const float* p = A + i * nk * v + l;
      float acc0 = 0.0f, acc1 = 0.0f;
      int64_t jj = 0;
      for (; jj + 16 <= nk; jj += 16, p += 16 * v) {  // 16 rows in flight (64 B per thread)
        float av[16];
#pragma unroll
        for (int q = 0; q < 16; q++) av[q] = __ldcs(p + q * v);
#pragma unroll
        for (int q = 0; q < 16; q += 2) {
          acc0 = __fmaf_rn(av[q], __ldg(x + jj + q), acc0);
          acc1 = __fmaf_rn(av[q + 1], __ldg(x + jj + q + 1), acc1);
        }
      }
      if (jj + 8 <= nk) {
        float av[8];
#pragma unroll
        for (int q = 0; q < 8; q++) av[q] = __ldcs(p + q * v);
#pragma unroll
        for (int q = 0; q < 8; q += 2) {
          acc0 = __fmaf_rn(av[q], __ldg(x + jj + q), acc0);
          acc1 = __fmaf_rn(av[q + 1], __ldg(x + jj + q + 1), acc1);
        }
        jj += 8;
        p += 8 * v;
      }
      if (jj < nk) {
        float av[7];
#pragma unroll
        for (int q = 0; q < 7; q++) av[q] = (jj + q < nk) ? __ldcs(p + q * v) : 0.0f;
#pragma unroll
        for (int q = 0; q < 7; q++)
          if (jj + q < nk) acc0 = __fmaf_rn(av[q], __ldg(x + jj + q), acc0);
      }
      y[o] = acc0 + acc1;
      i += di;
      l += dl;
      if (l >= v) {
        l -= v;
        i++;
      }
    }
    return;
  }
  // v == 1 (rows): a group of G lanes per row, eight predicated loads in
  // flight per lane (short rows too), shuffle reduction.
  const int lane = threadIdx.x & 31;
  const int p = lane & (G - 1);
  const int gw = 32 / G;  // groups per warp
  const int64_t ngroups = (int64_t)(kT / 32) * gw;
  for (int64_t base = (int64_t)(threadIdx.x >> 5) * gw; base < uv; base += ngroups) {
    const int64_t o = base + lane / G;
    float acc = 0.0f;
    if (o < uv) {
      const float* row = A + o * nk;
      for (int64_t j = p; j < nk; j += 8 * G) {
        float av[8], xv[8];
#pragma unroll
        for (int q = 0; q < 8; q++) {
          const bool ok = j + q * G < nk;
          av[q] = ok ? __ldcs(row + j + q * G) : 0.0f;
          xv[q] = ok ? __ldg(x + j + q * G) : 0.0f;
        }
#pragma unroll
        for (int q = 0; q < 8; q++) acc = __fmaf_rn(av[q], xv[q], acc);
      }
    }
    for (int off = G / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, off);
    if (o < uv && p == 0) y[o] = acc;
  }
}

// The power method's two passes over A (v >= 2): where v is even and A is
// 8-byte aligned each thread takes two adjacent outputs and loads pairs,
// twice the bytes in flight per thread for the same sixteen rows (a block
// of the register-held contraction streams at the rate its bytes in flight
// allow); otherwise blk_tvc.
__device__ void blk_tvc_pass(const float* __restrict__ A, int64_t u, int64_t nk, int64_t v,
                             const float* __restrict__ x, float* __restrict__ y, int G) {
  if (v % 2 != 0 || (reinterpret_cast<uintptr_t>(A) & 7) != 0) {
    blk_tvc(A, u, nk, v, x, y, G);
    return;
  }
  const int64_t uv2 = u * v / 2;  // output pairs
  int64_t q2 = threadIdx.x;
  if (q2 >= uv2) return;
  const int64_t v2 = v / 2;
  int64_t i = q2 / v2, l = 2 * (q2 - i * v2);
  const int64_t di = kT / v2, dl = 2 * (kT - di * v2);
  for (; q2 < uv2; q2 += kT) {
    const float* p = A + i * nk * v + l;
    float a0 = 0.0f, a1 = 0.0f;
    int64_t jj = 0;
    for (; jj + 16 <= nk; jj += 16, p += 16 * v) {
      float2 av[16];
#pragma unroll
      for (int q = 0; q < 16; q++) av[q] = __ldcs(reinterpret_cast<const float2*>(p + q * v));
#pragma unroll
      for (int q = 0; q < 16; q++) {
        const float xv = __ldg(x + jj + q);
        a0 = __fmaf_rn(av[q].x, xv, a0);
        a1 = __fmaf_rn(av[q].y, xv, a1);
      }
    }
    for (; jj < nk; jj++, p += v) {
      const float2 av = __ldcs(reinterpret_cast<const float2*>(p));
      const float xv = __ldg(x + jj);
      a0 = __fmaf_rn(av.x, xv, a0);
      a1 = __fmaf_rn(av.y, xv, a1);
    }
    y[i * v + l] = a0;
    y[i * v + l + 1] = a1;
    i += di;
    l += dl;
    if (l >= v) {
      l -= v;
      i++;
    }
  }
}

// w[c] = prod_{m < nm} x_m[digit_m(c)]
__device__ void blk_outer(float* w, int nm, const int64_t* dims, float* const* xs) {
  int64_t len = 1;
  for (int m = 0; m < nm; m++) len *= dims[m];
  for (int64_t c = threadIdx.x; c < len; c += kT) {
    int64_t rem = c;
    float acc = 1.0f;
    int64_t dig[TVC_MAX_ORDER];
    for (int m = nm - 1; m >= 0; m--) {
      dig[m] = rem % dims[m];
      rem /= dims[m];
    }
    acc = xs[0][dig[0]];
    for (int m = 1; m < nm; m++) acc *= xs[m][dig[m]];
    w[c] = acc;
  }
}

// x = z / ||z|| with the norm in FP64; returns the norm (all threads).
__device__ double blk_normalize(const float* z, float* x, int64_t n, double* red) {
  double s = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += kT) s = fma((double)z[i], (double)z[i], s);
  red[threadIdx.x] = s;
  __syncthreads();
  for (int off = kT / 2; off > 0; off >>= 1) {
    if ((int)threadIdx.x < off) red[threadIdx.x] += red[threadIdx.x + off];
    __syncthreads();
  }
  const double sigma = sqrt(red[0]);
  __syncthreads();
  if (isfinite(sigma) && sigma > 0.0)
    for (int64_t i = threadIdx.x; i < n; i += kT) x[i] = (float)((double)z[i] / sigma);
  __syncthreads();
  return sigma;
}

// Lanes per row of the contraction of a matrix with x_1.
__device__ __forceinline__ int rows_G(int64_t nk) { return nk >= 64 ? 32 : 8; }

// One block runs every sweep of one tensor's power method (the schedule of
// the single-tensor path: T = A x_1 x_1, W_1 = A x_0 x_0, W_j = W_{j-1} x_{j-1} ...,
// the trailing contractions against the outer product of the trailing
// vectors).  scratch: per block, 3 buffers of `slen` floats plus z.
__global__ void __launch_bounds__(kT) hopm_block_kernel(const HopmItem* __restrict__ items, int count, int iters,
                                                            int* counter, float* scratch, int64_t slen, int64_t zlen) {
  __shared__ int slot;
  __shared__ double red[kT];
  float* S1 = scratch + (int64_t)blockIdx.x * (3 * slen + zlen);
  float* S2 = S1 + slen;
  float* Wv = S2 + slen;
  float* z = Wv + slen;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) slot = atomicAdd(counter, 1);
    __syncthreads();
    const int b = slot;
    if (b >= count) break;
    const HopmItem& it = items[b];
    const int d = it.d;
    const int64_t* n = it.dims;
    int64_t N = 1;
    for (int m = 0; m < d; m++) N *= n[m];
    int status = TVC_OK;
    double sigma = 0.0;
    for (int t = 0; t < iters && status == TVC_OK; t++) {
      float* prev = S1;
      float* next = S2;
      for (int j = 0; j < d && status == TVC_OK; j++) {
        const float* zz = z;
        if (d == 2) {
          // z_j = A x_{1-j} x_{1-j}
          if (j == 0)
            blk_tvc(it.A, n[0], n[1], 1, it.x[1], z, rows_G(n[1]));
          else
            blk_tvc(it.A, 1, n[0], n[1], it.x[0], z, 1);
        } else if (j < 2) {
          int64_t rest2 = 1;
          for (int m = 2; m < d; m++) rest2 *= n[m];
          if (j == 0)
            blk_tvc_pass(it.A, n[0], n[1], rest2, it.x[1], S1, rows_G(n[1]));  // T = A x_1 x_1
          else
            blk_tvc_pass(it.A, 1, n[0], N / n[0], it.x[0], S1, 1);  // W_1 = A x_0 x_0
          __syncthreads();
          const float* wvec = it.x[2];
          if (d > 3) {
            blk_outer(Wv, d - 2, n + 2, it.x + 2);
            __syncthreads();
            wvec = Wv;
          }
          blk_tvc(S1, n[j], rest2, 1, wvec, z, 32);
          prev = S1;
          next = S2;
        } else {
          int64_t rest = 1;
          for (int m = j; m < d; m++) rest *= n[m];
          blk_tvc(prev, 1, n[j - 1], rest, it.x[j - 1], next, 1);  // W_j = W_{j-1} x_{j-1}
          __syncthreads();
          if (j == d - 1) {
            zz = next;
          } else {
            const float* wvec = it.x[d - 1];
            if (j < d - 2) {
              blk_outer(Wv, d - j - 1, n + j + 1, it.x + j + 1);
              __syncthreads();
              wvec = Wv;
            }
            blk_tvc(next, n[j], rest / n[j], 1, wvec, z, 32);
          }
          float* tmp = prev;
          prev = next;
          next = tmp;
        }
        __syncthreads();
        sigma = blk_normalize(zz, it.x[j], n[j], red);
        if (!isfinite(sigma)) status = TVC_ERR_NONFINITE;
        else if (sigma == 0.0) status = TVC_ERR_ZERO_NORM;
      }
    }
    if (threadIdx.x == 0) {
      if (it.lam) *it.lam = sigma;
      if (it.status) *it.status = status;
    }
  }
}

}  // namespace

size_t hopm_block_ws_bytes(int64_t slen, int64_t zlen) {
  return (size_t)device_sms() * kBlocksPerSM * (size_t)(3 * slen + zlen) * sizeof(float);
}

cudaError_t hopm_block_launch(const HopmItem* items, int count, int iters, int* counter, float* scratch, int64_t slen,
                              int64_t zlen, cudaStream_t st) {
  hopm_block_kernel<<<device_sms() * kBlocksPerSM, kT, 0, st>>>(items, count, iters, counter, scratch, slen, zlen);
  return cudaGetLastError();
}

}  // namespace tvcg
