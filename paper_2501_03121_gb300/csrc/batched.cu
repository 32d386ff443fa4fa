// Batched contractions and adjoints over many independent FP32 tensors of
// uneven order and shape, each batch in one persistent launch (the GPU
// counterpart of the paper's task-based execution, Section 4.3, where many
// TVCs overlap instead of joining after each one); the batched power method
// is in batched_hopm.cu.
//
// The host cuts every tensor (largest first) into work items and uploads the
// descriptors and items into the workspace; a persistent kernel of a few
// blocks per SM pulls items from an atomic work counter.  Where a tensor
// wants gx and another of its results, one item computes all of them for a
// range of columns (v >= 32) or rows (v == 1) from one read of A; the other
// cases have an item kind per result.  gx items of one tensor leave partial
// sums that the tensor's last item adds in a fixed order.  With
// TVC_BATCH_PREUPLOADED the descriptors of a previous call are reused and a
// call issues only a memset and one kernel, so it can be captured in a CUDA
// graph and replayed.
//
// Forward contraction of rows v == 1: a group of G lanes (G a power of two
// <= 32) computes one output, its lanes splitting the row; the autotuner
// picks G per shape class (n_k rounded to a power of two) by timing the
// candidates, untuned classes use a fixed rule.  For v >= 2 one thread
// computes one output, coalesced along l.
#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "common.cuh"
#include "internal.h"

namespace tvcg {
namespace {

constexpr int kBBT = 256;        // threads per block
constexpr int kBBlocksPerSM = 4;

struct BItem {
  const float* A;
  const float* x;
  float* y;
  const float* gy;
  float* gx;
  float* gA;
  int64_t u, nk, v;
  int gf;         // lanes per output of the forward contraction
  int gxk;        // gx items (slab ranges) of this tensor
  int64_t gxp;    // their partials: floats [gxp, gxp + gxk * nk) of the partial area (gxk > 1)
};

// ---------------------------------------------------- block-level routines

// Rows [r0, r1) of a matrix of rows of nk elements against x: G lanes (a
// power of two) per row, Q loads per lane and row and 16 / Q rows per group
// in flight, shuffle reduction.
template <int Q>
__device__ void blk_rows(const float* __restrict__ A, int64_t nk, const float* __restrict__ x, float* __restrict__ y,
                         int G, int64_t r0, int64_t r1) {
  constexpr int B = 16 / Q;
  const int lane = threadIdx.x & 31, p = lane & (G - 1), gw = 32 / G;
  for (int64_t base = r0 + (int64_t)(threadIdx.x >> 5) * gw * B; base < r1; base += (int64_t)(kBBT / 32) * gw * B) {
    const int64_t row0 = base + lane / G;
    float acc[B];
#pragma unroll
    for (int b = 0; b < B; b++) acc[b] = 0.0f;
    for (int64_t j = p; j - p < nk; j += Q * G) {
      float av[B][Q], xv[Q];
#pragma unroll
      for (int q = 0; q < Q; q++) {
        const bool in = j + q * G < nk;
        xv[q] = in ? __ldg(x + j + q * G) : 0.0f;
#pragma unroll
        for (int b = 0; b < B; b++)
          av[b][q] = (in && row0 + b * gw < r1) ? __ldcs(A + (row0 + b * gw) * nk + j + q * G) : 0.0f;
      }
#pragma unroll
      for (int b = 0; b < B; b++)
#pragma unroll
        for (int q = 0; q < Q; q++) acc[b] = __fmaf_rn(av[b][q], xv[q], acc[b]);
    }
    for (int off = G / 2; off > 0; off >>= 1) {
#pragma unroll
      for (int b = 0; b < B; b++) acc[b] += __shfl_xor_sync(0xFFFFFFFFu, acc[b], off);
    }
#pragma unroll
    for (int b = 0; b < B; b++)
      if (p == 0 && row0 + b * gw < r1) y[row0 + b * gw] = acc[b];
  }
}

// y[o] = sum_j A[(i*nk + j)*v + l] x[j], o = i*v + l < u*v; G lanes per output.
__device__ void blk_tvc(const float* __restrict__ A, int64_t u, int64_t nk, int64_t v, const float* __restrict__ x,
                        float* __restrict__ y, int G, int64_t o_begin = 0, int64_t o_end = -1) {
  const int64_t uv = (o_end < 0) ? u * v : o_end;
  if (v >= 2) {
    // One thread per output o = (i, l): the pair is found by one division
    // and then advanced by the block stride; sixteen rows of n_k in flight
    // through pointer increments (one block streams at the rate its bytes in
    // flight allow), only the last (< 8) rows predicated.
    int64_t o = o_begin + threadIdx.x;
    if (o >= uv) return;
    int64_t i = o / v, l = o - i * v;
    const int64_t stride = kBBT;
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
  // v == 1 (rows): a group of G lanes per row, Q loads per lane and row
  const int64_t q = (nk + G - 1) / G;
  if (q <= 1)
    blk_rows<1>(A, nk, x, y, G, o_begin, uv);
  else if (q <= 2)
    blk_rows<2>(A, nk, x, y, G, o_begin, uv);
  else if (q <= 4)
    blk_rows<4>(A, nk, x, y, G, o_begin, uv);
  else
    blk_rows<8>(A, nk, x, y, G, o_begin, uv);
}

// gA[(i*nk + j)*v + l] = gy[i*v + l] * x[j] over slabs i in [i0, i1) and
// rows j in [j0, j1), with coalesced stores: threads own columns l (v >= 32)
// or positions q = j*v + l of the slab (v < 32, whole slabs).
__device__ void blk_gA(const float* __restrict__ gy, const float* __restrict__ x, float* __restrict__ gA, int64_t nk,
                       int64_t v, int64_t i0, int64_t i1, int64_t j0, int64_t j1) {
  if (v >= 32) {
    for (int64_t l = threadIdx.x; l < v; l += kBBT)
      for (int64_t i = i0; i < i1; i++) {
        const float g = __ldg(gy + i * v + l);
        float* p = gA + (i * nk + j0) * v + l;
        for (int64_t j = j0; j < j1; j++, p += v) __stcs(p, g * __ldg(x + j));
      }
  } else {
    // columns q = j*v + l of the slab; slabs narrower than the block are
    // written by several phases of threads
    const int64_t S = nk * v;
    const int CW = (int)min(S, (int64_t)kBBT), P = kBBT / CW;
    const int ph = threadIdx.x / CW, cc = threadIdx.x - ph * CW;
    for (int64_t q = cc; ph < P && q < S; q += CW) {
      const int64_t j = q / v, l = q - j * v;
      const float xj = __ldg(x + j);
#pragma unroll 8
      for (int64_t i = i0 + ph; i < i1; i += P) __stcs(gA + i * S + q, __ldg(gy + i * v + l) * xj);
    }
  }
}

__device__ int grab(int* counter, int* slot) {
  __syncthreads();
  if (threadIdx.x == 0) *slot = atomicAdd(counter, 1);
  __syncthreads();
  return *slot;
}

// ------------------------------------------------------------ the kernels

// A unit of work: kind 0 = outputs [a0, a1) of the forward contraction,
// 1 = gx over slabs [a0, a1) and rows j in [c0, c1) (slab range e0 of the
// tensor's gxk, e1 gx items in all), 2 = gA over slabs [a0, a1) and rows
// [c0, c1), 3 = every wanted result over the columns [a0, a1), 4 = every
// wanted result over the rows i in [a0, a1) of v == 1 (e0, e1 as for gx), 5 =
// gx and gA over a rectangle (v < 32).
struct WItem {
  int b, kind;
  int64_t a0, a1, c0, c1;
  int e0, e1;
};

// gx over a rectangle of one tensor: slabs [i0, i1) x rows j in [j0, j1)
// (item ks of the tensor's gxk slab ranges):
//   part[j] = sum_{i in [i0,i1), l < v} A[(i*nk + j)*v + l] gy[i*v + l].
// Rows of v >= 32 go to warps: warp w takes the slabs i = i0 + w (mod 8) of
// every j (or, when the item has fewer than 8 slabs, the w-th 32-aligned
// segment of every row), lanes stride over l; each warp's sum for j (FP32
// folded every 64 products into a compensated pair, then a fixed xor tree) goes
// to red[w][j - j0] and the 8 warp sums are added in w order (j1 - j0 <=
// kGxJ).  Rows of v < 32 go to columns: the item's columns c = j*v + l
// (contiguous in every slab) are taken in chunks of at most kBBT; a chunk
// narrower than the block gives the spare threads alternate slabs (phases).
// Each thread streams its column down its slabs (eight in flight, folded
// every 64 slabs), the phases of a column are added in phase order and the
// columns of a j in l order.  With gxk > 1 the slab ranges write partials
// [ks][j] and the tensor's last item to finish (counted per tensor) sums them
// in slab-range order into gx and resets the counter: deterministic, no
// waiting.
constexpr int64_t kGxWarpRows = 32;  // v at or above which rows go to warps
constexpr int64_t kGxJ = 256;        // rows j per warp-mapped item
constexpr int kFusedRows = 512;      // rows n_k up to which columns are fused
constexpr int kFusedRowMax = 256;    // row lengths of the fused rows (v == 1)
constexpr int kFusedRowMin = 32;
// A warp's row sums of a fused item are compensated pairs, the errors kErr
// behind the sums.  More than kErr rows need none: the item is then at most
// 1024 columns (fused_per), one sum per warp and row.
constexpr int kErr = kFusedRows / 2;
static_assert(kFusedRowMax <= kErr && (1 << 19) / (kErr + 1) < 2 * 1024, "one sum per row above kErr rows");

// A term into a compensated pair (p[0], p[kErr]), and a pair (or its sum alone)
// into a compensated sum.
__device__ __forceinline__ void add_pair(float* p, float v) {
  float t, err;
  two_sum(p[0], v, t, err);
  p[0] = t;
  p[kErr] = __fadd_rn(p[kErr], err);
}
__device__ __forceinline__ void add_pair(KahanF32& s, const float* p, bool pair) {
  s.add(p[0]);
  if (pair) s.add(p[kErr] == p[kErr] ? p[kErr] : 0.0f);  // NaN: p[0] alone (see pair_value)
}

// After an item's partial sums of gx are written: the tensor's last item
// adds the gxk partials in order and resets the counter.
__device__ void finish_gx(const BItem& it, int items, int* cnt, const float* partials, int* flag) {
  if (it.gxk <= 1) return;
  const int t = threadIdx.x;
  __threadfence();
  __syncthreads();
  if (t == 0) *flag = (atomicAdd(cnt, 1) == items - 1);
  __syncthreads();
  if (*flag) {
    __threadfence();
    const float* Pp = partials + it.gxp;
    for (int64_t j = t; j < it.nk; j += kBBT) {
      KahanF32 sum;
#pragma unroll 8
      for (int q = 0; q < it.gxk; q++) sum.add(__ldcg(Pp + (int64_t)q * it.nk + j));
      it.gx[j] = sum.value();
    }
    if (t == 0) *cnt = 0;  // ready for the next launch
  }
  __syncthreads();
}

// gA (nullable): rows of v < 32 also write gA over the rectangle.
__device__ void blk_gx_rect(const BItem& it, float* __restrict__ gA, int64_t i0, int64_t i1, int64_t j0, int64_t j1, int ks, int items,
                            int* cnt, float* partials, float* red, int* flag) {
  const int64_t S = it.nk * it.v, v = it.v;
  float* dst = (it.gxk > 1) ? partials + it.gxp + (int64_t)ks * it.nk : it.gx;
  const int t = threadIdx.x;
  if (v >= kGxWarpRows) {
    const int w = t >> 5, lane = t & 31;
    const bool phase = i1 - i0 >= 8;
    const int64_t seg = phase ? v : ((v + 8 * 32 - 1) / (8 * 32)) * 32;
    const int64_t ls = phase ? 0 : min((int64_t)w * seg, v);
    const int64_t L = min(seg, v - ls);
    const int64_t ib = phase ? i0 + w : i0, di = phase ? 8 : 1;
    for (int64_t j = j0; j < j1; j++) {
      KahanF32 tot;
      int64_t i = ib;
      const float* a = it.A + (i * it.nk + j) * v + ls;
      const float* g = it.gy + i * v + ls;
      // folded every 16 lane passes (at most 64 products per partial sum)
      for (; i + 3 * di < i1; i += 4 * di, a += 4 * di * S, g += 4 * di * v)
        for (int64_t lb = 0; lb < L; lb += 16 * 32) {
          const int64_t le = min(lb + 16 * 32, L);
          float acc = 0.0f;
          for (int64_t l = lb + lane; l < le; l += 32) {
            const float x0 = __ldcs(a + l), x1 = __ldcs(a + di * S + l);
            const float x2 = __ldcs(a + 2 * di * S + l), x3 = __ldcs(a + 3 * di * S + l);
            const float y0 = __ldg(g + l), y1 = __ldg(g + di * v + l);
            const float y2 = __ldg(g + 2 * di * v + l), y3 = __ldg(g + 3 * di * v + l);
            acc = __fmaf_rn(x0, y0, acc);
            acc = __fmaf_rn(x1, y1, acc);
            acc = __fmaf_rn(x2, y2, acc);
            acc = __fmaf_rn(x3, y3, acc);
          }
          tot.add(acc);
        }
      for (; i < i1; i += di, a += di * S, g += di * v)
        for (int64_t lb = 0; lb < L; lb += 64 * 32) {
          const int64_t le = min(lb + 64 * 32, L);
          float acc = 0.0f;
          for (int64_t l = lb + lane; l < le; l += 32) acc = __fmaf_rn(__ldcs(a + l), __ldg(g + l), acc);
          tot.add(acc);
        }
      float sw = tot.value();
      for (int off = 16; off > 0; off >>= 1) sw = __fadd_rn(sw, __shfl_xor_sync(0xffffffffu, sw, off));
      if (lane == 0) red[w * kGxJ + (j - j0)] = sw;
    }
    __syncthreads();
    for (int64_t j = j0 + t; j < j1; j += kBBT) {
      float sj = red[j - j0];
      for (int q = 1; q < kBBT / 32; q++) sj = __fadd_rn(sj, red[q * kGxJ + (j - j0)]);
      dst[j] = sj;
    }
    __syncthreads();
  } else {
    const int64_t C = (j1 - j0) * v;  // the item's columns in one slab
    const int CW = (int)min(C, (int64_t)kBBT);
    const int P = kBBT / CW;  // slab phases
    const int ph = t / CW, cc = t - (t / CW) * CW;
    for (int64_t cb = 0; cb < C; cb += CW) {
      const int64_t c = j0 * v + cb + cc;  // column within the slab
      float acc = 0.0f;
      KahanF32 tot;
      if (ph < P && cb + cc < C) {
        const int64_t l = c - (c / v) * v;
        const int64_t di = P;
        const float* a = it.A + (i0 + ph) * S + c;
        const float* g = it.gy + (i0 + ph) * v + l;
        const float xj = gA ? __ldg(it.x + c / v) : 0.0f;
        float* o = gA + (i0 + ph) * S + c;
        int64_t i = i0 + ph;
        int blk = 0;
        for (; i + 7 * di < i1; i += 8 * di, a += 8 * di * S, g += 8 * di * v, o += 8 * di * S) {
          float av[8], gv[8];
#pragma unroll
          for (int q = 0; q < 8; q++) {
            av[q] = __ldcs(a + q * di * S);
            gv[q] = __ldg(g + q * di * v);
          }
#pragma unroll
          for (int q = 0; q < 8; q++) {
            acc = __fmaf_rn(av[q], gv[q], acc);
            if (gA) __stcs(o + q * di * S, gv[q] * xj);
          }
          if (++blk == 8) {
            tot.add(acc);
            acc = 0.0f;
            blk = 0;
          }
        }
        for (; i < i1; i += di, a += di * S, g += di * v, o += di * S) {
          const float gv = __ldg(g);
          acc = __fmaf_rn(__ldcs(a), gv, acc);
          if (gA) __stcs(o, gv * xj);
        }
        tot.add(acc);
      }
      red[t] = (ph < P && cb + cc < C) ? tot.value() : 0.0f;
      __syncthreads();
      if (t < CW && P > 1) {  // the phases of column cc, in phase order
        float sc = red[t];
        for (int q = 1; q < P; q++) sc = __fadd_rn(sc, red[q * CW + t]);
        red[t] = sc;
      }
      __syncthreads();
      // per j of the chunk: its columns in l order, added in chunk order
      const int64_t c0 = j0 * v + cb, c1 = min(c0 + CW, j1 * v);
      for (int64_t j = c0 / v + t; j * v < c1; j += kBBT) {
        const int64_t a0 = max(j * v, c0), a1 = min((j + 1) * v, c1);
        float sj = 0.0f;
        for (int64_t q = a0; q < a1; q++) sj = __fadd_rn(sj, red[q - c0]);
        dst[j] = (a0 == j * v) ? sj : __fadd_rn(dst[j], sj);  // the chunk holding l = 0 starts j
      }
      __syncthreads();
    }
  }
  finish_gx(it, items, cnt, partials, flag);
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

template <int VEC>
__device__ __forceinline__ void ld_vec(const float* p, float (&v)[VEC]) {
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

template <int VEC>
__device__ __forceinline__ void st_vec(float* p, const float (&v)[VEC], float m) {
  if constexpr (VEC == 4)
    __stcs(reinterpret_cast<float4*>(p), make_float4(v[0] * m, v[1] * m, v[2] * m, v[3] * m));
  else if constexpr (VEC == 2)
    __stcs(reinterpret_cast<float2*>(p), make_float2(v[0] * m, v[1] * m));
  else
    __stcs(p, v[0] * m);
}

// y, gx and gA (those that are wanted) of the columns o = (i, l) in [c0, c1)
// over all rows j, v >= 32: a thread owns four columns (VEC adjacent ones,
// 4 / VEC pieces 32 VEC apart), holds their gy and y sums in registers and
// walks the rows RB at a time: one load of A serves the column sum y += A x_j
// and the row sum of A gy, which a warp reduces over its lanes per RB rows
// into its own row of red; gA = gy x_j is written on the way.  Bound: one read
// of A and one write of gA (three passes over memory with an item kind per
// result).  512 tensors (2.1e9 elements) with all three results, with
// blk_rows_fused and the smaller items: 7.89 -> 4.52 ms; 40 tensors 3.5 ->
// 0.43 ms (plain row sums 4.46 and 0.43).
template <int VEC, bool ONE>
__device__ void blk_cols_fused(const BItem& it, int64_t c0, int64_t c1, int ks, int items, int* cnt, float* partials,
                               float* red, float* xsm, int* flag) {
  constexpr int RB = VEC == 1 ? 16 : 8, NQ = 4 / VEC;
  const int t = threadIdx.x, wid = t >> 5, lane = t & 31;
  const int nk = (int)it.nk;
  const int64_t v = it.v;
  const bool wy = it.y != nullptr, wgx = it.gx != nullptr, wgA = it.gA != nullptr;
  const bool small = it.u * v <= 0xFFFFFFFFll;  // 32-bit division of the columns
  float* const rw = red + wid * kFusedRows;  // the warp's row sums (pairs, see kErr)
  const bool pairs = nk <= kErr;
  if (wy || wgA)
    for (int j = t; j < nk; j += kBBT) xsm[j] = __ldg(it.x + j);
  if (wgx)
    for (int j = lane; j < nk; j += 32) {
      rw[j] = 0.0f;
      if (pairs) rw[kErr + j] = 0.0f;
    }
  __syncthreads();
  const int nbat = (nk + RB - 1) / RB, per = (nk + nbat - 1) / nbat;
  for (int64_t g = c0 + wid * 128; g < c1; g += (kBBT / 32) * 128) {
    int64_t off[NQ];
    float gc[NQ][VEC], y0[NQ][VEC], y1[NQ][VEC];
    const int64_t col0 = g + lane * VEC;
#pragma unroll
    for (int q = 0; q < NQ; q++) {
      const int64_t col = col0 + q * 32 * VEC;
      const bool ok = col < c1;
      const int64_t i = small ? (int64_t)((uint32_t)col / (uint32_t)v) : col / v;
      off[q] = (i * nk) * v + (col - i * v);
#pragma unroll
      for (int e = 0; e < VEC; e++) {
        gc[q][e] = (ok && (wgx || wgA)) ? __ldg(it.gy + col + e) : 0.0f;
        y0[q][e] = y1[q][e] = 0.0f;
      }
    }
    for (int jb = 0; jb < nk; jb += per) {
      const int nb = min(per, nk - jb);
      float acc[RB];
#pragma unroll
      for (int e = 0; e < RB; e++) acc[e] = 0.0f;
#pragma unroll
      for (int q = 0; q < NQ; q++) {
        const bool ok = col0 + q * 32 * VEC < c1;
        if (wy || wgx) {
          float a[RB][VEC];
          const float* p = it.A + off[q];
#pragma unroll
          for (int e = 0; e < RB; e++, p += v) {
#pragma unroll
            for (int c = 0; c < VEC; c++) a[e][c] = 0.0f;
            if (e < nb && ok) ld_vec<VEC>(p, a[e]);
          }
          if (wy) {
#pragma unroll
            for (int e = 0; e < RB; e += 2) {
              const float xa = e < nb ? xsm[jb + e] : 0.0f, xb = e + 1 < nb ? xsm[jb + e + 1] : 0.0f;
#pragma unroll
              for (int c = 0; c < VEC; c++) {
                if (e < nb) y0[q][c] = __fmaf_rn(a[e][c], xa, y0[q][c]);
                float& odd = ONE ? y0[q][c] : y1[q][c];
                if (e + 1 < nb) odd = __fmaf_rn(a[e + 1][c], xb, odd);
              }
            }
          }
#pragma unroll
          for (int e = 0; e < RB; e++)
#pragma unroll
            for (int c = 0; c < VEC; c++) acc[e] = __fmaf_rn(a[e][c], gc[q][c], acc[e]);
        }
        if (wgA && ok) {
          float* p = it.gA + off[q];
#pragma unroll
          for (int e = 0; e < RB; e++, p += v)
            if (e < nb) st_vec<VEC>(p, gc[q], xsm[jb + e]);
        }
        off[q] += per * v;
      }
      if (wgx) {
        const float sum = warp_add_many<RB>(acc);
        const int row = lane / (32 / RB);
        if (lane % (32 / RB) == 0 && row < nb) {
          if (pairs)
            add_pair(rw + jb + row, sum);
          else
            rw[jb + row] = sum;
        }
        __syncwarp();
      }
    }
    if (wy) {
#pragma unroll
      for (int q = 0; q < NQ; q++)
        if (col0 + q * 32 * VEC < c1) {
#pragma unroll
          for (int e = 0; e < VEC; e++) it.y[col0 + q * 32 * VEC + e] = y0[q][e] + y1[q][e];
        }
    }
  }
  __syncthreads();
  if (wgx) {
    float* dst = (it.gxk > 1) ? partials + it.gxp + (int64_t)ks * nk : it.gx;
    for (int j = t; j < nk; j += kBBT) {
      KahanF32 sum;
#pragma unroll
      for (int w = 0; w < kBBT / 32; w++) add_pair(sum, red + w * kFusedRows + j, pairs);
      dst[j] = sum.value();
    }
    finish_gx(it, items, cnt, partials, flag);
  }
  __syncthreads();
}

// The same for rows [i0, i1) of v == 1, 32 <= n_k <= 256: lanes own
// the columns j of up to eight chunks (x_j and the column sums gx in
// registers), a warp walks eight rows at a time and reduces their sums y.
__device__ void blk_rows_fused(const BItem& it, int64_t i0, int64_t i1, int ks, int items, int* cnt, float* partials,
                               float* red, int* flag) {
  constexpr int RB = 8, NC = kFusedRowMax / 32;
  const int t = threadIdx.x, wid = t >> 5, lane = t & 31;
  const int nk = (int)it.nk;
  const bool wy = it.y != nullptr, wgx = it.gx != nullptr, wgA = it.gA != nullptr;
  float xq[NC], cs[NC];
#pragma unroll
  for (int q = 0; q < NC; q++) {
    xq[q] = ((wy || wgA) && q * 32 + lane < nk) ? __ldg(it.x + q * 32 + lane) : 0.0f;
    cs[q] = 0.0f;
  }
  float* const cw = red + wid * kFusedRows + lane;  // the lane's column sums (pairs), folded every 64 rows
#pragma unroll
  for (int q = 0; q < NC; q++) cw[q * 32] = cw[q * 32 + kErr] = 0.0f;
  auto fold = [&]() {
#pragma unroll
    for (int q = 0; q < NC; q++) {
      add_pair(cw + q * 32, cs[q]);
      cs[q] = 0.0f;
    }
  };
  int blk = 0;
  for (int64_t i = i0 + wid * RB; i < i1; i += (kBBT / 32) * RB) {
    const int nb = (int)min((int64_t)RB, i1 - i);
    float pe[RB], acc[RB];
#pragma unroll
    for (int e = 0; e < RB; e++) {
      pe[e] = ((wgx || wgA) && e < nb) ? __ldg(it.gy + i + e) : 0.0f;
      acc[e] = 0.0f;
    }
#pragma unroll
    for (int q = 0; q < NC; q += 2) {
      if (q * 32 < nk) {
        float a[2][RB];
        const float* p = it.A + i * nk + q * 32 + lane;
        const bool ok0 = q * 32 + lane < nk, ok1 = q * 32 + 32 + lane < nk;
        if (wy || wgx) {
#pragma unroll
          for (int e = 0; e < RB; e++) {
            a[0][e] = (e < nb && ok0) ? __ldcs(p + e * nk) : 0.0f;
            a[1][e] = (e < nb && ok1) ? __ldcs(p + e * nk + 32) : 0.0f;
          }
#pragma unroll
          for (int h = 0; h < 2; h++)
#pragma unroll
            for (int e = 0; e < RB; e++) {
              acc[e] = __fmaf_rn(a[h][e], xq[q + h], acc[e]);
              cs[q + h] = __fmaf_rn(a[h][e], pe[e], cs[q + h]);
            }
        }
        if (wgA) {
          float* o = it.gA + i * nk + q * 32 + lane;
#pragma unroll
          for (int e = 0; e < RB; e++) {
            if (e < nb && ok0) __stcs(o + e * nk, pe[e] * xq[q]);
            if (e < nb && ok1) __stcs(o + e * nk + 32, pe[e] * xq[q + 1]);
          }
        }
      }
    }
    if (wy) {
      const float sum = warp_add_many<RB>(acc);
      const int row = lane / (32 / RB);
      if (lane % (32 / RB) == 0 && row < nb) it.y[i + row] = sum;
    }
    if (wgx && ++blk == 64 / RB) {
      fold();
      blk = 0;
    }
  }
  if (wgx) {
    fold();
    __syncthreads();
    float* dst = (it.gxk > 1) ? partials + it.gxp + (int64_t)ks * nk : it.gx;
    for (int j = t; j < nk; j += kBBT) {
      KahanF32 sum;
#pragma unroll
      for (int w = 0; w < kBBT / 32; w++) add_pair(sum, red + w * kFusedRows + j, true);
      dst[j] = sum.value();
    }
    finish_gx(it, items, cnt, partials, flag);
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kBBT, kBBlocksPerSM) tvc_batched_kernel(const BItem* __restrict__ items,
                                                           const WItem* __restrict__ work, int nwork, int* counter,
                                                           int* gx_counters, float* gx_partials) {
  __shared__ int slot;
  __shared__ float red[(kBBT / 32) * kFusedRows];
  __shared__ __align__(16) float xsm[kFusedRows];
  __shared__ int last_flag;
  for (int w = grab(counter, &slot); w < nwork; w = grab(counter, &slot)) {
    const WItem wi = work[w];
    const BItem it = items[wi.b];
    if (wi.kind == 0)
      blk_tvc(it.A, it.u, it.nk, it.v, it.x, it.y, it.gf, wi.a0, wi.a1);
    else if (wi.kind == 3) {
      const uintptr_t al = reinterpret_cast<uintptr_t>(it.A) | reinterpret_cast<uintptr_t>(it.gA);
      const int vec = it.v % 4 == 0 && al % 16 == 0 ? 4 : it.v % 2 == 0 && al % 8 == 0 ? 2 : 1;
      int* const cnt = gx_counters + wi.b;
      if (it.nk < 8) {
        if (vec == 4)
          blk_cols_fused<4, true>(it, wi.a0, wi.a1, wi.e0, wi.e1, cnt, gx_partials, red, xsm, &last_flag);
        else if (vec == 2)
          blk_cols_fused<2, true>(it, wi.a0, wi.a1, wi.e0, wi.e1, cnt, gx_partials, red, xsm, &last_flag);
        else
          blk_cols_fused<1, true>(it, wi.a0, wi.a1, wi.e0, wi.e1, cnt, gx_partials, red, xsm, &last_flag);
      } else if (vec == 4)
        blk_cols_fused<4, false>(it, wi.a0, wi.a1, wi.e0, wi.e1, cnt, gx_partials, red, xsm, &last_flag);
      else if (vec == 2)
        blk_cols_fused<2, false>(it, wi.a0, wi.a1, wi.e0, wi.e1, cnt, gx_partials, red, xsm, &last_flag);
      else
        blk_cols_fused<1, false>(it, wi.a0, wi.a1, wi.e0, wi.e1, cnt, gx_partials, red, xsm, &last_flag);
    } else if (wi.kind == 4)
      blk_rows_fused(it, wi.a0, wi.a1, wi.e0, wi.e1, gx_counters + wi.b, gx_partials, red, &last_flag);
    else if (wi.kind == 1 || wi.kind == 5)
      blk_gx_rect(it, wi.kind == 5 ? it.gA : nullptr, wi.a0, wi.a1, wi.c0, wi.c1, wi.e0, wi.e1, gx_counters + wi.b, gx_partials, red, &last_flag);
    else
      blk_gA(it.gy, it.x, it.gA, it.nk, it.v, wi.a0, wi.a1, wi.c0, wi.c1);
  }
}

// ------------------------------------------------------------------ host --

int64_t clog2(int64_t x) {
  int64_t r = 0;
  while ((int64_t(1) << r) < x) r++;
  return r;
}

// Autotuner cache of the forward contraction: (log2 v, log2 n_k) -> G.
std::mutex g_tune_mu;
std::map<std::pair<int, int>, int> g_tune;
std::map<void*, int> g_nwork;  // work items uploaded per workspace

int rule_G(int64_t nk) { return nk <= 64 ? 8 : nk <= 128 ? 16 : 32; }  // lanes per forward row (v == 1)

int pick_G(int64_t nk, int64_t v) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  auto it = g_tune.find({(int)clog2(v), (int)clog2(nk)});
  return it != g_tune.end() ? it->second : rule_G(nk);
}

struct BLayout {
  size_t off_counter = 0, off_items = 0, off_scratch = 0, off_gxcnt = 0, off_gxpart = 0, total = 0;
  int blocks = 0;
};

int64_t cdiv64(int64_t a, int64_t b) { return (a + b - 1) / b; }

// Elements of A per work item: about eight items per resident block, so
// that the last items of a small batch still fill the GPU (24..512 tensors
// of 8..192 per mode with a fixed 2^20: 2.1-7.9 ms, most of it the last
// items alone), within 2^15 .. 2^19 (an item still streams long runs).
int64_t item_elems(const std::vector<BItem>& items) {
  double total = 0.0;
  for (const BItem& it : items) total += (double)it.u * it.nk * it.v;
  const double per = total / ((double)device_sms() * kBBlocksPerSM * 8);
  int64_t ie = 1 << 15;
  while (ie < (1 << 19) && ie < per) ie *= 2;
  return ie;
}

// The fused item kind of a tensor (3: columns, 4: rows; 0: none): where one
// read of A serves gx and another result, or gx alone in the column case.
// Without gx nothing is shared (y reads A, gA does not), and separate items are
// faster: y and gA of 512 matrices of 20..200 per mode 111 us fused, 32 apart; of
// 4096 of 100..500 1321 / 654.  Neither do tiny tensors gain: all three results
// of 4096 of 4..12 per mode 81 / 49 us, of 8..16 84 / 68, of 16..24 139 / 146; gx of
// 8..16 39 / 43.
int fused_kind(const BItem& it) {
  if (!it.gx || it.u * it.nk * it.v < (it.y && it.gA ? 4000 : 1000)) return 0;
  if (it.v >= kGxWarpRows && it.nk <= kFusedRows) return 3;
  if (it.v == 1 && it.nk >= kFusedRowMin && it.nk <= kFusedRowMax && (it.y || it.gA)) return 4;
  return 0;
}

// Columns (kind 3) or rows (kind 4) per fused item.
int64_t fused_per(const BItem& it, int64_t ie) {
  if (it.v == 1) return std::min<int64_t>(1024, std::max<int64_t>(256, ie / it.nk / 256 * 256));
  return std::max<int64_t>(1024, ie / it.nk / 1024 * 1024);
}

int64_t assign_gx(std::vector<BItem>* items, int64_t ie);

// Rectangle of a gx item: jr rows j by sr slabs, about ie elements.
// Warp-mapped rows (v >= 32) take every slab of a j before cutting the slabs
// and keep 8 slabs (one per warp) where the tensor has them; column-mapped
// rows take whole slab widths.
void gx_rect(const BItem& it, int64_t ie, int64_t* jr, int64_t* sr) {
  const int64_t v = std::max<int64_t>(1, it.v);
  if (v >= kGxWarpRows)  // whole slab ranges per j first; at most kGxJ rows, 8 slabs when there are
    *jr = std::max<int64_t>(1, std::min<int64_t>(std::min(it.nk, kGxJ), ie / std::max<int64_t>(1, it.u * v)));
  else  // whole slab widths first (coalesced columns)
    *jr = std::max<int64_t>(1, std::min<int64_t>(it.nk, ie / v));
  *sr = std::max<int64_t>(1, std::min<int64_t>(it.u, ie / (*jr * v)));
  if (v >= kGxWarpRows) *sr = std::max(*sr, std::min<int64_t>(it.u, 8));
}

void make_work(std::vector<BItem>& items, int64_t ie, std::vector<WItem>* work) {
  assign_gx(&items, ie);
  work->clear();
  for (int b = 0; b < (int)items.size(); b++) {
    const BItem& it = items[b];
    const int64_t uv = it.u * it.v;
    if (const int kind = fused_kind(it)) {
      const int64_t per = fused_per(it, ie);
      int ks = 0;
      for (int64_t o = 0; o < uv; o += per, ks++)
        work->push_back({b, kind, o, std::min(uv, o + per), 0, 0, ks, (int)cdiv64(uv, per)});
      continue;
    }
    const bool with_gA = it.gx && it.gA && it.v < kGxWarpRows;  // one pass for both
    if (it.y) {
      const int64_t per = std::max<int64_t>(256, cdiv64(ie, it.nk) / 256 * 256);
      for (int64_t o = 0; o < uv; o += per) work->push_back({b, 0, o, std::min(uv, o + per), 0, 0, 0, 0});
    }
    if (it.gx) {  // rectangles (see assign_gx), partials summed by the tensor's last item
      int64_t jr, sr;
      gx_rect(it, ie, &jr, &sr);
      const int nitems = (int)(cdiv64(it.u, sr) * cdiv64(it.nk, jr));
      int ks = 0;
      for (int64_t i = 0; i < it.u; i += sr, ks++)
        for (int64_t j = 0; j < it.nk; j += jr)
          work->push_back({b, with_gA ? 5 : 1, i, std::min(it.u, i + sr), j, std::min(it.nk, j + jr), ks, nitems});
    }
    if (it.gA && !with_gA) {
      const int64_t S = it.nk * it.v;
      if (it.v >= 32) {
        // rectangles of slabs x rows
        const int64_t rows = std::max<int64_t>(1, std::min<int64_t>(it.nk, ie / it.v));
        const int64_t slabs = std::max<int64_t>(1, ie / (rows * it.v));
        for (int64_t i = 0; i < it.u; i += slabs)
          for (int64_t j = 0; j < it.nk; j += rows)
            work->push_back({b, 2, i, std::min(it.u, i + slabs), j, std::min(it.nk, j + rows), 0, 0});
      } else {
        const int64_t slabs = std::max<int64_t>(1, ie / S);
        for (int64_t i = 0; i < it.u; i += slabs)
          work->push_back({b, 2, i, std::min(it.u, i + slabs), 0, it.nk, 0, 0});
      }
    }
  }
}

// Workspace of a tensor batch: header, descriptors, work items (the exact
// count, from the same construction the call uses).
tvc_status check_tvc_descs(const tvc_batch_desc* d, int count, std::vector<BItem>* items);

// gx items per tensor (slab, column or row ranges of about ie elements) and
// the offsets of their partials; called on every item list by make_work.
int64_t assign_gx(std::vector<BItem>* items, int64_t ie) {
  int64_t off = 0;
  for (BItem& it : *items) {
    it.gxk = 0;
    it.gxp = 0;
    if (!it.gx) continue;
    if (fused_kind(it)) {
      it.gxk = (int)cdiv64(it.u * it.v, fused_per(it, ie));
    } else {
      int64_t jr, sr;
      gx_rect(it, ie, &jr, &sr);
      it.gxk = (int)cdiv64(it.u, sr);
    }
    if (it.gxk > 1) {
      it.gxp = off;
      off += (int64_t)it.gxk * it.nk;
    }
  }
  return off;
}

BLayout layout_tvc_items(const std::vector<BItem>& items, size_t nwork) {
  BLayout L;
  L.off_counter = 0;
  L.off_items = 256;
  L.off_scratch = L.off_items + align_up(items.size() * sizeof(BItem), 256);
  L.off_gxcnt = L.off_scratch + align_up(nwork * sizeof(WItem), 256);
  int64_t nparts = 0;
  for (const BItem& it : items)
    if (it.gxk > 1) nparts = std::max<int64_t>(nparts, it.gxp + (int64_t)it.gxk * it.nk);
  L.off_gxpart = L.off_gxcnt + align_up(items.size() * sizeof(int), 256);
  L.total = L.off_gxpart + align_up((size_t)std::max<int64_t>(1, nparts) * sizeof(float), 256);
  L.blocks = device_sms() * kBBlocksPerSM;
  return L;
}

tvc_status check_tvc_descs(const tvc_batch_desc* d, int count, std::vector<BItem>* items) {
  std::vector<std::pair<int64_t, int>> order;
  for (int b = 0; b < count; b++) {
    Shape s;
    if (make_shape(d[b].order, d[b].dims, d[b].mode, &s) != TVC_OK) return TVC_ERR_INVALID_ARG;
    if (!d[b].A) return TVC_ERR_INVALID_ARG;
    if (d[b].y && !d[b].x) return TVC_ERR_INVALID_ARG;
    if ((d[b].gx || d[b].gA) && !d[b].gy) return TVC_ERR_INVALID_ARG;
    if (d[b].gA && !d[b].x) return TVC_ERR_INVALID_ARG;
    order.push_back({s.N, b});
  }
  std::stable_sort(order.begin(), order.end(), [](auto& a, auto& b) { return a.first > b.first; });
  if (items) {
    items->clear();
    for (auto& pr : order) {
      const tvc_batch_desc& e = d[pr.second];
      Shape s;
      make_shape(e.order, e.dims, e.mode, &s);
      BItem it{};
      it.A = e.A;
      it.x = e.x;
      it.y = e.y;
      it.gy = e.gy;
      it.gx = e.gx;
      it.gA = e.gA;
      it.u = s.u;
      it.nk = s.nk;
      it.v = s.v;
      it.gf = pick_G(s.nk, s.v);
      it.gxk = 0;
      it.gxp = 0;
      items->push_back(it);
    }
  }
  return TVC_OK;
}

}  // namespace
}  // namespace tvcg

using namespace tvcg;

extern "C" size_t tvc_batched_workspace_size(const tvc_batch_desc* descs, int count) {
  if (count < 0 || (count > 0 && !descs)) return 0;
  std::vector<BItem> items;
  if (check_tvc_descs(descs, count, &items) != TVC_OK) return 0;
  std::vector<WItem> work;
  make_work(items, item_elems(items), &work);
  return layout_tvc_items(items, work.size()).total;
}

extern "C" tvc_status tvc_batched(const tvc_batch_desc* descs, int count, int flags, void* workspace, size_t ws_bytes,
                                  tvc_stream_t stream) {
  if (count < 0 || !descs) return TVC_ERR_INVALID_ARG;
  if (count == 0) return TVC_OK;
  std::vector<BItem> items;
  tvc_status rc = check_tvc_descs(descs, count, &items);
  if (rc != TVC_OK) return rc;
  std::vector<WItem> work;
  make_work(items, item_elems(items), &work);
  const BLayout L = layout_tvc_items(items, work.size());
  if (!workspace || ws_bytes < L.total) return TVC_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  char* w = static_cast<char*>(workspace);
  int* hdr = reinterpret_cast<int*>(w + L.off_counter);
  if (!(flags & TVC_BATCH_PREUPLOADED)) {
    const int nwork = (int)work.size();
    if (cudaMemcpyAsync(w + L.off_items, items.data(), items.size() * sizeof(BItem), cudaMemcpyHostToDevice, st) !=
            cudaSuccess ||
        cudaMemcpyAsync(w + L.off_scratch, work.data(), work.size() * sizeof(WItem), cudaMemcpyHostToDevice, st) !=
            cudaSuccess ||
        cudaMemcpyAsync(hdr + 1, &nwork, sizeof(int), cudaMemcpyHostToDevice, st) != cudaSuccess ||
        // per-tensor gx counters: zero now; the last item of a tensor resets its own
        cudaMemsetAsync(w + L.off_gxcnt, 0, items.size() * sizeof(int), st) != cudaSuccess)
      return TVC_ERR_CUDA;
    // The host vectors die here: wait for the copies (pageable sources).
    if (cudaStreamSynchronize(st) != cudaSuccess) return TVC_ERR_CUDA;
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_nwork[workspace] = nwork;
  }
  int nwork = 0;
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    auto itn = g_nwork.find(workspace);
    if (itn == g_nwork.end()) return TVC_ERR_INVALID_ARG;  // PREUPLOADED without a prior upload
    nwork = itn->second;
  }
  cudaMemsetAsync(hdr, 0, sizeof(int), st);
  tvc_batched_kernel<<<L.blocks, kBBT, 0, st>>>(reinterpret_cast<const BItem*>(w + L.off_items),
                                               reinterpret_cast<const WItem*>(w + L.off_scratch), nwork, hdr,
                                               reinterpret_cast<int*>(w + L.off_gxcnt),
                                               reinterpret_cast<float*>(w + L.off_gxpart));
  count_launches(1);
  return cuda_status(cudaGetLastError());
}

extern "C" tvc_status tvc_batched_autotune(const tvc_batch_desc* descs, int count, void* workspace, size_t ws_bytes,
                                           tvc_stream_t stream) {
  // Times the candidate lane counts of the forward contraction on the
  // tensors of every shape class and records the fastest; synchronises.
  if (count <= 0 || !descs) return TVC_ERR_INVALID_ARG;
  std::vector<BItem> items;
  tvc_status rc = check_tvc_descs(descs, count, &items);
  if (rc != TVC_OK) return rc;
  std::vector<WItem> allwork;
  const int64_t ie = item_elems(items);
  make_work(items, ie, &allwork);
  const BLayout L = layout_tvc_items(items, allwork.size());
  if (!workspace || ws_bytes < L.total) return TVC_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  char* w = static_cast<char*>(workspace);
  // every shape class of forward rows (v == 1, where lanes split a row)
  // with the tensors that belong to it
  std::map<std::pair<int, int>, std::vector<BItem>> classes;
  for (const BItem& it : items) {
    if (!it.y || it.v != 1) continue;
    BItem one = it;
    one.gx = nullptr;
    one.gA = nullptr;
    classes[{(int)clog2(it.v), (int)clog2(it.nk)}].push_back(one);
  }
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  const int cands[5] = {1, 4, 8, 16, 32};
  for (auto& kv : classes) {
    std::vector<BItem> sub = kv.second;  // at most 256 tensors of the class
    if (sub.size() > 256) sub.resize(256);
    float best = 1e30f;
    int bestG = rule_G(sub[0].nk);
    for (int G : cands) {
      for (BItem& it : sub) it.gf = G;
      std::vector<WItem> wk;
      make_work(sub, ie, &wk);
      if (wk.size() > allwork.size()) break;  // the workspace holds allwork
      cudaMemcpy(w + L.off_items, sub.data(), sub.size() * sizeof(BItem), cudaMemcpyHostToDevice);
      cudaMemcpy(w + L.off_scratch, wk.data(), wk.size() * sizeof(WItem), cudaMemcpyHostToDevice);
      float tot = 0.0f;
      for (int rep = 0; rep < 3; rep++) {
        cudaMemsetAsync(w + L.off_counter, 0, sizeof(int), st);
        cudaEventRecord(e0, st);
        tvc_batched_kernel<<<L.blocks, kBBT, 0, st>>>(reinterpret_cast<const BItem*>(w + L.off_items),
                                                     reinterpret_cast<const WItem*>(w + L.off_scratch),
                                                     (int)wk.size(), reinterpret_cast<int*>(w + L.off_counter),
                                                     reinterpret_cast<int*>(w + L.off_gxcnt),
                                                     reinterpret_cast<float*>(w + L.off_gxpart));
        cudaEventRecord(e1, st);
        cudaEventSynchronize(e1);
        float ms = 0.0f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (rep > 0) tot += ms;
      }
      count_launches(3);
      if (tot < best) {
        best = tot;
        bestG = G;
      }
    }
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tune[kv.first] = bestG;
  }
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_nwork.erase(workspace);  // the workspace no longer holds an uploaded batch
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  return cuda_status(cudaGetLastError());
}
