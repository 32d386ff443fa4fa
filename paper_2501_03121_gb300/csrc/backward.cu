// Adjoints of the contraction Y = A x_k x (the paper has no passage for them;
// they follow from the definition of Section 3 by differentiation):
//     gx[j]      = sum_{i,l} A[i][j][l] * gy[i][l]      (a contraction of A with
//                                                        the (d-1)-tensor gy)
//     gA[i][j][l] = gy[i][l] * x[j]  (+ beta * gA)     (a rank-1 write stream)
// in the u x n_k x v view of mode k.
//
// gx, v == 1 and k > 0: gx = (A viewed as u x n_k) x_0 gy, i.e. a TVC of
//   mode 0 on the unfolded view (the column kernel), with gy times the slab
//   scale for narrow storage.
// gx, FP32 arithmetic, mode 0 with rows of at most 512 bytes: gx = (A viewed as n_k x v) x_1 gy, a
//   TVC of the last mode (the row kernels).
// gx, otherwise: each thread owns 16-byte pieces of columns (i, l), keeps
//   their gy in registers (FP64 arithmetic: in shared memory) and streams the piece's rows, eight (rows off 16-byte
//   boundaries: four) in flight; a warp reduces the rows' dot products over
//   its lanes with halving exchanges into its own sums of a chunk of rows in
//   shared memory.  Blocks walk the pieces persistently and leave one partial
//   row each; a second kernel adds the blocks' partials in a fixed order.  A
//   is read once; gy once per chunk of rows.
// gA: threads own 16 bytes (or one element where rows or slabs are not whole
//   pieces) of columns (i, l), looping over j, when v >= 32, of positions (j,
//   l) of a slab, looping over slabs i, below.
#include <algorithm>

#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "ragged.cuh"

namespace tvcg {

constexpr int kBT = 256;  // threads per block
constexpr int kBW = kBT / kWarp;
constexpr int kGxRows = 256;  // rows per chunk at most

template <tvc_dtype DT>
struct GradArgs {
  const typename Elem<DT>::T* A;
  const void* gy;   // vector type (FP64 / FP32)
  const float* scales;
  void* partial;    // [nblk][nk], vector type
  int64_t u, nk, v, upi0, pps, nblk;
  int mode0;
  int rch;          // rows per chunk (<= kGxRows, kGx64Rows)
};

// ------------------------------------------------------------- gx, v >= 2

// A 16-byte piece as the compute type.
template <tvc_dtype DT>
__device__ __forceinline__ void gx_piece(const uint4& w, typename Elem<DT>::C (&r)[16 / Elem<DT>::kSize]) {
  if constexpr (DT == TVC_F64) {
    r[0] = __hiloint2double((int)w.y, (int)w.x);
    r[1] = __hiloint2double((int)w.w, (int)w.z);
  } else if constexpr (DT == TVC_F32D) {
    Elem<TVC_F32>::decode16(w, r);
  } else {
    Elem<DT>::decode16(w, r);
  }
}

// The sums over the warp's lanes of a[0..M-1], the kept values halved per
// exchange: lane L returns the sum of a[L / (32 / M)].
template <int M>
__device__ __forceinline__ float gx_lanes(float (&a)[M]) {
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

// The same for float-float pairs (s, c), joined into (s, c, e): with the error
// of c kept too, since c alone loses 2^-48 of the sum at every exchange.
template <int M>
__device__ __forceinline__ void gx_lanes(float (&s)[M], float (&c)[M], float& e0) {
  const int lane = threadIdx.x & 31;
  float e[M];
#pragma unroll
  for (int q = 0; q < M; q++) e[q] = 0.0f;
  auto join = [](float& s0, float& c0, float& r0, float s1, float c1, float r1) {
    float t, es, ec, et;
    two_sum(s0, s1, t, es);
    s0 = t;
    two_sum(c0, c1, t, ec);
    two_sum(t, es, c0, et);
    r0 = __fadd_rn(__fadd_rn(r0, r1), __fadd_rn(ec, et));
  };
#pragma unroll
  for (int h = M / 2, bit = 16; h >= 1; h >>= 1, bit >>= 1) {
    const bool up = lane & bit;
#pragma unroll
    for (int q = 0; q < h; q++) {
      const float os = up ? s[q] : s[q + h], oc = up ? c[q] : c[q + h], oe = up ? e[q] : e[q + h];
      s[q] = up ? s[q + h] : s[q];
      c[q] = up ? c[q + h] : c[q];
      e[q] = up ? e[q + h] : e[q];
      join(s[q], c[q], e[q], __shfl_xor_sync(0xFFFFFFFFu, os, bit), __shfl_xor_sync(0xFFFFFFFFu, oc, bit),
           bit == 16 ? 0.0f : __shfl_xor_sync(0xFFFFFFFFu, oe, bit));
    }
  }
#pragma unroll
  for (int bit = 16 / M; bit >= 1; bit >>= 1)
    join(s[0], c[0], e[0], __shfl_xor_sync(0xFFFFFFFFu, s[0], bit), __shfl_xor_sync(0xFFFFFFFFu, c[0], bit),
         __shfl_xor_sync(0xFFFFFFFFu, e[0], bit));
  e0 = e[0];
}

// Bound: HBM.  128^4 FP32, modes 0-2: 190 us and a reduction of 15 -> 163 and
// 3 (7.0 TB/s; the kernel before held 16 rows' sums and loads in 168
// registers, one block per SM); 12x93x44x11x82 FP32 mode 3 136 -> 62 us.  Resident blocks per SM (the grid is
// one wave of them):
template <tvc_dtype DT>
inline constexpr int kGxBlocks = DT == TVC_E4M3 ? 2 : 3;

// AL: every row of A starts on a 16-byte boundary.
template <tvc_dtype DT, bool AL>
__global__ void __launch_bounds__(kBT, kGxBlocks<DT>) tvc_gradx_kernel(const GradArgs<DT> a) {
  using E = Elem<DT>;
  constexpr int ES = E::kSize, VEC = 16 / ES, RB = AL ? 8 : 4;
  __shared__ float2 sums[kBW][kGxRows];  // compensated pairs
  const int64_t b = blockIdx.x % a.nblk, j0 = blockIdx.x / a.nblk * a.rch;
  const int jn = (int)min((int64_t)a.rch, a.nk - j0);
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  float2* const mine = sums[warp];
  for (int j = lane; j < jn; j += 32) mine[j] = make_float2(0.0f, 0.0f);
  __syncwarp();
  const uint64_t sb = (uint64_t)a.v * ES;
  const int64_t pieces = a.u * a.pps;
  for (int64_t q0 = b * kBT; q0 < pieces; q0 += a.nblk * kBT) {
    const int64_t q = q0 + t;
    const bool ok = q < pieces;
    const int64_t i = ok ? piece_row(q, a.pps) : 0;
    const int64_t l = ok ? (q - i * a.pps) * VEC : 0;
    const int nv = ok ? (int)min((int64_t)VEC, a.v - l) : 0, bytes = nv * ES;
    uint64_t ad = reinterpret_cast<uint64_t>(a.A) + (uint64_t)((i * a.nk + j0) * a.v + l) * ES;
    const float* const gyp = static_cast<const float*>(a.gy) + i * a.v + l;
    float gf[VEC], sc = 1.0f;  // gy of the piece times the slab scale (zero past the row)
    if constexpr (kNarrow<DT>) {
      if (!a.mode0 && a.scales) sc = __ldg(a.scales + i / a.upi0);
    }
#pragma unroll
    for (int e = 0; e < VEC; e++) gf[e] = e < nv ? __fmul_rn(__ldg(gyp + e), sc) : 0.0f;
    for (int j = 0; j < jn; j += RB) {
      Chunks ch[RB];
      uint32_t sh[RB];
#pragma unroll
      for (int e = 0; e < RB; e++) {
        ch[e].a = ch[e].b = make_uint4(0u, 0u, 0u, 0u);
        if (ok && j + e < jn) {
          if constexpr (AL)
            ch[e].a = __ldcs(reinterpret_cast<const uint4*>(ad));
          else
            ld_chunks(ad, bytes, ch[e]);
        }
        sh[e] = (uint32_t)ad & 15;
        ad += sb;
      }
      float s[RB];
#pragma unroll
      for (int e = 0; e < RB; e++) {
        float r[VEC];
        gx_piece<DT>(AL ? ch[e].a : cut<ES>(ch[e], sh[e]), r);
        if (nv < VEC) {  // what follows the row is another row
#pragma unroll
          for (int x = 0; x < VEC; x++) r[x] = x < nv ? r[x] : 0.0f;
        }
        s[e] = 0.0f;
#pragma unroll
        for (int x = 0; x < VEC; x++) s[e] = __fmaf_rn(r[x], gf[x], s[e]);
      }
      const float v = gx_lanes<RB>(s);
      const int row = lane / (32 / RB);
      if (lane % (32 / RB) == 0 && j + row < jn) {
        const float2 o = mine[j + row];
        float sum, err;
        two_sum(o.x, v, sum, err);
        mine[j + row] = make_float2(sum, __fadd_rn(o.y, err));
      }
      __syncwarp();
    }
  }
  __syncthreads();
  for (int j = t; j < jn; j += kBT) {
    KahanF32 k;
    for (int w = 0; w < kBW; w++) {
      const float2 o = sums[w][j];
      k.add(o.x);
      k.add(o.y == o.y ? o.y : 0.0f);  // NaN: o.x alone (see pair_value)
    }
    float val = k.value();
    if constexpr (kNarrow<DT>) {
      if (a.mode0 && a.scales) val = __fmul_rn(val, __ldg(a.scales + j0 + j));
    }
    static_cast<float*>(a.partial)[b * a.nk + j0 + j] = val;
  }
}

// The same in FP64.
template <int M>
__device__ __forceinline__ double gx_lanes(double (&a)[M]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int h = M / 2, bit = 16; h >= 1; h >>= 1, bit >>= 1) {
    const bool up = lane & bit;
#pragma unroll
    for (int e = 0; e < h; e++) {
      const double mine = up ? a[e + h] : a[e], other = up ? a[e] : a[e + h];
      a[e] = mine + __shfl_xor_sync(0xFFFFFFFFu, other, bit);
    }
  }
  double r = a[0];
#pragma unroll
  for (int bit = 16 / M; bit >= 1; bit >>= 1) r += __shfl_xor_sync(0xFFFFFFFFu, r, bit);
  return r;
}

// FP64 arithmetic (FP64 and single-double storage): a thread adds the
// float-float products of a row over the kp pieces of its tile (256 kp pieces)
// before they are joined over the lanes, so that the exchanges and the FP64
// sums behind them are paid once per kp pieces.
// An element outside the exact window enters the pairs as zero and an FP64
// sum of the thread (its slots) by a multiply-add; exact zeros need neither.  gy
// outside its window (a mean loss over a large tensor is) is first scaled by a
// power of two per warp and tile.
// Bound: latency and the FP32 pipe.  us of gx on 17x52x68x18x31 mode 1 / 128x128x128x16
// mode 1 / 300x200x256 mode 0 / 40x21x33000 mode 1, FP64: 93 / 87 / 47 / 84
// (2.9-3.4 TB/s); 1% zeros the same; 1% of the elements nonzero and below 2^-64
// 157 / 149 / 80 / 139; all of them 204 / 191 / 101 / 174; gy below 2^-32 93 / 87
// / 47 / 84.  Single-double: 75 / 68 / 43 / 66.  A kernel that joined the lanes
// in plain pairs after every piece took 80 / 84 / 44 / 73 on plain data, 336 /
// 386 / 175 / 284 with 1% zeros or a small gy, and was up to nine times further
// off (480x161 mode 0: 1.6e-14 of the terms' root sum of squares, 3.1e-15 here).
template <tvc_dtype DT>
inline constexpr int kGxTile = DT == TVC_F64 ? 4 : 2;  // pieces per thread and tile at most (48 KB of shared memory)
constexpr int kGx64Rows = 128;                          // rows per chunk at most
constexpr int kGx64Blocks = 3;                          // resident per SM (2: up to 7% slower, 4: 15-30%)

// ah + al of an element, both zero outside the window; `out` collects the bits
// of nonzero elements there.
__device__ __forceinline__ void gx_split(double v, float& ah, float& al, uint32_t& out) {
  const uint32_t lo = (uint32_t)__double2loint(v), hi = (uint32_t)__double2hiint(v);
  const bool in = hi * 2u - kDfWindowBase < (1u << 28);
  const uint32_t hb = in ? __funnelshift_l(lo, hi - 0x38000000u, 3) | (hi & 0x80000000u) : 0u;
  ah = __uint_as_float(hb);
  al = __fmul_rn(__uint2float_rn(in ? lo & 0x1FFFFFFFu : 0u), __uint_as_float((hb & 0xFF800000u) - 0x1A000000u));
  if (!in) out |= hi * 2u | lo;
}
__device__ __forceinline__ void gx_split(float v, float& ah, float& al, uint32_t& out) {
  const bool in = df_out_of_window(v) == 0;
  ah = in ? v : 0.0f;
  al = 0.0f;
  if (!in) out |= __float_as_uint(v) << 1;
}

// split_x of an entry in the window, or zero, by integer operations (its
// conversions and subtraction in FP64 cost a tenth of the kernel): the entry
// rounded to 24 bits, and the signed rest.
__device__ __forceinline__ XSplit gx_split_gy(double g) {
  const uint64_t w = (uint64_t)__double_as_longlong(g);
  if (w << 1 == 0) return XSplit{0.0f, 0.0f};
  const uint64_t r = w + (1u << 28);
  const uint32_t lo = (uint32_t)r, hi = (uint32_t)(r >> 32);
  XSplit p;
  p.xh = __uint_as_float(__funnelshift_l(lo, hi - 0x38000000u, 3) | (hi & 0x80000000u));
  // units of 2^-52 of the unrounded exponent
  const uint32_t unit = (((uint32_t)(w >> 32) - 0x38000000u) << 3 & 0x7F800000u) - 0x1A000000u;
  const float rest = __int2float_rn((int)(lo & 0x1FFFFFFFu) - (1 << 28));
  p.xl = __fmul_rn((int64_t)w < 0 ? -rest : rest, __uint_as_float(unit));
  return p;
}

__device__ __forceinline__ double gx_dfma(double a, const double* g, double d) { return dfma_slow(a, g, d); }
__device__ __forceinline__ double gx_dfma(float a, const double* g, double d) { return dfma_slow_f(a, g, d); }

template <tvc_dtype DT, bool AL>
__global__ void __launch_bounds__(kBT, kGx64Blocks) tvc_gradx64_kernel(const GradArgs<DT> a) {
  using E = Elem<DT>;
  using T = typename E::T;
  constexpr int ES = E::kSize, VEC = 16 / ES, RB = AL ? 8 : 4, KP = kGxTile<DT>;
  extern __shared__ __align__(16) unsigned char gx_smem[];
  double* const sums = reinterpret_cast<double*>(gx_smem);            // [kBW][kGx64Rows]
  double* const slots = sums + kBW * kGx64Rows;                       // [RB][kBT]
  int64_t* const offs = reinterpret_cast<int64_t*>(slots + RB * kBT);  // [KP][kBT]: 8 * element of row 0 + elements inside the row, < 0: no piece
  float2* const gsm = reinterpret_cast<float2*>(offs + KP * kBT);     // [KP][VEC][kBT]: split gy
  const int64_t b = blockIdx.x % a.nblk, j0 = blockIdx.x / a.nblk * a.rch;
  const int jn = (int)min((int64_t)a.rch, a.nk - j0);
  const int t = threadIdx.x, lane = t & 31;
  double* const mine = sums + (t >> 5) * kGx64Rows;
  double* const slot = slots + t;
  for (int j = lane; j < jn; j += 32) mine[j] = 0.0;
#pragma unroll
  for (int e = 0; e < RB; e++) slot[e * kBT] = 0.0;
  __syncwarp();
  const T* const A = static_cast<const T*>(a.A) + j0 * a.v;
  const double* const gy = static_cast<const double*>(a.gy);
  // an even share of the pieces per block
  const int64_t pieces = a.u * a.pps, qe = pieces * (b + 1) / a.nblk;
  for (int64_t q0 = pieces * b / a.nblk; q0 < qe; q0 += KP * kBT) {
    const int kp = (int)min((int64_t)KP, (qe - q0 + kBT - 1) / kBT);
    // the thread's pieces and their gy
    uint32_t gout = 0;   // VEC bits per piece: entries that stay outside the window
    double scale = 1.0;  // of the warp's pairs
    double g[KP][VEC];
    int most = 0;        // exponent field of the largest entry below 2^1000
    bool in = true;
    auto inside = [](double v) {  // the window of an entry, or zero
      const uint32_t hi = (uint32_t)__double2hiint(v) << 1, lo = (uint32_t)__double2loint(v);
      return hi - ((1023u - 32) << 21) < (64u << 21) || (hi | lo) == 0;
    };
#pragma unroll
    for (int k = 0; k < KP; k++) {
      const int64_t q = q0 + k * kBT + t;
      const bool ok = q < qe;
      const int64_t i = ok ? piece_row(q, a.pps) : 0, l = ok ? (q - i * a.pps) * VEC : 0;
      offs[k * kBT + t] = ok ? (i * a.nk * a.v + l) * 8 + min((int64_t)VEC, a.v - l) : -1;
#pragma unroll
      for (int x = 0; x < VEC; x++) {
        g[k][x] = ok && l + x < a.v ? __ldg(gy + i * a.v + l + x) : 0.0;
        const int f = __double2hiint(g[k][x]) >> 20 & 0x7FF;
        if (f < 2023) most = max(most, f);
        in = in && inside(g[k][x]);
      }
    }
    if (!__all_sync(0xFFFFFFFFu, in)) {
      most = __reduce_max_sync(0xFFFFFFFFu, most);
      if (most > 23) {
        // the power of two that takes the largest entry to [1, 2), and back
        scale = __hiloint2double(most << 20, 0);
        const double down = __hiloint2double((2046 - most) << 20, 0);
#pragma unroll
        for (int k = 0; k < KP; k++)
#pragma unroll
          for (int x = 0; x < VEC; x++) g[k][x] *= down;
      }
    }
#pragma unroll
    for (int k = 0; k < KP; k++)
#pragma unroll
      for (int x = 0; x < VEC; x++) {
        XSplit p{0.0f, 0.0f};
        if (inside(g[k][x]))
          p = gx_split_gy(g[k][x]);
        else
          gout |= 1u << (k * VEC + x);
        gsm[(k * VEC + x) * kBT + t] = make_float2(p.xh, p.xl);
      }
    for (int j = 0; j < jn; j += RB) {
      const int rows = min(RB, jn - j);
      float s[RB], c[RB];
#pragma unroll
      for (int e = 0; e < RB; e++) s[e] = c[e] = 0.0f;
      bool extra = false;
      for (int k = 0; k < kp; k++) {
        if (offs[k * kBT + t] < 0) break;
        const int64_t off = offs[k * kBT + t] >> 3;
        const int nv = AL ? VEC : (int)(offs[k * kBT + t] & 7);
        const T* const p = A + off + j * a.v;
        const uint64_t ad = reinterpret_cast<uint64_t>(p);
        Chunks ch[RB];
#pragma unroll
        for (int e = 0; e < RB; e++) {
          if constexpr (AL)
            ch[e].a = e < rows ? __ldcs(reinterpret_cast<const uint4*>(p + e * a.v)) : make_uint4(0u, 0u, 0u, 0u);
          else {
            ch[e].a = ch[e].b = make_uint4(0u, 0u, 0u, 0u);
            if (e < rows) ld_chunks(ad + (uint64_t)(e * a.v) * ES, nv * ES, ch[e]);
          }
        }
        auto row = [&](int e, typename E::C (&r)[VEC]) {
          gx_piece<DT>(AL ? ch[e].a : cut<ES>(ch[e], (uint32_t)(ad + (uint64_t)(e * a.v) * ES) & 15), r);
        };
        XSplit xs[VEC];
#pragma unroll
        for (int x = 0; x < VEC; x++) {
          const float2 w = gsm[(k * VEC + x) * kBT + t];
          xs[x] = XSplit{w.x, w.y};
        }
        uint32_t out = 0;
#pragma unroll
        for (int e = 0; e < RB; e++) {
          typename E::C r[VEC];
          row(e, r);
#pragma unroll
          for (int x = 0; x < VEC; x++) {
            if (!AL && x >= nv) continue;  // another row's
            float ah, al;
            gx_split(r[x], ah, al, out);
            const float pr = __fmul_rn(ah, xs[x].xh);
            float er = __fmaf_rn(ah, xs[x].xh, -pr);
            er = __fmaf_rn(ah, xs[x].xl, er);
            er = __fmaf_rn(al, xs[x].xh, er);
            float sum, err;
            two_sum(s[e], pr, sum, err);
            s[e] = sum;
            c[e] = __fadd_rn(c[e], __fadd_rn(err, er));
          }
        }
        const uint32_t go = gout >> (k * VEC) & ((1u << VEC) - 1);
        if (out | go) {  // what the pairs left out
          const int64_t q = q0 + k * kBT + t, i = piece_row(q, a.pps);
          const double* const gp = gy + i * a.v + (q - i * a.pps) * VEC;
#pragma unroll
          for (int e = 0; e < RB; e++) {
            if (e >= rows) break;
            typename E::C r[VEC];
            row(e, r);
#pragma unroll
            for (int x = 0; x < VEC; x++)
              if (x < nv && ((go >> x & 1) || (df_out_of_window(r[x]) != 0 && r[x] != 0)))
                slot[e * kBT] = gx_dfma(r[x], gp + x, slot[e * kBT]);
          }
          extra = true;
        }
      }
      float e0;
      gx_lanes<RB>(s, c, e0);
      const int row = lane / (32 / RB);
      double d = ((double)s[0] + (double)c[0]) + (double)e0;
      if (scale != 1.0) d *= scale;
      if (__any_sync(0xFFFFFFFFu, extra)) {
        double w[RB];
#pragma unroll
        for (int e = 0; e < RB; e++) {
          w[e] = slot[e * kBT];
          slot[e * kBT] = 0.0;
        }
        d += gx_lanes<RB>(w);
      }
      if (lane % (32 / RB) == 0 && row < rows) mine[j + row] += d;
      __syncwarp();
    }
  }
  __syncthreads();
  for (int j = t; j < jn; j += kBT) {
    double val = sums[j];
    for (int w = 1; w < kBW; w++) val += sums[w * kGx64Rows + j];
    static_cast<double*>(a.partial)[b * a.nk + j0 + j] = val;
  }
}

// Shared memory of that kernel.
template <tvc_dtype DT, bool AL>
constexpr int gx64_smem() {
  return (kBW * kGx64Rows + (AL ? 8 : 4) * kBT) * 8 + kGxTile<DT> * kBT * (8 + 16 / Elem<DT>::kSize * 8);
}

// gx[j] = the blocks' partial sums in FP64, 32 entries per block: each warp a
// contiguous share of the blocks in order, then the warps in order.
template <class V>
__global__ void __launch_bounds__(kBT) tvc_gradx_reduce_kernel(const V* __restrict__ partial, V* __restrict__ gx,
                                                              int64_t nk, int64_t nblk) {
  __shared__ double sums[kBW][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t j = (int64_t)blockIdx.x * 32 + lane;
  double s = 0.0;
  if (j < nk) {
#pragma unroll 8
    for (int64_t b = nblk * w / kBW; b < nblk * (w + 1) / kBW; b++) s += (double)partial[b * nk + j];
  }
  sums[w][lane] = s;
  __syncthreads();
  if (w == 0 && j < nk) {
    for (int q = 1; q < kBW; q++) s += sums[q][lane];
    gx[j] = (V)s;
  }
}

// gy'[i] = gy[i] * scale[i / upi0] (narrow storage, v == 1, mode > 0).
__global__ void tvc_scale_gy_kernel(const float* __restrict__ gy, const float* __restrict__ scales, float* out,
                                    int64_t u, int64_t upi0) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < u; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = scales ? __fmul_rn(gy[i], scales[i / upi0]) : gy[i];
}

// ------------------------------------------------------------------- gA

// W products from p on in one store (W elements of 16 bytes, or one); BETA:
// plus beta times what is there.
template <class V, int W, bool BETA>
__device__ __forceinline__ void gA_store(V* p, const V (&g)[W], const V (&x)[W], double beta) {
  V val[W];
#pragma unroll
  for (int e = 0; e < W; e++) {
    val[e] = g[e] * x[e];
    if constexpr (BETA) val[e] += (V)beta * p[e];
  }
  if constexpr (W > 1) {
    uint4 o;
    memcpy(&o, val, 16);
    __stcs(reinterpret_cast<uint4*>(p), o);
  } else {
    __stcs(p, val[0]);
  }
}

// Bound: HBM writes (128^4 FP32 158-162 us in every mode; mode 3 412 with one
// position per thread), FP64 the rate of its multiplications (33.5e6 elements
// 139 -> 71 us with eight rows unrolled).
// v >= 32: a thread owns W adjacent columns (i, l) and walks the rows j of
// its part of n_k (blockIdx.y).  W > 1: v a multiple of W, gA 16-byte aligned.
template <class V, int W, bool BETA>
__global__ void __launch_bounds__(256) tvc_gradA_cols_kernel(const V* __restrict__ gy, const V* __restrict__ x,
                                                             V* __restrict__ gA, int64_t uv, int64_t nk, int64_t v,
                                                             int64_t chunk, double beta) {
  const int64_t j0 = blockIdx.y * chunk, j1 = min(nk, j0 + chunk);
  for (int64_t o = ((int64_t)blockIdx.x * 256 + threadIdx.x) * W; o < uv; o += (int64_t)gridDim.x * 256 * W) {
    const int64_t i = o / v, l = o - i * v;
    V g[W];
#pragma unroll
    for (int e = 0; e < W; e++) g[e] = __ldg(gy + o + e);
    V* p = gA + (i * nk + j0) * v + l;
#pragma unroll 8
    for (int64_t j = j0; j < j1; j++, p += v) {
      const V xj = __ldg(x + j);
      V xs[W];
#pragma unroll
      for (int e = 0; e < W; e++) xs[e] = xj;
      gA_store<V, W, BETA>(p, g, xs, beta);
    }
  }
}

// v < 32: a thread owns W adjacent positions q = j*v + l of the slab (x_j in
// registers) and walks the slabs; a block narrower than the slab's pieces
// takes several slabs at once.  W > 1: the slab a multiple of W elements, gA
// 16-byte aligned.
template <class V, int W, bool BETA>
__global__ void __launch_bounds__(256) tvc_gradA_slab_kernel(const V* __restrict__ gy, const V* __restrict__ x,
                                                             V* __restrict__ gA, int64_t u, int64_t nk, int64_t v,
                                                             int CW, double beta) {
  const int64_t S = nk * v;
  const int P = 256 / CW, ph = threadIdx.x / CW;
  const int64_t q = ((int64_t)blockIdx.x * CW + threadIdx.x - ph * CW) * W;
  if (ph >= P || q >= S) return;
  V xs[W];
  int l[W];
#pragma unroll
  for (int e = 0; e < W; e++) {
    const int64_t j = (q + e) / v;
    xs[e] = __ldg(x + j);
    l[e] = (int)(q + e - j * v);
  }
#pragma unroll 4
  for (int64_t i = (int64_t)blockIdx.y * P + ph; i < u; i += (int64_t)gridDim.y * P) {
    V g[W];
#pragma unroll
    for (int e = 0; e < W; e++) g[e] = __ldg(gy + i * v + l[e]);
    gA_store<V, W, BETA>(gA + i * S + q, g, xs, beta);
  }
}

// ----------------------------------------------------------------- host --

namespace {

struct GxPlan {
  bool via_tvc = false;   // v == 1
  bool via_rows = false;  // mode 0, short rows
  int rch = 8;        // rows per chunk
  bool al = false;    // rows of A on 16-byte boundaries
  int64_t nchunks = 1, nblk = 1, pps = 1;
  size_t ws_partial = 0, ws_gy = 0, ws_tvc = 0, total = 0;
  Shape view;  // via_tvc: (u, nk) mode 0; via_rows: (nk, v) mode 1
};

int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

GxPlan plan_gx(const Shape& s, tvc_dtype dt, const void* A) {
  GxPlan g;
  const size_t vs = vec_size(dt);
  if (s.v == 1 && s.mode > 0) {
    g.via_tvc = true;
    const int64_t d2[2] = {s.u, s.nk};
    make_shape(2, d2, 0, &g.view);
    const tvc_dtype tdt = (dt == TVC_F64) ? TVC_F64 : dt;
    g.ws_tvc = 0;
    for (uintptr_t al = elem_size(tdt); al <= 256; al *= 2)
      g.ws_tvc = std::max(g.ws_tvc, tvc_ws_bytes(g.view, tdt, reinterpret_cast<const void*>(al)));
    if (dt == TVC_BF16 || dt == TVC_E4M3 || dt == TVC_F16) g.ws_gy = align_up((size_t)s.u * 4, 256);
    g.total = align_up(g.ws_tvc, 256) + g.ws_gy;
    return g;
  }
  const int64_t es = (int64_t)elem_size(dt);
  g.al = (s.v * es) % 16 == 0 && aligned(A, 16);
  g.pps = cdiv(s.v * es, 16);
  if (s.mode == 0 && g.pps <= 32 && vs == 4) {
    // short rows of a matrix n_k x v: gx = rows . gy, a TVC of its last mode (a
    // block here would keep a few lanes busy: 261039 entries of order one E4M3
    // 296 us, 16409x17 BF16 19)
    g.via_rows = true;
    const int64_t d2[2] = {s.nk, s.v};
    make_shape(2, d2, 1, &g.view);
    for (uintptr_t al = elem_size(dt); al <= 256; al *= 2)
      g.ws_tvc = std::max(g.ws_tvc, tvc_ws_bytes(g.view, dt, reinterpret_cast<const void*>(al)));
    g.total = g.ws_tvc;
    return g;
  }
  // One wave of blocks: chunks of 256 rows, or fewer (down to 32) where the
  // pieces alone do not fill it.
  const int64_t wave = (int64_t)device_sms() * (dt == TVC_E4M3 ? kGxBlocks<TVC_E4M3> : kGxBlocks<TVC_F32>);
  const int64_t pieces = s.u * g.pps, tiles = cdiv(pieces, kBT);
  if (vs == 8) {
    const int64_t wave = (int64_t)device_sms() * kGx64Blocks;
    // FP64 arithmetic: the cut of the rows that leaves the shortest block, in
    // rows of 256 pieces (the preparation of gy costs about two)
    int64_t cost = INT64_MAX;
    for (int64_t n = cdiv(s.nk, kGx64Rows); n <= std::min(wave, std::max(cdiv(s.nk, kGx64Rows), cdiv(s.nk, 16))); n++) {
      const int64_t rch = cdiv(cdiv(s.nk, n), 8) * 8, nch = cdiv(s.nk, rch);
      const int64_t nblk = std::max<int64_t>(1, std::min(tiles, wave / nch));
      const int64_t c = cdiv(cdiv(pieces, nblk), kBT) * (rch + 2) * std::max<int64_t>(1, cdiv(nch * nblk, wave));
      if (c < cost) {
        cost = c;
        g.rch = (int)rch;
        g.nchunks = nch;
        g.nblk = nblk;
      }
    }
    if (cost == INT64_MAX) {  // more chunks than a wave
      g.rch = kGx64Rows;
      g.nchunks = cdiv(s.nk, g.rch);
      g.nblk = 1;
    }
  } else if (tiles < wave) {
    // few pieces: the cut of the rows with the shortest time, in rows of 256
    // pieces (a tile costs about four beside its own, a block 16), down to eight rows
    // (130x260 E4M3 mode 0 11 -> 5 us)
    double cost = 0.0;
    const int64_t n0 = cdiv(s.nk, kGxRows), n1 = cdiv(s.nk, 8);
    for (int64_t n = n0;; n = std::min(n1, std::max(n + 1, n * 5 / 4))) {
      const int64_t rch = cdiv(cdiv(s.nk, n), 8) * 8, nch = cdiv(s.nk, rch);
      const int64_t nblk = std::max<int64_t>(1, std::min(tiles, wave / nch));
      const double c = (double)(cdiv(tiles, nblk) * (rch + 4) + 16) * (double)std::max<int64_t>(1, cdiv(nch * nblk, wave));
      if (n == n0 || c < cost) {
        cost = c;
        g.rch = (int)rch;
        g.nchunks = nch;
        g.nblk = nblk;
      }
      if (n == n1) break;
    }
  } else {
    g.nchunks = std::max(cdiv(s.nk, kGxRows), std::min(cdiv(s.nk, 32), wave / tiles));
    g.rch = (int)(cdiv(cdiv(s.nk, g.nchunks), 8) * 8);
    g.nchunks = cdiv(s.nk, g.rch);
    g.nblk = std::max<int64_t>(1, std::min(tiles, wave / g.nchunks));
  }
  g.ws_partial = align_up((size_t)g.nblk * s.nk * vs, 256);
  g.total = g.ws_partial;
  return g;
}

template <tvc_dtype DT>
tvc_status run_gx(const GxPlan& g, const Shape& s, const void* A, const void* gy, void* gx, const float* scales,
                  void* ws, cudaStream_t st) {
  using V = typename Elem<DT>::V;
  GradArgs<DT> a;
  a.A = static_cast<const typename Elem<DT>::T*>(A);
  a.gy = gy;
  a.scales = scales;
  a.partial = ws;
  a.u = s.u;
  a.nk = s.nk;
  a.v = s.v;
  a.pps = g.pps;
  a.nblk = g.nblk;
  a.upi0 = s.upi0 > 0 ? s.upi0 : 1;
  a.mode0 = s.mode == 0;
  a.rch = g.rch;
  const unsigned grid = (unsigned)(g.nblk * g.nchunks);
  if constexpr (kF64Acc<DT>) {
    if (g.al)
      tvc_gradx64_kernel<DT, true><<<grid, kBT, gx64_smem<DT, true>(), st>>>(a);
    else
      tvc_gradx64_kernel<DT, false><<<grid, kBT, gx64_smem<DT, false>(), st>>>(a);
  } else {
    if (g.al)
      tvc_gradx_kernel<DT, true><<<grid, kBT, 0, st>>>(a);
    else
      tvc_gradx_kernel<DT, false><<<grid, kBT, 0, st>>>(a);
  }
  tvc_gradx_reduce_kernel<V><<<(unsigned)cdiv(s.nk, 32), kBT, 0, st>>>(static_cast<const V*>(ws), static_cast<V*>(gx), s.nk, g.nblk);
  count_launches(2);
  return cuda_status(cudaGetLastError());
}

tvc_status grad_x(const Shape& s, const void* A, const void* gy, void* gx, tvc_dtype dt, const float* scales,
                  void* ws, size_t ws_bytes, cudaStream_t st) {
  const GxPlan g = plan_gx(s, dt, A);
  if (g.total > 0 && (ws == nullptr || ws_bytes < g.total)) return TVC_ERR_WORKSPACE;
  if (g.via_rows) return tvc_launch(A, g.view, gy, gx, dt, scales, 1.0, 0.0, ws, g.ws_tvc, st);
  if (g.via_tvc) {
    char* w = static_cast<char*>(ws);
    const void* gyv = gy;
    if (dt == TVC_BF16 || dt == TVC_E4M3 || dt == TVC_F16) {
      float* gys = reinterpret_cast<float*>(w + align_up(g.ws_tvc, 256));
      const int blocks = (int)std::min<int64_t>(cdiv(s.u, 256), 4096);
      tvc_scale_gy_kernel<<<blocks, 256, 0, st>>>(static_cast<const float*>(gy), scales, gys, s.u,
                                                  s.upi0 > 0 ? s.upi0 : 1);
      count_launches(1);
      gyv = gys;
    }
    // Mode 0 of the unfolded u x n_k view, the slab scales already in gy.
    return tvc_launch(A, g.view, gyv, gx, dt, nullptr, 1.0, 0.0, ws, g.ws_tvc, st);
  }
  switch (dt) {
    case TVC_F64: return run_gx<TVC_F64>(g, s, A, gy, gx, scales, ws, st);
    case TVC_F32D: return run_gx<TVC_F32D>(g, s, A, gy, gx, scales, ws, st);
    case TVC_F32: return run_gx<TVC_F32>(g, s, A, gy, gx, scales, ws, st);
    case TVC_BF16: return run_gx<TVC_BF16>(g, s, A, gy, gx, scales, ws, st);
    case TVC_E4M3: return run_gx<TVC_E4M3>(g, s, A, gy, gx, scales, ws, st);
    case TVC_F16: return run_gx<TVC_F16>(g, s, A, gy, gx, scales, ws, st);
  }
  return TVC_ERR_INVALID_ARG;
}

template <class V, int W, bool BETA>
void launch_gA_w(const Shape& s, const V* x, const V* gy, V* gA, double beta, cudaStream_t st) {
  const int64_t blocks = (int64_t)device_sms() * 16;
  if (s.v >= 32) {
    const int64_t bx = std::min<int64_t>(cdiv(s.uv, 256 * W), blocks);
    const int64_t by = std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(cdiv(s.nk, 8), 65535), blocks / bx));
    const int64_t chunk = cdiv(s.nk, by);
    tvc_gradA_cols_kernel<V, W, BETA><<<dim3((unsigned)bx, (unsigned)cdiv(s.nk, chunk)), 256, 0, st>>>(
        gy, x, gA, s.uv, s.nk, s.v, chunk, beta);
  } else {
    const int64_t pieces = s.nk * s.v / W;
    const int CW = (int)std::min<int64_t>(pieces, 256);
    const int64_t bx = cdiv(pieces, CW);
    const int64_t by = std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(cdiv(s.u, 256 / CW), 65535), blocks / bx));
    tvc_gradA_slab_kernel<V, W, BETA><<<dim3((unsigned)bx, (unsigned)by), 256, 0, st>>>(gy, x, gA, s.u, s.nk, s.v, CW,
                                                                                       beta);
  }
}

// Widest stores that the rows (v >= 32) or slabs (v < 32) allow.
template <class V, bool BETA>
void launch_gA(const Shape& s, const V* x, const V* gy, V* gA, double beta, cudaStream_t st) {
  constexpr int W = 16 / (int)sizeof(V);
  if (aligned(gA, 16) && (s.v >= 32 ? s.v : s.nk * s.v) % W == 0)
    launch_gA_w<V, W, BETA>(s, x, gy, gA, beta, st);
  else
    launch_gA_w<V, 1, BETA>(s, x, gy, gA, beta, st);
}

template <class V>
tvc_status grad_A(const Shape& s, const V* x, const V* gy, V* gA, double beta, cudaStream_t st) {
  if (beta != 0.0)
    launch_gA<V, true>(s, x, gy, gA, beta, st);
  else
    launch_gA<V, false>(s, x, gy, gA, beta, st);
  count_launches(1);
  return cuda_status(cudaGetLastError());
}

}  // namespace

size_t tvc_backward_ws_bytes(const Shape& s, tvc_dtype dt) {
  size_t need = 0;
  for (uintptr_t al = elem_size(dt); al <= 256; al *= 2)
    need = std::max(need, plan_gx(s, dt, reinterpret_cast<const void*>(al)).total);
  return need;
}

}  // namespace tvcg

using namespace tvcg;

extern "C" size_t tvc_backward_workspace_size(int order, const int64_t* dims, int mode, tvc_dtype dtype) {
  Shape s;
  if (!valid_dtype(dtype) || make_shape(order, dims, mode, &s) != TVC_OK) return 0;
  return tvc_backward_ws_bytes(s, dtype);
}

extern "C" tvc_status tvc_backward(const void* A, int order, const int64_t* dims, int mode, const void* x,
                                   const void* gy, void* gx, void* gA, tvc_dtype dtype, const float* slab_scales,
                                   double beta_A, void* workspace, size_t ws_bytes, tvc_stream_t stream) {
  if (!valid_dtype(dtype)) return TVC_ERR_INVALID_ARG;
  Shape s;
  tvc_status st = make_shape(order, dims, mode, &s);
  if (st != TVC_OK) return st;
  const size_t vs = vec_size(dtype);
  if (!gy || !aligned(gy, vs)) return TVC_ERR_INVALID_ARG;
  if (gx && (!A || !aligned(A, elem_size(dtype)) || !aligned(gx, vs))) return TVC_ERR_INVALID_ARG;
  if (gA && (!x || !aligned(x, vs) || !aligned(gA, vs))) return TVC_ERR_INVALID_ARG;
  cudaStream_t cs = (cudaStream_t)stream;
  if (gx) {
    st = grad_x(s, A, gy, gx, dtype, slab_scales, workspace, ws_bytes, cs);
    if (st != TVC_OK) return st;
  }
  if (gA) {
    if (vs == 8)  // FP64 vectors: TVC_F64, TVC_F32D
      st = grad_A<double>(s, static_cast<const double*>(x), static_cast<const double*>(gy), static_cast<double*>(gA),
                          beta_A, cs);
    else
      st = grad_A<float>(s, static_cast<const float*>(x), static_cast<const float*>(gy), static_cast<float*>(gA),
                         beta_A, cs);
  }
  return st;
}
