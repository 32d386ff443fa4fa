// Tensor-matrix contraction on the CUDA cores for FP32 accumulation at any
// alignment (FP32, BF16, F16, E4M3 storage): the shapes that neither the
// tensor-core kernels nor the copy pipelines of tmc.cu take.
//
// Both kernels are register-blocked so that one shared-memory read of X
// serves several elements of A, and multiply in pairs (fma.rn.f32x2, two IEEE
// multiply-adds per instruction):
//   cols (v > 1): a thread owns four adjacent columns and the RP rows of X of
//        its pass; per row j of A it loads its elements once, reads X[.][j]
//        by broadcast and updates 4 x RP sums, pairs along r.  Fewer columns
//        than threads: phases of rows, joined in shared memory at the end.
//   rows (v == 1): four lanes share two rows of A; per four elements of a row a
//        lane reads X[r][j..j+3] once for its two rows, pairs along j.
// Aligned loads run ahead by a batch of four rows or pieces: 1024^3 FP32 mode 2, R = 16: 2610 us with the kernel before, 1090
// without loads ahead, about 1000 with; eight columns per thread and half the warps
// 1250; a ring of eight rows, each loaded when its slot is free, 1875 (waiting
// for one load then waits for younger ones too).
// Elements are loaded in windows cut out of two aligned words (see
// ragged.cuh), so rows may start anywhere.  Sums are two-level: 64 products
// in registers, the running totals in shared memory.  The passes of one tile
// (R > 16) are neighbouring blocks, so A comes from L2 for the later ones.
// Bound: the multiply-adds (0.43 ms per 1e9 elements at R = 16) and latency;
// HBM for small R.  The kernels before took one element per thread at a time
// (RP / 4 reads of X and RP multiply-adds each).
#pragma once

#include <algorithm>
#include <mutex>
#include <set>
#include <type_traits>

#include "common.cuh"
#include "internal.h"

namespace tvcg {
namespace {

constexpr int kTsT = 256;
constexpr int kTsJ = 64;    // rows j per stage of X (cols): one fold
constexpr int kTsK = 128;   // entries j per stage of X (rows)
constexpr int kTsKp = kTsK + 4;

// Resident blocks per SM: few rows of X are bound by the loads in flight.
__host__ __device__ constexpr int ts_blocks(int rp) { return rp <= 4 ? 4 : rp <= 8 ? 3 : 2; }

using u64 = unsigned long long;

__device__ __forceinline__ u64 pack2(float lo, float hi) {
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unpack2(u64 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
// Two FP32 multiply-adds in one instruction, each an IEEE fma.
__device__ __forceinline__ void fma2(u64& acc, u64 a, u64 b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}

// Raw window of BYTES bytes at ad (valid: bytes that are wanted, at least
// one): the aligned words that hold it, and the cut.
template <int BYTES>
struct Window {
  static_assert(BYTES >= 4 && BYTES <= 16, "four elements of 1, 2 or 4 bytes");
  static constexpr int N = BYTES / 4;
  uint32_t w[2 * N];

  template <bool AL>
  __device__ __forceinline__ void load(uint64_t ad, int valid) {
    const uint64_t lo = AL ? ad : ad & ~(uint64_t)(BYTES - 1);
    const bool two = !AL && (int)(ad - lo) + valid > BYTES;
    if constexpr (BYTES == 16) {
      const uint4* p = reinterpret_cast<const uint4*>(lo);
      const uint4 a = __ldcs(p);
      w[0] = a.x;
      w[1] = a.y;
      w[2] = a.z;
      w[3] = a.w;
      if constexpr (!AL) {
        const uint4 b = two ? __ldcs(p + 1) : make_uint4(0u, 0u, 0u, 0u);
        w[4] = b.x;
        w[5] = b.y;
        w[6] = b.z;
        w[7] = b.w;
      }
    } else if constexpr (BYTES == 8) {
      const uint2* p = reinterpret_cast<const uint2*>(lo);
      const uint2 a = __ldcs(p);
      w[0] = a.x;
      w[1] = a.y;
      if constexpr (!AL) {
        const uint2 b = two ? __ldcs(p + 1) : make_uint2(0u, 0u);
        w[2] = b.x;
        w[3] = b.y;
      }
    } else {
      const unsigned* p = reinterpret_cast<const unsigned*>(lo);
      w[0] = __ldcs(p);
      if constexpr (!AL) w[1] = two ? __ldcs(p + 1) : 0u;
    }
  }

  // The window's words, for an address with the low bits k.
  template <bool AL, int ES>
  __device__ __forceinline__ void cut(uint32_t k) {
    if constexpr (!AL) {
      if constexpr (N == 4) {
        if (k & 8) {
#pragma unroll
          for (int e = 0; e < 6; e++) w[e] = w[e + 2];
        }
      }
      if constexpr (N >= 2) {
        if (k & 4) {
#pragma unroll
          for (int e = 0; e <= N; e++) w[e] = w[e + 1 < 2 * N ? e + 1 : e];
        }
      }
      if constexpr (ES < 4) {
        const uint32_t s = (k & 3) * 8;
#pragma unroll
        for (int e = 0; e < N; e++) w[e] = __funnelshift_r(w[e], w[e + 1], s);
      }
    }
  }

  // The first C elements, zero from nv on.
  template <tvc_dtype DT, int C>
  __device__ __forceinline__ void decode(float (&v)[C], int nv) const {
    if constexpr (DT == TVC_F32) {
#pragma unroll
      for (int e = 0; e < C; e++) v[e] = __uint_as_float(w[e]);
    } else if constexpr (DT == TVC_E4M3) {
#pragma unroll
      for (int e = 0; e < C; e += 4) Elem<DT>::word4(w[e / 4], v + e);
    } else {
#pragma unroll
      for (int e = 0; e < C; e += 2) Elem<DT>::word2(w[e / 2], v[e], v[e + 1]);
    }
    if (nv < C) {
#pragma unroll
      for (int e = 0; e < C; e++) v[e] = e < nv ? v[e] : 0.0f;
    }
  }
};

__device__ __forceinline__ void ts_emit(const TmcSimt& a, int64_t y, float val) {
  if (a.splits > 1) {
    a.partial[blockIdx.y * a.uRv + y] = val;
  } else {
    float out = (float)a.alpha * val;
    if (a.beta != 0.0) out += (float)a.beta * a.Y[y];
    a.Y[y] = out;
  }
}

// Rows of a phase per stage of X: a multiple of the rows loaded ahead, 64 at
// most (one partial sum), about 256 over the phases (P <= 32).
__host__ __device__ inline int ts_stage_rows(int P) { return P < 4 ? kTsJ : P >= 32 ? 8 : 256 / P / 8 * 8; }

// ------------------------------------------------------------------ cols --

template <tvc_dtype DT, int RP, bool AL>
__global__ void __launch_bounds__(kTsT, ts_blocks(RP)) tmc_cols_simt_kernel(const TmcSimt a) {
  constexpr int ES = Elem<DT>::kSize, C = 4, XP = RP + 4, U = 4;  // U: rows per load batch
  using Win = Window<C * ES>;
  extern __shared__ __align__(16) float ts_smem[];
  const int t = threadIdx.x, w = a.w, P = kTsT / w, ph = t / w, ll = t - ph * w;
  const int RS = ts_stage_rows(P), SJ = RS * P;  // rows per stage of X, of one phase and in all
  float* const Xs = ts_smem;               // [SJ][XP]
  float* const tot = ts_smem + SJ * XP;    // [RP * C][kTsT] (several folds or phases only)
  const int64_t tile = blockIdx.x / a.passes;
  const int64_t r0 = (int64_t)(blockIdx.x - tile * a.passes) * RP;
  const int64_t ppr = (a.v + C - 1) / C, q = tile * w + ll;
  const bool act = ph < P && q < a.u * ppr;
  const int64_t i = act ? piece_row(q, ppr) : 0;
  const int64_t l = act ? (q - i * ppr) * C : 0;
  const int nv = act ? (int)min((int64_t)C, a.v - l) : 0;
  const int64_t j0 = (int64_t)blockIdx.y * a.chunk, j1 = min(a.nk, j0 + a.chunk);
  const uint64_t sb = (uint64_t)a.v * ES * P;
  uint64_t ad = reinterpret_cast<uint64_t>(a.A) + (uint64_t)((i * a.nk + j0 + ph) * a.v + l) * ES;
  const bool fold_scale = kNarrow<DT> && a.mode0 && a.scales;
  u64 acc[C][RP / 2];
#pragma unroll
  for (int c = 0; c < C; c++)
#pragma unroll
    for (int r = 0; r < RP / 2; r++) acc[c][r] = 0ull;
  // this thread's rows j0 + ph, j0 + ph + P, ...: `left` not loaded yet
  int64_t left = act && j0 + ph < j1 ? (j1 - j0 - ph + P - 1) / P : 0;
  Win wa[U];
  [[maybe_unused]] Win wb[U];  // AL: the batch after the one in wa, loaded ahead
  auto fetch = [&](Win (&win)[U]) {
#pragma unroll
    for (int e = 0; e < U; e++) {
      if (e < left) win[e].template load<AL>(ad, nv * ES);
      ad += sb;
    }
    left -= U;
  };
  uint64_t use = ad;  // address of the next row to multiply
  if constexpr (AL) fetch(wa);
  bool folded = false;
  auto fold = [&]() {
#pragma unroll
    for (int c = 0; c < C; c++)
#pragma unroll
      for (int r = 0; r < RP / 2; r++) {
        const float2 s = unpack2(acc[c][r]);
        float* o = tot + (c * RP + 2 * r) * kTsT + t;
        o[0] = folded ? o[0] + s.x : s.x;
        o[kTsT] = folded ? o[kTsT] + s.y : s.y;
        acc[c][r] = 0ull;
      }
    folded = true;
  };
  int cnt = 0;  // products since the last fold
  for (int64_t jc = j0; jc < j1; jc += SJ) {
    const int jn = (int)min((int64_t)SJ, j1 - jc);
    __syncthreads();  // the previous stage is consumed
    for (int x = t; x < RP * SJ; x += kTsT) {
      const int r = x / SJ, jl = x - r * SJ;
      float xv = 0.0f;
      if (r0 + r < a.R && jl < jn) {
        xv = __ldg(a.X + (r0 + r) * a.nk + jc + jl);
        if (fold_scale) xv *= __ldg(a.scales + jc + jl);  // k = 0: row j lies in slab j
      }
      Xs[jl * XP + r] = xv;
    }
    __syncthreads();
    if (!act) continue;
    const int rows = ph < jn ? (jn - ph + P - 1) / P : 0;  // RS but in the last stage
    if (cnt + rows > 64) {
      fold();
      cnt = 0;
    }
    cnt += rows;
    const float* xr = Xs + ph * XP;
    auto multiply = [&](Win (&win)[U], int n) {
#pragma unroll
      for (int e = 0; e < U; e++) {
        if (e < n) {
          win[e].template cut<AL, ES>((uint32_t)use & (C * ES - 1));
          float v[C];
          win[e].template decode<DT, C>(v, C);
          u64 vv[C];
#pragma unroll
          for (int c = 0; c < C; c++) vv[c] = pack2(v[c], v[c]);
#pragma unroll
          for (int r = 0; r < RP / 4; r++) {
            const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(xr + 4 * r);
#pragma unroll
            for (int c = 0; c < C; c++) {
              fma2(acc[c][2 * r], vv[c], x.x);
              fma2(acc[c][2 * r + 1], vv[c], x.y);
            }
          }
        }
        use += sb;
        xr += P * XP;
      }
    };
    if constexpr (AL) {
      // whole pairs of batches (2 U divides RS), so each stage starts with wa
      for (int jl = 0; jl < rows; jl += 2 * U) {
        fetch(wb);
        multiply(wa, rows - jl);
        fetch(wa);
        multiply(wb, rows - jl - U);
      }
    } else {
      // two windows per row leave no room for a batch ahead
      for (int jl = 0; jl < rows; jl += U) {
        fetch(wa);
        multiply(wa, rows - jl);
      }
    }
  }
  float sc = 1.0f;
  if constexpr (kNarrow<DT>) {
    if (act && !a.mode0 && a.scales) sc = __ldg(a.scales + i / a.upi0);
  }
  if (P == 1) {
    if (!act) return;
#pragma unroll
    for (int r = 0; r < RP / 2; r++)
#pragma unroll
      for (int c = 0; c < C; c++) {
        if (c < nv) {
          float2 s = unpack2(acc[c][r]);
          if (folded) {
            const float* o = tot + (c * RP + 2 * r) * kTsT + t;
            s.x += o[0];
            s.y += o[kTsT];
          }
          const int64_t y = (i * a.R + r0 + 2 * r) * a.v + l + c;
          if (r0 + 2 * r < a.R) ts_emit(a, y, s.x * sc);
          if (r0 + 2 * r + 1 < a.R) ts_emit(a, y + a.v, s.y * sc);
        }
      }
    return;
  }
  if (act) fold();
  __syncthreads();
  // one output per thread, its phases in order
  for (int x = t; x < w * C * RP; x += kTsT) {
    const int m = x / w, xl = x - m * w, c = m / RP, r = m - c * RP;
    const int64_t xq = tile * w + xl;
    if (xq >= a.u * ppr || r0 + r >= a.R) continue;
    const int64_t xi = xq / ppr, xc = (xq - xi * ppr) * C + c;
    if (xc >= a.v) continue;
    KahanF32 k;
    for (int p = 0; p < P; p++) k.add(tot[m * kTsT + p * w + xl]);
    float xs = 1.0f;
    if constexpr (kNarrow<DT>) {
      if (!a.mode0 && a.scales) xs = __ldg(a.scales + xi / a.upi0);
    }
    ts_emit(a, (xi * a.R + r0 + r) * a.v + xc, k.value() * xs);
  }
}

// ------------------------------------------------------------------ rows --

template <tvc_dtype DT, int RP, bool AL>
__global__ void __launch_bounds__(kTsT, ts_blocks(RP)) tmc_rows_simt_kernel(const TmcSimt a) {
  constexpr int ES = Elem<DT>::kSize, C = 4, G = 4, RB = 2, U = AL ? 4 : 2;  // U: pieces loaded ahead
  using Win = Window<C * ES>;
  extern __shared__ __align__(16) float ts_smem[];
  float* const Xt = ts_smem;                  // [RP][kTsKp]
  float* const tot = ts_smem + RP * kTsKp;    // [RB * RP][kTsT] (long rows only)
  const int t = threadIdx.x, p = t & (G - 1);
  const int64_t tile = blockIdx.x / a.passes;
  const int64_t r0 = (int64_t)(blockIdx.x - tile * a.passes) * RP;
  const int64_t row0 = tile * (kTsT / G) * RB + t / G;  // rows row0 + b * kTsT / G
  const int64_t j0 = (int64_t)blockIdx.y * a.chunk, j1 = min(a.nk, j0 + a.chunk);
  const uint64_t rb = (uint64_t)a.nk * ES;
  const uint64_t base = reinterpret_cast<uint64_t>(a.A) + (uint64_t)row0 * rb;
  const bool fold_scale = kNarrow<DT> && a.mode0 && a.scales;
  u64 acc[RB][RP];
#pragma unroll
  for (int b = 0; b < RB; b++)
#pragma unroll
    for (int r = 0; r < RP; r++) acc[b][r] = 0ull;
  int stage = 0;
  bool folded = false;
  auto fold = [&]() {  // at most 64 products per partial sum
#pragma unroll
    for (int b = 0; b < RB; b++)
#pragma unroll
      for (int r = 0; r < RP; r++) {
        const float2 s = unpack2(acc[b][r]);
        float* o = tot + (b * RP + r) * kTsT + t;
        *o = folded ? *o + (s.x + s.y) : s.x + s.y;
        acc[b][r] = 0ull;
      }
    folded = true;
  };
  // this lane's pieces j0 + p C, j0 + (p + G) C, ...: the next one to load
  int64_t next = j0 + p * C;
  bool in[RB];
#pragma unroll
  for (int b = 0; b < RB; b++) in[b] = row0 + b * (kTsT / G) < a.u;
  Win win[U][RB];
  auto fetch = [&](int e) {
    if (next < j1) {
      const int n = (int)min((int64_t)C, j1 - next);
#pragma unroll
      for (int b = 0; b < RB; b++)
        if (in[b]) win[e][b].template load<AL>(base + (uint64_t)b * (kTsT / G) * rb + (uint64_t)next * ES, n * ES);
    }
    next += G * C;
  };
#pragma unroll
  for (int e = 0; e < U; e++) fetch(e);
  for (int64_t jc = j0; jc < j1; jc += kTsK) {
    const int jn = (int)min((int64_t)kTsK, j1 - jc);
    __syncthreads();  // the previous stage is consumed
    for (int x = t; x < RP * kTsK; x += kTsT) {
      const int r = x / kTsK, jl = x % kTsK;
      float xv = 0.0f;
      if (r0 + r < a.R && jl < jn) {
        xv = __ldg(a.X + (r0 + r) * a.nk + jc + jl);
        if (fold_scale) xv *= __ldg(a.scales + jc + jl);  // order 1: entry j lies in slab j
      }
      Xt[r * kTsKp + jl] = xv;
    }
    __syncthreads();
    // kTsK / (G C) = 8 pieces per lane and stage, a multiple of U
    for (int k0 = p * C; k0 < jn; k0 += U * G * C) {
#pragma unroll
      for (int e = 0; e < U; e++) {
        const int k = k0 + e * G * C;
        if (k < jn) {
          const int nv = min(C, jn - k);
          u64 v2[RB][2];
#pragma unroll
          for (int b = 0; b < RB; b++) {
            float v[C] = {0.0f, 0.0f, 0.0f, 0.0f};
            if (in[b]) {
              const uint64_t ad = base + (uint64_t)b * (kTsT / G) * rb + (uint64_t)(jc + k) * ES;
              win[e][b].template cut<AL, ES>((uint32_t)ad & (C * ES - 1));
              win[e][b].template decode<DT, C>(v, nv);
            }
            v2[b][0] = pack2(v[0], v[1]);
            v2[b][1] = pack2(v[2], v[3]);
          }
          fetch(e);
#pragma unroll
          for (int r = 0; r < RP; r++) {
            const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(Xt + r * kTsKp + k);
#pragma unroll
            for (int b = 0; b < RB; b++) {
              fma2(acc[b][r], v2[b][0], x.x);
              fma2(acc[b][r], v2[b][1], x.y);
            }
          }
        }
      }
    }
    if (++stage == 4 && jc + kTsK < j1) {
      fold();
      stage = 0;
    }
  }
  float s[RB * RP];
#pragma unroll
  for (int b = 0; b < RB; b++)
#pragma unroll
    for (int r = 0; r < RP; r++) {
      const float2 f = unpack2(acc[b][r]);
      s[b * RP + r] = f.x + f.y;
      if (folded) s[b * RP + r] += tot[(b * RP + r) * kTsT + t];
    }
  // over the four lanes, halving the kept values: lane p keeps the quarter p
  constexpr int H = RB * RP / 2, Q = H / 2;
#pragma unroll
  for (int e = 0; e < H; e++) {
    const float mine = (p & 2) ? s[e + H] : s[e], other = (p & 2) ? s[e] : s[e + H];
    s[e] = mine + __shfl_xor_sync(0xFFFFFFFFu, other, 2);
  }
#pragma unroll
  for (int e = 0; e < Q; e++) {
    const float mine = (p & 1) ? s[e + Q] : s[e], other = (p & 1) ? s[e] : s[e + Q];
    s[e] = mine + __shfl_xor_sync(0xFFFFFFFFu, other, 1);
  }
  const int e0 = (p >> 1) * H + (p & 1) * Q;
#pragma unroll
  for (int e = 0; e < Q; e++) {
    const int b = (e0 + e) / RP, r = (e0 + e) % RP;
    const int64_t row = row0 + b * (kTsT / G);
    if (row < a.u && r0 + r < a.R) {
      float sc = 1.0f;
      if constexpr (kNarrow<DT>) {
        if (!a.mode0 && a.scales) sc = __ldg(a.scales + row / a.upi0);
      }
      ts_emit(a, row * a.R + r0 + r, s[e] * sc);
    }
  }
}

// ------------------------------------------------------------------ host --

// Most shared memory a launch with RP rows of X asks for: columns with several
// folds or phases (ts_stage_rows(P) * P <= 256 rows per stage of X).
template <int RP>
inline constexpr int kTsSmemMax = (256 * (RP + 4) + RP * 4 * kTsT) * (int)sizeof(float);

// Opts a kernel in to `bytes` of dynamic shared memory, once per kernel and
// device: the attribute belongs to the kernel, so a limit per launch would let
// one host thread lower what another is about to launch with.
inline cudaError_t smem_limit(const void* kern, int bytes) {
  static std::mutex mu;
  static std::set<std::pair<int, const void*>> done;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lk(mu);
  if (done.count({dev, kern})) return cudaSuccess;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) done.insert({dev, kern});
  return e;
}

template <tvc_dtype DT, int RP>
tvc_status launch_rp(const TmcSimt& a, bool al, cudaStream_t st) {
  const dim3 grid((unsigned)(a.blocks_x * a.passes), (unsigned)a.splits);
  size_t smem;
  void (*kern)(const TmcSimt);
  if (a.v == 1) {
    smem = ((size_t)RP * kTsKp + (a.chunk > 4 * kTsK ? (size_t)2 * RP * kTsT : 0)) * sizeof(float);
    kern = al ? tmc_rows_simt_kernel<DT, RP, true> : tmc_rows_simt_kernel<DT, RP, false>;
  } else {
    const int P = kTsT / a.w;
    smem = ((size_t)ts_stage_rows(P) * P * (RP + 4) + (P > 1 || a.chunk > 64 ? (size_t)RP * 4 * kTsT : 0)) * sizeof(float);
    if constexpr (RP > 4)
      kern = al ? tmc_cols_simt_kernel<DT, RP, true> : tmc_cols_simt_kernel<DT, RP, false>;
    else
      return TVC_ERR_UNSUPPORTED;  // columns against up to four rows of X stay with tmc.cu
  }
  const cudaError_t e = smem_limit(reinterpret_cast<const void*>(kern), kTsSmemMax<RP>);
  if (e != cudaSuccess) return cuda_status(e);
  kern<<<grid, kTsT, smem, st>>>(a);
  return cuda_status(cudaGetLastError());
}

template <tvc_dtype DT>
tvc_status launch_dt(const TmcSimt& a, bool al, cudaStream_t st) {
  switch (a.rp) {
    case 4: return launch_rp<DT, 4>(a, al, st);
    case 8: return launch_rp<DT, 8>(a, al, st);
    case 12: return launch_rp<DT, 12>(a, al, st);
    default: return launch_rp<DT, 16>(a, al, st);
  }
}

}  // namespace

}  // namespace tvcg
