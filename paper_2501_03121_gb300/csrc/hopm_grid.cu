// Power method of one tensor in one cooperative launch: every sweep of
// tensors small enough that launches, not memory, set the time.
//
// The schedule of hopm.cu (T = A x_1 x_1, W_1 = A x_0 x_0, W_j = W_{j-1}
// x_{j-1}, trailing contractions against the outer product of the trailing
// vectors) with d grid barriers per sweep in place of its 3d or more kernels:
// in each phase a block computes a contiguous range of the outputs of one
// contraction, contracts that range with the trailing vectors (its part of
// z_j), and after the barrier every block adds the parts and normalises for
// itself, so the vectors, the norm and the status live in every block and
// need no further exchange.  Neighbouring ranges meet in at most one entry of
// z_j, so a phase leaves blocks + n_j partial sums, at index entry + block.
// Parts and W buffers alternate between phases: a block writes one again
// only after a barrier behind its last reader.
//
// Bound: latency; about half of the 10.5 us of a phase of FP64 128^3 (FP32: 7)
// is the contraction, the rest the barrier, the parts, norm and x_j.  One block of
// 512 threads per SM: 1024 threads of 64 registers measured 30-60% slower.  See hopm_grid_wanted for the line to the queued
// kernels.  A run of a tensor beyond a few MB fills the GPU (hg_blocks), so several
// on different streams follow one another.
#include <algorithm>
#include <mutex>
#include <set>

#include "common.cuh"
#include "internal.h"
#include "ragged.cuh"
#include "tvc_args.cuh"

namespace tvcg {
namespace {

constexpr int kHgT = 512;
constexpr int kHgW = kHgT / kWarp;
constexpr int kHgMaxVec = 4096;  // vector entries (all modes, padded) held per block
constexpr int kHgRedBytes = 32 * 1024;  // phases' sums: at most 512 threads of 64 bytes
constexpr int kHgOut = 4096;            // outputs of a block held in shared memory
constexpr long long kHgWaitLimit = 4000000000LL;  // clocks a barrier is waited for
constexpr int kHgError = 41;

__device__ int g_hopm_grid_error = 0;

struct HgArgs {
  const void* A;
  int d, iters;
  int64_t dims[TVC_MAX_ORDER];
  void* x[TVC_MAX_ORDER];
  const float* scales;
  double tol;
  double* lam_out;
  int* sweeps_out;
  int* status_out;
  double* lam_hist;
  unsigned* arrived;  // barrier arrivals, zero at launch
  void *bufA, *bufB;  // T and W_j
  void* parts[2];     // partial sums of z_j: blocks + max n each
};

// Waits for `want` arrivals in all, counted modulo 2^32 (ten million sweeps of
// three modes pass it); false when the wait gave up (the error word is set, the
// block leaves).
__device__ bool grid_barrier(unsigned* arrived, unsigned want, int* flag) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(arrived, 1u);
    bool ok = true;
    const long long t0 = clock64();
    unsigned v;
    for (;;) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(arrived) : "memory");
      if (arrivals_reached(v, want)) break;
      if (clock64() - t0 > kHgWaitLimit) {
        atomicExch(&g_hopm_grid_error, kHgError);
        ok = false;
        break;
      }
    }
    *flag = ok;
  }
  __syncthreads();
  return *flag != 0;
}

// Plain FP32 sums of at most 64 products.
template <int VEC>
struct AccPlain {
  float a[VEC];
  __device__ __forceinline__ void init() {
#pragma unroll
    for (int e = 0; e < VEC; e++) a[e] = 0.0f;
  }
  __device__ __forceinline__ void mac(const float (&v)[VEC], float x) {
#pragma unroll
    for (int e = 0; e < VEC; e++) a[e] = __fmaf_rn(v[e], x, a[e]);
  }
  __device__ __forceinline__ float result(int e) const { return a[e]; }
};

// Float-float pairs of at most 64 products (common.cuh), without a branch per
// element: `bad` collects the elements outside the exact window, an entry of
// x outside its own makes the pair NaN; either way the caller computes the
// sums again with FP64 multiply-adds.
template <int VEC>
struct AccPairs {
  float s[VEC], c[VEC];
  uint32_t bad;
  __device__ __forceinline__ void init() {
    bad = 0;
#pragma unroll
    for (int e = 0; e < VEC; e++) s[e] = c[e] = 0.0f;
  }
  template <class A>
  __device__ __forceinline__ void mac(const A (&v)[VEC], XSplit x) {
#pragma unroll
    for (int e = 0; e < VEC; e++) df_step(s[e], c[e], bad, v[e], x);
  }
  __device__ __forceinline__ bool redo() const {
    bool r = bad != 0;
#pragma unroll
    for (int e = 0; e < VEC; e++) r = r || !isfinite(__fadd_rn(s[e], c[e]));
    return r;
  }
  __device__ __forceinline__ double result(int e) const { return (double)s[e] + (double)c[e]; }
};

// Decoding of a 16-byte piece into the compute type.
template <tvc_dtype DT>
__device__ __forceinline__ void decode_piece(const uint4& w, typename Elem<DT>::C (&r)[16 / Elem<DT>::kSize]) {
  if constexpr (DT == TVC_F64) {
    r[0] = __hiloint2double((int)w.y, (int)w.x);
    r[1] = __hiloint2double((int)w.w, (int)w.z);
  } else if constexpr (DT == TVC_F32D) {
    Elem<TVC_F32>::decode16(w, r);
  } else {
    Elem<DT>::decode16(w, r);
  }
}

// One phase of a sweep as a block sees it, worked out once per launch: the
// contraction over mode k of the u x nk x v view of src (A for j <= 1, else
// W_{j-1}), its pieces of `vec` outputs (pps per row of v, Q in all), the
// block's pieces [qa, qb) = outputs [oa, ob), entry z of z_j being R of them,
// and their tiling: m chunks of w pieces, P phases of rp rows.
struct HgPhase {
  int nk, nj, k;
  uint32_t u, v, pps, Q, qa, qb, oa, ob, R;
  int vec, m, w, P, rp;
};

// What a block keeps in shared memory: the vectors (V), the contracted one as
// the products want it (split pieces, or FP32 with the slab scales), the
// phases, the blocks that hold the parts of each entry, and buffers for the
// phases' partial sums and the block's outputs.
template <class V>
struct HgShared {
  V* x[TVC_MAX_ORDER];  // into xall
  uint32_t dims[TVC_MAX_ORDER];
  int at[TVC_MAX_ORDER];  // start of mode m's entries in xall
  HgPhase ph[TVC_MAX_ORDER];
  double red64[kHgW + 2];
  int flag;
  V wred[kHgW][kHgW];
  V zs[64];  // entries of z_j that a warp each summed
  uint16_t b0[kHgMaxVec], b1[kHgMaxVec];  // blocks [b0, b1] hold the parts of an entry
  alignas(16) V xall[kHgMaxVec];
  alignas(16) float2 xc[kHgMaxVec];  // XSplit, or one float each in .x
  alignas(16) V y[kHgOut];
  alignas(16) unsigned char red[kHgRedBytes];
};

// First piece of block b of B (Q pieces in all), and the block of a piece.
__device__ __forceinline__ uint32_t hg_first(uint32_t Q, int b, int B) { return (uint32_t)((uint64_t)Q * b / B); }
__device__ __forceinline__ int hg_block_of(uint32_t Q, uint32_t q, int B) {
  return (int)((((uint64_t)q + 1) * B - 1) / Q);
}

// The tiling with the fewest loads per thread; at most 64 rows per thread, so
// that a thread's sums need no folding.
__device__ void hg_tile(HgPhase& f) {
  const int n = (int)(f.qb - f.qa), Pmin = (f.nk + 63) / 64;
  const int wmax = kHgT / Pmin;
  const int m0 = max(1, (n + wmax - 1) / wmax);
  int cost = INT32_MAX;
  for (int m = m0; m < m0 + 6; m++) {
    const int w = max(1, (n + m - 1) / m);
    // Phases: up to 16, more for long contracted modes (in rows: four for a
    // chunk, one for eight phases' sums).
    for (int p = 16; p <= 128; p *= 2) {
      const int P = max(Pmin, min(p, min(kHgT / w, (f.nk + 3) / 4)));
      const int c = m * ((f.nk + P - 1) / P + 4 + (P > 16 ? P / 8 : 0));
      if (c < cost) {
        cost = c;
        f.m = m;
        f.w = w;
        f.P = P;
      }
    }
    if (w <= 8) break;
  }
  f.rp = (f.nk + f.P - 1) / f.P;
}

// prod_{m = from}^{d-1} x_m[digit_m(l)]
template <class V>
__device__ __forceinline__ V hg_outer(const HgShared<V>& s, int d, int from, uint32_t l) {
  if (from >= d) return (V)1;
  uint32_t rem = l;
  V r = (V)1;
  for (int m = d - 1; m > from; m--) {
    const uint32_t n = s.dims[m], q = rem / n;
    r *= s.x[m][rem - q * n];
    rem = q;
  }
  return r * s.x[from][rem];
}

// The block's outputs of phase f: y = src x_k x.  They go to dst (nullable)
// and, times the outer product of the vectors from mode `from` on (nothing
// for the last mode), to s.y where they fit (fits).  AL: every row of src
// starts on a 16-byte boundary.  scales (nullable): one per i.
template <tvc_dtype DT, bool AL, class V>
__device__ __noinline__ void hg_contract(HgShared<V>& s, const HgPhase& f, const void* src, const double* xd,
                                         const float* scales, V* dst, int d, int from, bool fits) {
  using E = Elem<DT>;
  constexpr int ES = E::kSize, VEC = 16 / ES, RB = 4;  // rows in flight per thread (8 spill: 5-30% slower)
  const int t = threadIdx.x, w = f.w, P = f.P;
  const int ph = t / w, ll = t - ph * w;
  const int j0 = min(f.nk, ph * f.rp), j1 = ph < P ? min(f.nk, j0 + f.rp) : j0;
  const uint64_t sb = (uint64_t)f.v * ES;
  V* const red = reinterpret_cast<V*>(s.red);  // [P][w][VEC]
  for (int c = 0; c < f.m; c++) {
    const uint32_t q = f.qa + c * w + ll;
    const bool ok = q < f.qb && ph < P;
    if (ok) {
      const uint32_t i = q / f.pps, l = (q - i * f.pps) * VEC;
      const int bytes = (int)min((uint32_t)VEC, f.v - l) * ES;
      // FP64 arithmetic: the branch-free pairs where the loads leave them room
      // (16-byte aligned rows: 128^3 42 -> 39 us per sweep, 50x20x100x76 98 ->
      // 75), the checked ones else (225x333x73: 66 against 80)
      constexpr bool kPairs = kF64Acc<DT> && AL;
      using Acc = std::conditional_t<!kF64Acc<DT>, AccPlain<VEC>, std::conditional_t<kPairs, AccPairs<VEC>, AccF64<VEC>>>;
      Acc acc;
      acc.init();
      const uint64_t ad0 = reinterpret_cast<uint64_t>(src) + (((uint64_t)i * f.nk + j0) * f.v + l) * ES;
      uint64_t ad = ad0;
      for (int j = j0; j < j1; j += RB) {
        Chunks ch[RB];
        uint32_t sh[RB];
#pragma unroll
        for (int e = 0; e < RB; e++) {
          if (j + e < j1) {
            if constexpr (AL)
              ch[e].a = __ldcg(reinterpret_cast<const uint4*>(ad));
            else
              ld_chunks(ad, bytes, ch[e]);
          }
          sh[e] = (uint32_t)ad & 15;
          ad += sb;
        }
#pragma unroll
        for (int e = 0; e < RB; e++)
          if (j + e < j1) {
            typename E::C r[VEC];
            decode_piece<DT>(AL ? ch[e].a : cut<ES>(ch[e], sh[e]), r);
            const float2 xv = s.xc[j + e];
            if constexpr (kPairs)
              acc.mac(r, XSplit{xv.x, xv.y});
            else if constexpr (kF64Acc<DT>)
              acc.emul(r, xd + j + e, XSplit{xv.x, xv.y});
            else
              acc.mac(r, xv.x);
          }
      }
      V* const o = red + (ph * w + ll) * VEC;
      if constexpr (kF64Acc<DT> && !kPairs) acc.fold();
#pragma unroll
      for (int e = 0; e < VEC; e++) o[e] = acc.result(e);
      if constexpr (kPairs) {
        if (acc.redo()) {
          const int nv = bytes / ES;
          for (int e = 0; e < nv; e++) {
            double sum = 0.0;
            for (int j = j0; j < j1; j++)
              sum = fma((double)*reinterpret_cast<const typename E::T*>(ad0 + (j - j0) * sb + e * ES), xd[j], sum);
            o[e] = sum;
          }
        }
      }
    }
    __syncthreads();
    // one output per thread: its phases' sums in phase order
    const uint32_t qc = f.qa + c * w;
    const int outs = (int)min((uint32_t)w, f.qb - qc) * VEC;
    for (int r = t; r < outs; r += kHgT) {
      const uint32_t qr = qc + r / VEC, i = qr / f.pps, l = (qr - i * f.pps) * VEC + r % VEC;
      if (l < f.v) {
        V val;
        if constexpr (kF64Acc<DT>) {
          val = red[r];
          for (int p = 1; p < P; p++) val += red[p * w * VEC + r];
        } else {
          KahanF32 k;
          for (int p = 0; p < P; p++) k.add(red[p * w * VEC + r]);
          val = k.value();
          if (scales) val *= __ldg(scales + i);
        }
        const uint32_t o = i * f.v + l;
        if (dst) dst[o] = val;
        if (fits) s.y[o - f.oa] = val * hg_outer(s, d, from, o % f.R);
      }
    }
    __syncthreads();
  }
}

// A sum in V: compensated in FP32 (z_j of few entries adds hundreds of products
// per thread, and a part per block), plain in FP64.
template <class V>
struct HgSum : KahanF32 {};
template <>
struct HgSum<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double v) { s += v; }
  __device__ __forceinline__ double value() const { return s; }
};

// The block's products (s.y, or global y times the outer product when they
// do not fit) summed per entry of z_j into part[z + block].
template <class V>
__device__ void hg_parts(HgShared<V>& s, const HgPhase& f, int d, int from, const V* y, bool fits, V* part) {
  const int t = threadIdx.x, wid = t >> 5, lane = t & 31;
  const uint32_t R = f.R, za = f.oa / R, ze = (f.ob - 1) / R + 1;
  auto term = [&](uint32_t o) { return fits ? s.y[o - f.oa] : (V)(__ldcg(y + o) * hg_outer(s, d, from, o % R)); };
  if (ze - za >= kHgW) {  // short pieces: a warp each
    for (uint32_t z = za + wid; z < ze; z += kHgW) {
      const uint32_t lb = min(f.ob, (z + 1) * R);
      HgSum<V> sum;
      for (uint32_t o = max(f.oa, z * R) + lane; o < lb; o += 32) sum.add(term(o));
      V a = sum.value();
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xFFFFFFFFu, a, off);
      if (lane == 0) part[z + blockIdx.x] = a;
    }
    return;
  }
  for (uint32_t z = za; z < ze; z++) {
    const uint32_t lb = min(f.ob, (z + 1) * R);
    HgSum<V> sum;
    for (uint32_t o = max(f.oa, z * R) + t; o < lb; o += kHgT) sum.add(term(o));
    V a = sum.value();
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xFFFFFFFFu, a, off);
    if (lane == 0) s.wred[z - za][wid] = a;
  }
  __syncthreads();
  if (wid < (int)(ze - za)) {
    V a = lane < kHgW ? s.wred[wid][lane] : (V)0;
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) a += __shfl_xor_sync(0xFFFFFFFFu, a, off);
    if (lane == 0) part[za + wid + blockIdx.x] = a;
  }
}

template <tvc_dtype DT, class V = typename Elem<DT>::V>
__global__ void __launch_bounds__(kHgT, 1) hopm_grid_kernel(const HgArgs a) {
  constexpr tvc_dtype VDT = kF64Acc<DT> ? TVC_F64 : TVC_F32;
  constexpr int ES = Elem<DT>::kSize, VS = (int)sizeof(V);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  HgShared<V>& s = *reinterpret_cast<HgShared<V>*>(smem_raw);
  const int t = threadIdx.x, B = gridDim.x, b = blockIdx.x, d = a.d;
  if (t < d) {
    const int j = t;
    int at = 0;
    for (int m = 0; m < j; m++) at += ((int)a.dims[m] + 3) / 4 * 4;
    s.at[j] = at;
    s.x[j] = s.xall + at;
    s.dims[j] = (uint32_t)a.dims[j];
    HgPhase f;
    f.k = j == 0 ? 1 : j - 1;
    f.nj = (int)a.dims[j];
    f.nk = (int)a.dims[f.k];
    f.u = j == 0 ? (uint32_t)f.nj : 1u;
    f.R = 1;
    for (int m = j < 2 ? 2 : j + 1; m < d; m++) f.R *= (uint32_t)a.dims[m];
    f.v = j == 0 ? f.R : f.nj * f.R;
    f.vec = 16 / (j <= 1 ? ES : VS);
    f.pps = (f.v + f.vec - 1) / f.vec;
    f.Q = f.u * f.pps;
    f.qa = hg_first(f.Q, b, B);
    f.qb = hg_first(f.Q, b + 1, B);
    const uint32_t ia = f.qa / f.pps, ib = f.qb / f.pps;
    f.oa = ia * f.v + (f.qa - ia * f.pps) * f.vec;
    f.ob = ib * f.v + min(f.v, (f.qb - ib * f.pps) * f.vec);
    hg_tile(f);
    s.ph[j] = f;
  }
  __syncthreads();
  for (int m = 0; m < d; m++) {
    const HgPhase& f = s.ph[m];
    for (int i = t; i < f.nj; i += kHgT) {
      s.x[m][i] = static_cast<const V*>(a.x[m])[i];
      if (m < d - 1) {
        const uint32_t q0 = m == 0 ? i * f.pps : i * f.R / f.vec;
        const uint32_t q1 = m == 0 ? q0 + f.pps - 1 : ((i + 1) * f.R - 1) / f.vec;
        s.b0[s.at[m] + i] = (uint16_t)hg_block_of(f.Q, q0, B);
        s.b1[s.at[m] + i] = (uint16_t)hg_block_of(f.Q, q1, B);
      }
    }
  }
  __syncthreads();
  unsigned want = 0;
  int status = TVC_OK, sweeps = 0, par = 0;
  double lam = 0.0;
  bool done = false;
  for (int it = 0; it < a.iters && !done; it++) {
    const void* src = a.A;
    for (int j = 0; j < d && !done; j++) {
      const HgPhase& f = s.ph[j];
      const bool last = j == d - 1;
      for (int i = t; i < f.nk; i += kHgT) {
        if constexpr (kF64Acc<DT>) {
          const XSplit p = split_x(s.x[f.k][i]);
          s.xc[i] = make_float2(p.xh, p.xl);
        } else {
          float xv = s.x[f.k][i];
          if constexpr (kNarrow<DT>) {
            if (j == 1 && a.scales) xv = __fmul_rn(xv, __ldg(a.scales + i));  // row i lies in slab i
          }
          s.xc[i] = make_float2(xv, 0.0f);
        }
      }
      __syncthreads();
      V* const part = static_cast<V*>(a.parts[par]);
      V* const W = static_cast<V*>((j & 1) || j == 0 ? a.bufA : a.bufB);
      if (f.qa < f.qb) {
        const int from = j < 2 ? 2 : j + 1;
        const bool fits = !last && f.ob - f.oa <= kHgOut;
        V* const dst = last ? part : (j == 0 && fits) ? nullptr : W;
        const float* sc = (j == 0 && kNarrow<DT>) ? a.scales : nullptr;
        const double* xd = nullptr;
        if constexpr (kF64Acc<DT>) xd = s.x[f.k];
        const bool al = ((uint64_t)f.v * (j <= 1 ? ES : VS)) % 16 == 0 && (reinterpret_cast<uintptr_t>(src) & 15) == 0;
        if (j <= 1) {
          if (al)
            hg_contract<DT, true, V>(s, f, src, xd, sc, dst, d, from, fits);
          else
            hg_contract<DT, false, V>(s, f, src, xd, sc, dst, d, from, fits);
        } else {
          if (al)
            hg_contract<VDT, true, V>(s, f, src, xd, nullptr, dst, d, from, fits);
          else
            hg_contract<VDT, false, V>(s, f, src, xd, nullptr, dst, d, from, fits);
        }
        if (!last) hg_parts<V>(s, f, d, from, W, fits, part);
      }
      if (j > 0) src = W;
      want += (unsigned)B;
      if (!grid_barrier(a.arrived, want, &s.flag)) {  // results invalid, as the error word says
        if (b == 0 && t == 0 && a.status_out) *a.status_out = TVC_ERR_TIMEOUT;
        return;
      }
      // z_j from the parts, its norm and x_j, in every block alike
      auto entry = [&](int i) {
        if (last) return __ldcg(part + i);
        const int b0 = s.b0[s.at[j] + i], b1 = s.b1[s.at[j] + i];
        HgSum<V> z;
        z.add(__ldcg(part + i + b0));
        for (int p = b0 + 1; p <= b1; p++)
          if (f.Q >= (uint32_t)B || hg_first(f.Q, p, B) < hg_first(f.Q, p + 1, B)) z.add(__ldcg(part + i + p));
        return z.value();
      };
      const bool many = !last && f.nj <= 64 && f.nj * 4 <= B;  // many parts per entry: a warp each
      if (many) {
        for (int i = t >> 5; i < f.nj; i += kHgW) {
          HgSum<V> sum;
          for (int p = s.b0[s.at[j] + i] + (t & 31); p <= s.b1[s.at[j] + i]; p += 32)
            if (hg_first(f.Q, p, B) < hg_first(f.Q, p + 1, B)) sum.add(__ldcg(part + i + p));
          V z = sum.value();
#pragma unroll
          for (int off = 16; off > 0; off >>= 1) z += __shfl_xor_sync(0xFFFFFFFFu, z, off);
          if ((t & 31) == 0) s.zs[i] = z;
        }
        __syncthreads();
      }
      // this thread's first entry
      const V z0 = t >= f.nj ? (V)0 : many ? s.zs[t] : entry(t);
      double ss = (double)z0 * (double)z0;
      for (int i = t + kHgT; i < f.nj; i += kHgT) {
        const double z = (double)entry(i);
        ss = fma(z, z, ss);
      }
      const int nw = min(kHgW, (f.nj + 31) / 32);
      if ((t >> 5) < nw) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) ss += __shfl_xor_sync(0xFFFFFFFFu, ss, off);
        if ((t & 31) == 0) s.red64[t >> 5] = ss;
      }
      __syncthreads();
      if (t < 32) {
        double sum = t < nw ? s.red64[t] : 0.0;
        for (int off = 8; off > 0; off >>= 1)
          if (nw > off) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, off);
        if (t == 0) {
          // sqrt(sum) from its reciprocal root, corrected once
          const double inv = rsqrt(sum), sg = sum * inv;
          s.red64[kHgW] = sum == 0.0 ? 0.0 : fma(fma(-sg, sg, sum), 0.5 * inv, sg);
          s.red64[kHgW + 1] = inv;
        }
      }
      __syncthreads();
      const double sigma = s.red64[kHgW], inv = s.red64[kHgW + 1];
      if (!isfinite(sigma) || sigma == 0.0) {
        status = isfinite(sigma) ? TVC_ERR_ZERO_NORM : TVC_ERR_NONFINITE;
        done = true;
      } else {
        for (int i = t; i < f.nj; i += kHgT) {
          // z / sigma: the quotient by the reciprocal, corrected once
          const double z = (double)(i < kHgT ? z0 : entry(i)), q = z * inv;
          s.x[j][i] = (V)fma(fma(-q, sigma, z), inv, q);
        }
        if (last) {
          const double prev = lam;
          sweeps++;
          lam = sigma;
          if (b == 0 && t == 0 && a.lam_hist) a.lam_hist[sweeps - 1] = sigma;
          const double scale = sigma > 1e-300 ? sigma : 1e-300;
          if (a.tol > 0.0 && sweeps >= 2 && fabs(sigma - prev) <= a.tol * scale) done = true;
        }
      }
      __syncthreads();
      par ^= 1;
    }
  }
  if (b == 0 && a.iters > 0) {
    for (int m = 0; m < d; m++)
      for (int i = t; i < s.ph[m].nj; i += kHgT) static_cast<V*>(a.x[m])[i] = s.x[m][i];
    if (t == 0) {
      if (a.lam_out) *a.lam_out = lam;
      if (a.sweeps_out) *a.sweeps_out = sweeps;
      if (a.status_out) *a.status_out = status;
    }
  }
}

template <tvc_dtype DT>
cudaError_t hg_launch(const HgArgs& a, int blocks, cudaStream_t st) {
  using V = typename Elem<DT>::V;
  const void* const kern = reinterpret_cast<const void*>(&hopm_grid_kernel<DT, V>);
  const int smem = (int)sizeof(HgShared<V>);
  {
    static std::mutex mu;
    static std::set<int> ready;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(mu);
    if (!ready.count(dev)) {
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
      if (e != cudaSuccess) return e;
      ready.insert(dev);
    }
  }
  HgArgs copy = a;
  void* args[] = {&copy};
  return cudaLaunchCooperativeKernel(kern, dim3((unsigned)blocks), dim3(kHgT), args, (size_t)smem, st);
}

}  // namespace

// Sizes the grid kernel takes: every mode's vector in shared memory and rows
// of A that are at least four pieces long; and the sizes for which it pays:
// beyond them the queued kernels, with more loads in flight per SM, win back
// what their launches cost.  us per sweep, queued / here: FP64 128^3 (17 MB)
// 121 / 32, 200x300x256 (123 MB) 144 / 97, 101x90x70x80 (407 MB) 309 / 280; FP32
// 128^3 80 / 22, 400^3 (256 MB) 158 / 161; BF16 101x90x70x80 (102 MB) 143 / 105,
// 400^3 (128 MB) 127 / 105, 989x197x570 (222 MB) 172 / 255; E4M3 400^3 (64 MB) 116 /
// 63.  Rows off 16-byte boundaries pay up to three quarters of that but for E4M3
// (425x12x101x77 FP32, 159 MB, 132 / 142; 112x192x487 FP64, 84 MB, 180 / 126), and T
// and W_1 at most 12 MB (they are written and read by every sweep: 25x2x33x804x28 E4M3, 74 MB
// of W_1, 277 / 353; 4x20x948x502 FP32, 38 MB, 196 / 248).
bool hopm_grid_wanted(int order, const int64_t* dims, tvc_dtype dt) {
  if (order < 3) return false;
  const int64_t es = (int64_t)elem_size(dt);
  int64_t most = es == 8 ? 160000000 : es >= 2 ? 104000000 : 72000000;
  int64_t N = 1, sum = 0, rest2 = 1;
  for (int m = 2; m < order; m++) {
    if (dims[m] > kHgMaxVec) return false;
    rest2 *= dims[m];
    if (rest2 > most) return false;
  }
  if (es > 1 && rest2 * es % 16 != 0) most = most / 4 * 3;
  for (int m = 0; m < order; m++) {
    if (dims[m] > kHgMaxVec) return false;
    N *= dims[m];
    if (N * es > most) return false;
    sum += (dims[m] + 3) / 4 * 4;
  }
  if (N / std::min(dims[0], dims[1]) * (int64_t)vec_size(dt) > 12000000) return false;
  return sum <= kHgMaxVec && rest2 * es >= 64;
}

// Blocks of a run: one per SM for the larger tensors, fewer for those whose
// phases are then mostly barrier, so that runs on several streams share the GPU
// (a block fills its SM).  us per sweep alone / eight runs at once, one block
// per SM -> this rule: FP64 16^3 23.6 / 23.0 -> 20.6 / 2.7, 32^3 27.8 / 27.2 -> 22.9
// / 3.0, 64^3 25.5 / 24.8 -> 25.8 / 12.6; FP32 32^3 21.0 / 20.3 -> 17.6 / 2.3, 64^3
// 19.8 / 19.0 -> 19.9 / 2.6, 100^3 21.5 / 21.1 -> 21.3 / 9.  (Queued kernels, captured,
// alone / eight at once: FP64 16^3 42 / 6.3, 64^3 70 / 10, 128^3 79 / 13 against 31 /
// 31 here, which still takes the whole GPU.)
static int hg_blocks(int64_t N, tvc_dtype dt) {
  const int64_t per = dt == TVC_F64 || dt == TVC_F32D ? 3500 : 16000;  // elements
  return (int)std::min<int64_t>(device_sms(), std::max<int64_t>(16, (N + per - 1) / per));
}

// Bytes of its partial sums and barrier word (beside T and W_j).
size_t hopm_grid_ws_bytes(int order, const int64_t* dims, tvc_dtype dt) {
  int64_t n = 1;
  for (int m = 0; m < order; m++) n = std::max(n, dims[m]);
  return 256 + 2 * align_up((size_t)(n + device_sms() + 1) * vec_size(dt), 256);
}

tvc_status hopm_grid_launch(const void* A, int order, const int64_t* dims, void* const* x, int iters, double tol,
                            double* lam_out, int* sweeps_out, int* status_out, double* lam_hist, tvc_dtype dt,
                            const float* scales, void* bufA, void* bufB, void* ws, cudaStream_t st) {
  HgArgs a{};
  a.A = A;
  a.d = order;
  a.iters = iters;
  int64_t n = 1, N = 1;
  for (int m = 0; m < order; m++) {
    a.dims[m] = dims[m];
    a.x[m] = x[m];
    n = std::max(n, dims[m]);
    N *= dims[m];
  }
  a.scales = scales;
  a.tol = tol;
  a.lam_out = lam_out;
  a.sweeps_out = sweeps_out;
  a.status_out = status_out;
  a.lam_hist = lam_hist;
  const int blocks = hg_blocks(N, dt);
  a.arrived = static_cast<unsigned*>(ws);
  const size_t part = align_up((size_t)(n + blocks + 1) * vec_size(dt), 256);
  a.parts[0] = static_cast<char*>(ws) + 256;
  a.parts[1] = static_cast<char*>(ws) + 256 + part;
  a.bufA = bufA;
  a.bufB = bufB;
  if (cudaMemsetAsync(ws, 0, 256, st) != cudaSuccess) return cuda_status(cudaGetLastError());
  cudaError_t e = cudaErrorInvalidValue;
  switch (dt) {
    case TVC_F64: e = hg_launch<TVC_F64>(a, blocks, st); break;
    case TVC_F32: e = hg_launch<TVC_F32>(a, blocks, st); break;
    case TVC_F32D: e = hg_launch<TVC_F32D>(a, blocks, st); break;
    case TVC_BF16: e = hg_launch<TVC_BF16>(a, blocks, st); break;
    case TVC_F16: e = hg_launch<TVC_F16>(a, blocks, st); break;
    case TVC_E4M3: e = hg_launch<TVC_E4M3>(a, blocks, st); break;
  }
  count_launches(1);
  if (e != cudaSuccess) cudaGetLastError();
  if (e == cudaErrorCooperativeLaunchTooLarge) return TVC_ERR_UNSUPPORTED;
  return cuda_status(e);
}

tvc_status hopm_grid_device_error(int* code_out, int clear) {
  if (cudaMemcpyFromSymbol(code_out, g_hopm_grid_error, sizeof(int)) != cudaSuccess) return TVC_ERR_CUDA;
  if (clear) {
    const int zero = 0;
    if (cudaMemcpyToSymbol(g_hopm_grid_error, &zero, sizeof(int)) != cudaSuccess) return TVC_ERR_CUDA;
  }
  return TVC_OK;
}

}  // namespace tvcg
