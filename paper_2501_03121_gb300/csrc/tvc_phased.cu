// Few outputs (v > 1): a block covers w 16-byte pieces of the outputs and P =
// 256 / w phases of rows, so that tensors whose outputs fill only part of the
// GPU still run on all of it with few partial results in memory.
//
// The column kernels give every piece of outputs one thread that walks its
// rows: few outputs left most lanes of a block idle and thousands of splits
// of the rows to be added by a second kernel, small tensors a handful of
// blocks.  Here the phases of a block meet in shared memory, in phase order.
// Bound: HBM for long rows (8388608x128 mode 0 FP32 7.0 TB/s, BF16 5.7, FP64
// 5.3), latency for small tensors (128^3: one load round and the reduction).
#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "ragged.cuh"
#include "tvc_args.cuh"

namespace tvcg {
namespace {

constexpr int kPhT = 256;

// A 16-byte piece as the compute type.
template <tvc_dtype DT>
__device__ __forceinline__ void piece(const uint4& w, typename Elem<DT>::C (&r)[16 / Elem<DT>::kSize]) {
  if constexpr (DT == TVC_F64) {
    r[0] = __hiloint2double((int)w.y, (int)w.x);
    r[1] = __hiloint2double((int)w.w, (int)w.z);
  } else if constexpr (DT == TVC_F32D) {
    Elem<TVC_F32>::decode16(w, r);
  } else {
    Elem<DT>::decode16(w, r);
  }
}

// AL: every row starts on a 16-byte boundary.  FP64 arithmetic splits x
// itself (no split pieces in memory): the block's rows of x wait in shared
// memory, kPhX at a time.
constexpr int kPhX = 1024;

template <tvc_dtype DT, bool AL>
__global__ void __launch_bounds__(kPhT, DT == TVC_E4M3 ? 2 : 3) tvc_cols_phased_kernel(const TvcArgs<DT> a, int64_t pps, int w) {
  if (skip(a.done)) return;
  using E = Elem<DT>;
  using V = typename E::V;
  constexpr int ES = E::kSize, VEC = 16 / ES, kPhRows = AL ? 8 : 4;  // rows in flight per thread
  __shared__ float2 xs[kF64Acc<DT> ? kPhX : 1];
  __shared__ V red[kPhT * VEC];
  const int t = threadIdx.x, P = kPhT / w, ph = t / w, ll = t - ph * w;
  const int64_t q = (int64_t)blockIdx.x * w + ll;
  const bool ok = q < a.u * pps;
  const int64_t i = ok ? piece_row(q, pps) : 0;
  const int64_t l = ok ? (q - i * pps) * VEC : 0;
  const int nv = (int)min((int64_t)VEC, a.v - l), bytes = nv * ES;
  const int64_t jb = (int64_t)blockIdx.y * a.chunk, je = min(a.nk, jb + a.chunk);
  const uint64_t sb = (uint64_t)a.v * ES, sp = sb * P;
  using Acc = std::conditional_t<kF64Acc<DT>, AccF64<VEC>, AccF32<VEC>>;
  Acc acc;
  acc.init();
  for (int64_t jc = jb; jc < je; jc += kPhX) {
    const int64_t j1 = min(je, jc + kPhX);
    if constexpr (kF64Acc<DT>) {
      __syncthreads();
      for (int64_t j = jc + t; j < j1; j += kPhT) {
        const XSplit p = split_x(__ldg(static_cast<const double*>(a.x) + j));
        xs[j - jc] = make_float2(p.xh, p.xl);
      }
      __syncthreads();
    }
    if (!ok) continue;
    uint64_t ad = reinterpret_cast<uint64_t>(a.A) + (uint64_t)((i * a.nk + jc + ph) * a.v + l) * ES;
    int blk = 0;
    for (int64_t j = jc + ph; j < j1; j += kPhRows * P) {
      Chunks c[kPhRows];
      uint32_t sh[kPhRows];
#pragma unroll
      for (int e = 0; e < kPhRows; e++) {
        if (j + e * P < j1) {
          if constexpr (AL)
            c[e].a = __ldcs(reinterpret_cast<const uint4*>(ad));
          else
            ld_chunks(ad, bytes, c[e]);
        }
        sh[e] = (uint32_t)ad & 15;
        ad += sp;
      }
#pragma unroll
      for (int e = 0; e < kPhRows; e++)
        if (j + e * P < j1) {
          typename E::C r[VEC];
          piece<DT>(AL ? c[e].a : cut<ES>(c[e], sh[e]), r);
          if constexpr (kF64Acc<DT>) {
            const float2 xp = xs[j + e * P - jc];
            acc.emul(r, static_cast<const double*>(a.x) + j + e * P, XSplit{xp.x, xp.y});
          } else {
            acc.mac(r, xval(a, j + e * P));
          }
        }
      if (++blk == 64 / kPhRows) {
        acc.fold();
        blk = 0;
      }
    }
    acc.fold();
  }
#pragma unroll
  for (int e = 0; e < VEC; e++) red[t * VEC + e] = acc.result(e);
  __syncthreads();
  // one output per thread, its phases in order
  for (int r = t; r < w * VEC; r += kPhT) {
    const int64_t qr = (int64_t)blockIdx.x * w + r / VEC;
    if (qr >= a.u * pps) break;
    const int64_t ir = piece_row(qr, pps);
    const int64_t lr = (qr - ir * pps) * VEC + r % VEC;
    if (lr >= a.v) continue;
    if constexpr (kF64Acc<DT>) {
      double s = red[r];
      for (int p = 1; p < P; p++) s += red[p * w * VEC + r];
      emit(a, blockIdx.y, ir * a.v + lr, s);
    } else {
      KahanF32 s;
      for (int p = 0; p < P; p++) s.add(red[p * w * VEC + r]);
      emit(a, blockIdx.y, ir * a.v + lr, __fmul_rn(s.value(), out_scale(a, ir)));
    }
  }
}

}  // namespace

template <tvc_dtype DT>
void cols_phased_launch(const TvcArgs<DT>& a, dim3 grid, int64_t pps, int w, bool al, cudaStream_t st) {
  if (al)
    tvc_cols_phased_kernel<DT, true><<<grid, kPhT, 0, st>>>(a, pps, w);
  else
    tvc_cols_phased_kernel<DT, false><<<grid, kPhT, 0, st>>>(a, pps, w);
}
template void cols_phased_launch<TVC_F64>(const TvcArgs<TVC_F64>&, dim3, int64_t, int, bool, cudaStream_t);
template void cols_phased_launch<TVC_F32>(const TvcArgs<TVC_F32>&, dim3, int64_t, int, bool, cudaStream_t);
template void cols_phased_launch<TVC_F32D>(const TvcArgs<TVC_F32D>&, dim3, int64_t, int, bool, cudaStream_t);
template void cols_phased_launch<TVC_BF16>(const TvcArgs<TVC_BF16>&, dim3, int64_t, int, bool, cudaStream_t);
template void cols_phased_launch<TVC_F16>(const TvcArgs<TVC_F16>&, dim3, int64_t, int, bool, cudaStream_t);
template void cols_phased_launch<TVC_E4M3>(const TvcArgs<TVC_E4M3>&, dim3, int64_t, int, bool, cudaStream_t);

}  // namespace tvcg
