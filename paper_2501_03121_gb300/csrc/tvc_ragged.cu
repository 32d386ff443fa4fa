// Contractions whose rows do not start on 16-byte boundaries (row lengths
// that are not whole 16-byte pieces, or a tensor that starts off one): the
// column kernel (v >= 32) and the row kernel (v == 1) with 16-byte loads at
// any alignment.
//
// A thread's 16 bytes of a row are cut out of the two aligned 16-byte chunks
// that hold them: the chunks are loaded (the second only when it holds a
// wanted byte, so nothing beyond the tensor's last 16-byte granule is
// touched) and shifted together in registers.  A warp's second chunks are its
// first ones one lane further, so they hit L1 and the traffic from L2 stays
// that of the row.  The kernels these shapes had before load one or two
// elements at a time, which is bound by instructions and by bytes in flight:
// BF16 175^4 modes 0-2 3.9 TB/s -> 6.5, E4M3 979^3 modes 0, 1 1.9 -> 4.6, FP32
// 63^5 modes 0-2 6.0 -> 6.7.
#include "common.cuh"
#include "internal.h"
#include "ragged.cuh"
#include "tvc_args.cuh"

namespace tvcg {
namespace {

constexpr int kRgThreads = 256;
constexpr int kRgRowBatch = kRaggedRowBatch;
// Products per lane and row between folds (two partial sums of half as many
// each): short chains, so that the error of a row stays that of the kernels
// with 32 lanes per row (BF16 rows of 175: 7.5e-8 relative; 64 products:
// 9.5e-8), at 1-3% of the rate.
template <tvc_dtype DT>
inline constexpr int kRgRowFold = DT == TVC_F32 ? 8 : 16;

// Rows in flight per thread (two chunks each) and resident blocks per SM of
// the column kernel, the fastest of the pairs that fit the registers (GB/s on
// 63^5 FP32 mode 0 / 175^4 BF16 mode 0 / 979^3 E4M3 mode 0): 4 rows x 5
// blocks 6756 / 5795 / -, 4 x 6 6402 / 6122 / -, 6 x 4 6715 / 6543 / -, 8 x 3
// 5632 / 6532 / -; E4M3 4 x 3 4616, 4 x 4 4606, 6 x 2 4437, 8 x 2 4553.  FP32
// takes 6 x 4 for its shorter rows (v = 63, n_k = 64: 6273 against 5940).
template <tvc_dtype DT>
inline constexpr int kRgRows = DT == TVC_E4M3 ? 4 : 6;
template <tvc_dtype DT>
inline constexpr int kRgBlocks = DT == TVC_E4M3 ? 3 : 4;

// ------------------------------------------------------------------ COLS --

// One thread owns the 16-byte piece p of the columns of slab i (the last
// piece of a row may be partial) and walks the rows of its part of n_k.
template <tvc_dtype DT>
__global__ void __launch_bounds__(kRgThreads, kRgBlocks<DT>) tvc_cols_ragged_kernel(const TvcArgs<DT> a, int64_t pps) {
  if (skip(a.done)) return;
  using E = Elem<DT>;
  constexpr int ES = E::kSize, VEC = 16 / ES;
  const int64_t q = (int64_t)blockIdx.x * kRgThreads + threadIdx.x;
  if (q >= a.u * pps) return;
  const int64_t i = piece_row(q, pps);
  const int64_t l = (q - i * pps) * VEC;
  const int nv = (int)min((int64_t)VEC, a.v - l), bytes = nv * ES;
  const int64_t j0 = (int64_t)blockIdx.y * a.chunk, j1 = min(a.nk, j0 + a.chunk);
  const uint64_t sb = (uint64_t)a.v * ES;
  uint64_t ad = reinterpret_cast<uint64_t>(a.A) + (uint64_t)((i * a.nk + j0) * a.v + l) * ES;
  const int64_t o = i * a.v + l;
  // Plain sums of up to 64 products in registers, folded into compensated pairs
  // that wait in shared memory (they are touched once per 64 rows; in
  // registers they would take the room of the loads in flight).
  extern __shared__ float2 pairs[];  // [VEC][threads]
  float2* const my = pairs + threadIdx.x;
  float s[VEC];
#pragma unroll
  for (int e = 0; e < VEC; e++) {
    s[e] = 0.0f;
    my[e * kRgThreads] = make_float2(0.0f, 0.0f);
  }
  int blk = 0;
  auto fold = [&]() {
#pragma unroll
    for (int e = 0; e < VEC; e++) {
      const float2 t = my[e * kRgThreads];
      float sum, err;
      two_sum(t.x, s[e], sum, err);
      my[e * kRgThreads] = make_float2(sum, __fadd_rn(t.y, err));
      s[e] = 0.0f;
    }
  };
  auto mac = [&](const Chunks& c, uint64_t at, int64_t j) {
    float r[VEC];
    E::decode16(cut<ES>(c, (uint32_t)at & 15), r);
    const float xv = xval(a, j);
#pragma unroll
    for (int e = 0; e < VEC; e++) s[e] = __fmaf_rn(r[e], xv, s[e]);
  };
  constexpr int RB = kRgRows<DT>;
  int64_t j = j0;
  for (; j + RB <= j1; j += RB, ad += RB * sb) {
    Chunks c[RB];
#pragma unroll
    for (int e = 0; e < RB; e++) ld_chunks(ad + e * sb, bytes, c[e]);
#pragma unroll
    for (int e = 0; e < RB; e++) mac(c[e], ad + e * sb, j + e);
    if (++blk == 64 / RB) {
      fold();
      blk = 0;
    }
  }
  if (j < j1) {
    Chunks c[RB - 1];
#pragma unroll
    for (int e = 0; e < RB - 1; e++)
      if (j + e < j1) ld_chunks(ad + e * sb, bytes, c[e]);
#pragma unroll
    for (int e = 0; e < RB - 1; e++)
      if (j + e < j1) mac(c[e], ad + e * sb, j + e);
  }
  fold();
  const float sc = out_scale(a, i);
#pragma unroll
  for (int e = 0; e < VEC; e++)
    if (e < nv) {
      const float2 t = my[e * kRgThreads];
      emit(a, blockIdx.y, o + e, __fmul_rn(pair_value(t.x, t.y), sc));
    }
}

// ------------------------------------------------------------------ ROWS --

// G lanes (a power of two) share a row, lane p taking its 16-byte pieces p,
// p + G, ...; a group walks four rows at once, so that the entries of x of a
// piece, in registers, serve four rows (FP32 accumulation; two rows measured
// 5-15% slower on rows of 100 elements and more).  GB/s on 0.3e9 elements,
// before -> now: rows of 63 FP32 3445 -> 4421, BF16 2007 -> 3462, E4M3 1203 ->
// 2541; of 331 4032 -> 5096, 1612 -> 4081, 929 -> 2944; of 979 4529 -> 5547,
// 2118 -> 4574, 1343 -> 3265.  Three resident blocks (E4M3: 98 -> 80
// registers): rows of 979 E4M3 2849 -> 3265.
// Ordinary loads but for E4M3: a row's last chunk is the next row's first, and
// a neighbouring group may reach it when an evict-first line is gone (rows of
// 63 FP32 854 -> 787 us on 4.0 GB; every mode of 63^5 in turn 3313 -> 3165, of
// BF16 175^4 1402 -> 1349, of E4M3 979^3 675 -> 681).  The columns, 3-10% slower
// with them, keep evict-first (F16 972980x347 mode 0 230 against 252 us).
template <tvc_dtype DT>
__global__ void __launch_bounds__(kRgThreads, 3) tvc_rows_ragged_kernel(const TvcArgs<DT> a, int G) {
  if (skip(a.done)) return;
  using E = Elem<DT>;
  constexpr int ES = E::kSize, VEC = 16 / ES, RB = kRgRowBatch;
  const int lane = threadIdx.x & 31, p = lane & (G - 1), gw = kWarp / G;
  // rows row0 + b * gw, b < RB: neighbouring groups take neighbouring rows
  const int64_t w = (int64_t)blockIdx.x * (kRgThreads / kWarp) + (threadIdx.x >> 5);
  const int64_t row0 = w * gw * RB + lane / G;
  const int64_t j0 = (int64_t)blockIdx.y * a.chunk, j1 = min(a.nk, j0 + a.chunk);
  const uint64_t rb = (uint64_t)a.nk * ES;
  const uint64_t base = reinterpret_cast<uint64_t>(a.A) + (uint64_t)row0 * rb;
  AccF32<RB> acc;  // even products, and the folded sums
  acc.init();
  float odd[RB] = {};
  auto fold = [&]() {
#pragma unroll
    for (int b = 0; b < RB; b++) {
      acc.a[b] = __fadd_rn(acc.a[b], odd[b]);
      odd[b] = 0.0f;
    }
    acc.fold();
  };
  int blk = 0;
  for (int64_t j = j0 + p * VEC; j < j1; j += (int64_t)G * VEC) {
    const int nv = (int)min((int64_t)VEC, j1 - j);
    Chunks c[RB];
#pragma unroll
    for (int b = 0; b < RB; b++) {
      c[b].a = c[b].b = make_uint4(0u, 0u, 0u, 0u);
      if (row0 + b * gw < a.u) ld_chunks<DT != TVC_E4M3>(base + b * gw * rb + (uint64_t)j * ES, nv * ES, c[b]);
    }
    float xq[VEC];
    if (nv == VEC) {
      xvec<DT, VEC>(a, j, xq);
    } else {
#pragma unroll
      for (int e = 0; e < VEC; e++) xq[e] = e < nv ? xval(a, j + e) : 0.0f;
    }
#pragma unroll
    for (int b = 0; b < RB; b++) {
      float r[VEC];
      E::decode16(cut<ES>(c[b], (uint32_t)(base + b * gw * rb + (uint64_t)j * ES) & 15), r);
      if (nv < VEC) {  // what follows the row is another row: not its products
#pragma unroll
        for (int e = 0; e < VEC; e++) r[e] = e < nv ? r[e] : 0.0f;
      }
#pragma unroll
      for (int e = 0; e < VEC; e += 2) {
        acc.a[b] = __fmaf_rn(r[e], xq[e], acc.a[b]);
        odd[b] = __fmaf_rn(r[e + 1], xq[e + 1], odd[b]);
      }
    }
    if ((blk += VEC) >= kRgRowFold<DT>) {
      fold();
      blk = 0;
    }
  }
  fold();
#pragma unroll
  for (int b = 0; b < RB; b++) {
    float t = acc.result(b);
    for (int off = G / 2; off > 0; off >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, off);
    const int64_t row = row0 + b * gw;
    if (p == 0 && row < a.u) emit(a, blockIdx.y, row, __fmul_rn(t, out_scale(a, row)));
  }
}

}  // namespace

template <tvc_dtype DT>
void cols_ragged_launch(const TvcArgs<DT>& a, dim3 grid, int64_t pps, cudaStream_t st) {
  constexpr int bytes = 16 / Elem<DT>::kSize * kRgThreads * (int)sizeof(float2);
  tvc_cols_ragged_kernel<DT><<<grid, kRgThreads, bytes, st>>>(a, pps);
}
template void cols_ragged_launch<TVC_F32>(const TvcArgs<TVC_F32>&, dim3, int64_t, cudaStream_t);
template void cols_ragged_launch<TVC_BF16>(const TvcArgs<TVC_BF16>&, dim3, int64_t, cudaStream_t);
template void cols_ragged_launch<TVC_F16>(const TvcArgs<TVC_F16>&, dim3, int64_t, cudaStream_t);
template void cols_ragged_launch<TVC_E4M3>(const TvcArgs<TVC_E4M3>&, dim3, int64_t, cudaStream_t);

template <tvc_dtype DT>
void rows_ragged_launch(const TvcArgs<DT>& a, dim3 grid, int G, cudaStream_t st) {
  tvc_rows_ragged_kernel<DT><<<grid, kRgThreads, 0, st>>>(a, G);
}
template void rows_ragged_launch<TVC_F32>(const TvcArgs<TVC_F32>&, dim3, int, cudaStream_t);
template void rows_ragged_launch<TVC_BF16>(const TvcArgs<TVC_BF16>&, dim3, int, cudaStream_t);
template void rows_ragged_launch<TVC_F16>(const TvcArgs<TVC_F16>&, dim3, int, cudaStream_t);
template void rows_ragged_launch<TVC_E4M3>(const TvcArgs<TVC_E4M3>&, dim3, int, cudaStream_t);

}  // namespace tvcg
