// FP32 and BF16 instances of the register-blocked tensor-matrix contraction
// (tmc_simt.cuh), and its planning helpers.
#include "tmc_simt.cuh"

namespace tvcg {

// Rows of X per pass: the fewest passes of at most 16, evenly filled.
int tmc_simt_rp(int64_t R) {
  const int64_t passes = (R + 15) / 16;
  return (int)(((R + passes - 1) / passes + 3) / 4 * 4);
}

int tmc_simt_resident(int rp) { return ts_blocks(rp); }

// Pieces of four columns per tile (v > 1): all of them when there are fewer
// than threads, which then take phases of rows (at most 32).
int tmc_simt_width(int64_t u, int64_t v) {
  return (int)std::max<int64_t>(8, std::min<int64_t>(kTsT, u * ((v + 3) / 4)));
}

// Blocks along the outputs.
int64_t tmc_simt_blocks(int64_t u, int64_t v) {
  if (v == 1) return (u + kTsT / 2 - 1) / (kTsT / 2);
  const int64_t pieces = u * ((v + 3) / 4), w = tmc_simt_width(u, v);
  return (pieces + w - 1) / w;
}

tvc_status tmc_simt_launch(const TmcSimt& a, tvc_dtype dt, cudaStream_t st) {
  const int64_t es = (int64_t)elem_size(dt), bytes = 4 * es;  // of a window
  const bool al = ((a.v == 1 ? a.nk : a.v) * es) % bytes == 0 && aligned(a.A, (size_t)bytes);
  switch (dt) {
    case TVC_F32: return launch_dt<TVC_F32>(a, al, st);
    case TVC_BF16: return launch_dt<TVC_BF16>(a, al, st);
    case TVC_F16:
    case TVC_E4M3: return tmc_simt_launch_narrow(a, dt, al, st);
    default: return TVC_ERR_INVALID_ARG;
  }
}

}  // namespace tvcg
