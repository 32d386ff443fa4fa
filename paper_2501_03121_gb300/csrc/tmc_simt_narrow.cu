// F16 and E4M3 instances of the register-blocked tensor-matrix contraction
// (tmc_simt.cuh), apart so that the two halves compile side by side.
#include "tmc_simt.cuh"

namespace tvcg {

tvc_status tmc_simt_launch_narrow(const TmcSimt& a, tvc_dtype dt, bool al, cudaStream_t st) {
  return dt == TVC_F16 ? launch_dt<TVC_F16>(a, al, st) : launch_dt<TVC_E4M3>(a, al, st);
}

}  // namespace tvcg
