// FP8-E4M3 form of the warp-specialised decode with stochastic filtering.
#include "tc_decode_ws.cuh"

namespace ntc {

cudaError_t launch_decode_ws_f8_stoch(const ntc_material& m, const float* uvl, int64_t n, void* out,
                                      int out_dtype, int filter, uint64_t jkey, cudaStream_t s) {
  return dispatch_f8<kWsStoch>(m, uvl, n, out, out_dtype, filter, jkey, s);
}

}  // namespace ntc
