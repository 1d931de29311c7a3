// Warp-specialised tensor-core decode (FP16) with stochastic filtering.
#include "tc_decode_ws.cuh"

namespace ntc {

cudaError_t launch_decode_ws_stoch(const ntc_material& m, const float* uvl, int64_t n, void* out,
                                   int out_dtype, int filter, uint64_t jkey, cudaStream_t s, bool fast) {
  return dispatch_f16<kWsStoch>(m, uvl, n, out, out_dtype, filter, jkey, s, fast);
}

}  // namespace ntc
