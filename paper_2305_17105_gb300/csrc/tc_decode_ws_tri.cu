// Warp-specialised tensor-core decode (FP16) with trilinear filtering.
#include "tc_decode_ws.cuh"

namespace ntc {

cudaError_t launch_decode_ws_tri(const ntc_material& m, const float* uvl, int64_t n, void* out,
                                 int out_dtype, int filter, uint64_t jkey, cudaStream_t s, bool fast) {
  return dispatch_f16<kWsTri>(m, uvl, n, out, out_dtype, filter, jkey, s, fast);
}

}  // namespace ntc
