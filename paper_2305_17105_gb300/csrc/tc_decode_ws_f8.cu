// FP8-E4M3 form of the warp-specialised tensor-core decode (kind::f8f6f4),
// one instantiation per fast-layout class and the generic layout; its own
// translation units so that it compiles beside the FP16 instantiations.
#include "tc_decode_ws.cuh"

namespace ntc {

cudaError_t launch_decode_ws_f8(const ntc_material& m, const float* uvl, int64_t n, void* out,
                                int out_dtype, int filter, uint64_t jkey, cudaStream_t s) {
  switch (ws_mode(m, true, fast_layout_ok(m), filter, out_dtype)) {
    case kWsStoch: return launch_decode_ws_f8_stoch(m, uvl, n, out, out_dtype, filter, jkey, s);
    case kWsTri: return launch_decode_ws_f8_tri(m, uvl, n, out, out_dtype, filter, jkey, s);
    case kWsRows: return launch_decode_ws_f8_rows(m, uvl, n, out, out_dtype, filter, jkey, s);
    default: return dispatch_f8<kWsPlain>(m, uvl, n, out, out_dtype, filter, jkey, s);
  }
}

}  // namespace ntc
