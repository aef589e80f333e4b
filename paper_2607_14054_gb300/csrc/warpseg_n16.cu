// The warp-segment and streaming kernels at N = 16 (a translation unit per N:
// they take the longest to compile).
#include "warpseg.cuh"

namespace sosf {

const void* warpseg_fn_16(bool cr) {
    return cr ? reinterpret_cast<const void*>(&sos_warpseg_kernel<16, true>)
              : reinterpret_cast<const void*>(&sos_warpseg_kernel<16, false>);
}
const void* stream_fn_16() { return reinterpret_cast<const void*>(&sos_stream_kernel<16>); }

}  // namespace sosf
