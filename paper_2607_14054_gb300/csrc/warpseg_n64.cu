// The warp-segment and streaming kernels at N = 64 (a translation unit per N:
// they take the longest to compile).
#include "warpseg.cuh"

namespace sosf {

const void* warpseg_fn_64(bool cr) {
    return cr ? reinterpret_cast<const void*>(&sos_warpseg_kernel<64, true>)
              : reinterpret_cast<const void*>(&sos_warpseg_kernel<64, false>);
}
const void* stream_fn_64() { return reinterpret_cast<const void*>(&sos_stream_kernel<64>); }

}  // namespace sosf
