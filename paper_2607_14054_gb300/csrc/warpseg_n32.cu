// The warp-segment and streaming kernels at N = 32 (a translation unit per N:
// they take the longest to compile).
#include "warpseg.cuh"

namespace sosf {

const void* warpseg_fn_32(bool cr) {
    return cr ? reinterpret_cast<const void*>(&sos_warpseg_kernel<32, true>)
              : reinterpret_cast<const void*>(&sos_warpseg_kernel<32, false>);
}
const void* stream_fn_32() { return reinterpret_cast<const void*>(&sos_stream_kernel<32>); }

}  // namespace sosf
