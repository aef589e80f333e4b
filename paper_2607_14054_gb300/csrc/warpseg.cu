// Launches of the warp-segment and streaming kernels (warpseg.cuh).
#include "sos_common.cuh"

namespace sosf {

constexpr int kWsWarps = 4;  // warps per CTA, as in warpseg.cuh
constexpr int kWsThreads = kWsWarps * 32;

const void* warpseg_fn_16(bool cr);
const void* warpseg_fn_32(bool cr);
const void* warpseg_fn_64(bool cr);
const void* stream_fn_16();
const void* stream_fn_32();
const void* stream_fn_64();

namespace {
const void* ws_fn(int N, bool cr) {
    return N == 16 ? warpseg_fn_16(cr) : N == 32 ? warpseg_fn_32(cr) : warpseg_fn_64(cr);
}
// two group slots per warp, or twelve slots for ext_n(N) (WsCfg::kSmem)
size_t ws_smem(int N) {
    const size_t own = 32 * (size_t)(N + 4) * 2 * kWsWarps;
    const size_t far = 32 * (size_t)(ext_n(N) + 4) * 12;
    return sizeof(float) * (own > far ? own : far);
}
}  // namespace

// CTAs of the warp-segment kernel (algo 2: the cyclic-reduction one)
// resident per SM of the current device, whose slot is dev (0 on error)
int warpseg_ctas_per_sm(int N, int algo, int dev) {
    static int s_occ[kDeviceSlots][2][3] = {};
    if (dev < 0) return 0;
    const int idx = N == 16 ? 0 : N == 32 ? 1 : 2, a = algo == 2 ? 1 : 0;
    if (s_occ[dev][a][idx] == 0) {
        const void* fn = ws_fn(N, a == 1);
        // all of the SM's memory as shared memory: with the default split the
        // last of the CTAs that fit may be left for a second wave
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)ws_smem(N)) != cudaSuccess ||
            cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 cudaSharedmemCarveoutMaxShared) != cudaSuccess)
            return 0;
        int occ = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, kWsThreads, ws_smem(N)) !=
            cudaSuccess)
            return 0;
        s_occ[dev][a][idx] = occ;
    }
    return s_occ[dev][a][idx];
}

int warpseg_warps_per_cta() { return kWsWarps; }

cudaError_t launch_stream(const Params& p, int64_t chunk, int64_t seg_len, int32_t maxseg,
                          int32_t foreign, cudaStream_t stream) {
    const void* fn = p.N == 16 ? stream_fn_16() : p.N == 32 ? stream_fn_32() : stream_fn_64();
    static bool attr[kDeviceSlots][3] = {};
    const int dev = p.dev;
    if (dev < 0) return cudaErrorInvalidDevice;
    const int idx = p.N == 16 ? 0 : p.N == 32 ? 1 : 2;
    if (!attr[dev][idx]) {
        const cudaError_t e =
            cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ws_smem(p.N));
        if (e != cudaSuccess) return e;
        attr[dev][idx] = true;
    }
    void* args[] = {const_cast<Params*>(&p), &chunk, &seg_len, &maxseg, &foreign};
    const int64_t warps = (int64_t)p.C * maxseg;
    const unsigned grid = (unsigned)((warps + kWsWarps - 1) / kWsWarps);
    return cudaLaunchKernel(fn, dim3(grid), dim3(kWsThreads), args, ws_smem(p.N), stream);
}

cudaError_t launch_warpseg(const Params& p, int64_t grid, cudaStream_t stream, bool early) {
    if (warpseg_ctas_per_sm(p.N, p.algo, p.dev) < 1) return cudaErrorInvalidConfiguration;
    if (grid < 1) return cudaSuccess;
    return launch_params(ws_fn(p.N, p.algo == 2), grid, kWsThreads, ws_smem(p.N), p, stream,
                         early);
}

}  // namespace sosf
