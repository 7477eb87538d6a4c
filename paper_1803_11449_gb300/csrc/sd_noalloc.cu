// sd_noalloc.cu -- sd_update_noalloc: the DHLA update (Algorithm 1) in place,
// for callers that must not allocate device memory.
//
// Who needs it: a packet-ingest thread on a latency budget (cudaMalloc can
// synchronise the whole device and take milliseconds), and programs whose
// device memory is entirely owned by another allocator (a framework's
// caching allocator, or a pool reserved at start-up) where an extra
// cudaMalloc may fail or fragment the pool.  The caller passes the pairs and
// the DHLA it owns; the entry point allocates nothing and has no scratch.
//
// The kernel is k_update with Algorithm 1's own test ("if the bit is 1,
// continue") as a cached load before each L2 reduction: a repeated bit costs
// no reduction, so neither a heavy host nor one pair repeated serialises.
// Binning by DHLA slice through a fixed 16 MiB scratch, which sweeps the
// whole DHLA once per scratch fill, was slower at every size on GB300 (us,
// slices and in place on an empty DHLA): core sketch 2^17 pairs 27 and 10,
// 2^20 123 and 112, 2^24 1654 and 1092, 2^26 6682 and 3157; 256 MiB DHLA
// 2^20 439 and 106, 2^24 8076 and 1665; one pair 2^20 times 1448 and 12.
//
// Launch failures are read from the runtime's per-thread error state, which
// also holds errors that earlier, unrelated runtime calls left there.  So a
// call first looks at that state without clearing it, and when an error is
// already pending it returns SD_ERR_CUDA with nothing queued: it neither
// reports nor consumes the caller's own error.
#include <cstring>

#include "sd.h"
#include "sd_common.cuh"

extern "C" int sd_update_noalloc(const sd_params *p, uint32_t *grid, const uint32_t *pairs, uint64_t n,
                                 void *cuda_stream) {
    using namespace sd;
    if (sd_check_params(p) != SD_OK || !grid || (n && !pairs) || ((uintptr_t)pairs & 3u) ||
        ((uintptr_t)grid & 15u))
        return SD_ERR_ARG;
    if (n == 0) return SD_OK;
    if (cudaPeekAtLastError() != cudaSuccess) return SD_ERR_CUDA;  // an earlier call's error is pending
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return SD_ERR_CUDA;
    // both buffers must be device (or managed) memory of the current device
    for (const void *ptr : {static_cast<const void *>(grid), static_cast<const void *>(pairs)}) {
        cudaPointerAttributes a;
        if (cudaPointerGetAttributes(&a, ptr) != cudaSuccess) {
            cudaGetLastError();  // the lookup's own error (none was pending before it)
            return SD_ERR_ARG;
        }
        if (a.type == cudaMemoryTypeDevice && a.device != dev) return SD_ERR_ARG;
        if (a.type != cudaMemoryTypeDevice && a.type != cudaMemoryTypeManaged) return SD_ERR_ARG;
    }

    // geometry and hash constants, as for a handle with the same parameters
    Geometry G;
    geometry_of(p, &G);
    constexpr uint64_t kMostWords = 1ull << 27;  // DHLAs of up to 512 MiB
    if ((uint64_t)G.dirs * G.dir_words > kMostWords) return SD_ERR_TOO_LARGE;

    int num_sms = 0;
    if (cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return SD_ERR_CUDA;
    // test-then-set; a short batch is spread over as many SMs as it reaches
    Tuning T;
    std::memset(&T, 0, sizeof T);
    T.mode = 1;
    const bool shorter = n < (uint64_t)num_sms * 4096;
    T.block_threads = shorter ? 128 : 512;
    T.unroll = shorter ? 1 : 2;
    return launch_update(pairs, n, grid, G, T, num_sms, (cudaStream_t)cuda_stream) == cudaSuccess ? SD_OK : SD_ERR_CUDA;
}
