// pf_batch.cu -- what a set of trackers does outside its steps, one launch for all of them:
// back to frame 0, and one frame's estimates gathered from the trackers' rings.
//
// Both are bound by launch and copy latency, not by their few kilobytes.  One kernel takes the
// place of three stream operations a tracker (reset) and of two blocking copies a tracker
// (estimates): 256 trackers reset, stepped 6
// frames and read with 6 calls took 30 ms, 1.3 ms with these.
#include <stddef.h>

#include <algorithm>

#include "pf_internal.h"

namespace pfk {
namespace {

constexpr int kResetThreads = 128;

// Block (i, y): tracker i's state (y = 0) and every gridDim.y-th part of its descriptors.
__global__ void __launch_bounds__(kResetThreads) reset_kernel(const TrackerDev *trk, const TrackerState *init) {
    const int i = static_cast<int>(blockIdx.x);
    TrackerState *st = trk[i].state;
    if (blockIdx.y == 0) {
        // (the state is 8-byte words; t is the first, epoch and status the second)
        static_assert(offsetof(TrackerState, t) == 0 && offsetof(TrackerState, M) == 16 && sizeof(TrackerState) % 8 == 0,
                      "word copies of the state skip the launch counter and the status word");
        const int k = static_cast<int>(threadIdx.x);
        if (k < static_cast<int>(sizeof(TrackerState) / 8) && k != 1)
            reinterpret_cast<uint64_t *>(st)[k] = reinterpret_cast<const uint64_t *>(init + i)[k];
    }
    const int words = trk[i].ntiles * static_cast<int>(sizeof(LookbackDesc) / 16);
    uint4 *look = reinterpret_cast<uint4 *>(trk[i].look);
    for (int k = static_cast<int>(blockIdx.y * blockDim.x + threadIdx.x); k < words;
         k += static_cast<int>(gridDim.y * blockDim.x))
        look[k] = make_uint4(0u, 0u, 0u, 0u);
}

__global__ void gather_estimates_kernel(const TrackerDev *trk, int n, int64_t frame, double *out) {
    const int i = static_cast<int>(blockIdx.x * blockDim.x + threadIdx.x);
    if (i >= n) return;
    const double *e = trk[i].est_ring + 2 * (frame % trk[i].est_cap);
    out[2 * i] = e[0];
    out[2 * i + 1] = e[1];
}

}  // namespace

int launch_reset(const TrackerDev *trk, const TrackerState *init, int n, int max_tiles, void *stream) {
    const int64_t words = static_cast<int64_t>(max_tiles) * static_cast<int64_t>(sizeof(LookbackDesc) / 16);
    const unsigned parts = static_cast<unsigned>(std::min<int64_t>(32, std::max<int64_t>(1, words / (2 * kResetThreads))));
    reset_kernel<<<dim3(static_cast<unsigned>(n), parts), kResetThreads, 0, static_cast<cudaStream_t>(stream)>>>(trk, init);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

int launch_gather_estimates(const TrackerDev *trk, int n, int64_t frame, double *out, void *stream) {
    const unsigned blocks = static_cast<unsigned>((n + 127) / 128);
    gather_estimates_kernel<<<blocks, 128, 0, static_cast<cudaStream_t>(stream)>>>(trk, n, frame, out);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

}  // namespace pfk
