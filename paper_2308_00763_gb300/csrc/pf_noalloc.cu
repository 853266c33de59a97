// pf_noalloc.cu -- pf_step_frame_noalloc: one frame of the filter for callers that
// cannot allocate device memory.
//
// Some embedders cannot call cudaMalloc: a host program whose CUDA memory is owned and
// budgeted by another runtime (a graphics or inference engine that hands out buffers), a
// real-time loop that forbids allocation after start-up, or code running inside a
// stream-ordered section where an allocation would synchronise the device.  They can still
// provide their own input and output buffers; what the step needs beyond those (the
// decoupled-lookback descriptors, per-tile partial sums, counters and the tracker's
// descriptor) lives here, in a file-scope device array that exists in every GPU's memory
// as soon as the library is loaded and stays there until the process exits.
#include <cuda.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stddef.h>
#include <stdint.h>
#include <string.h>

#include <mutex>

#include "pf.h"
#include "pf_internal.h"
#include "pf_host.h"

using namespace pfk;

namespace {

constexpr int64_t kMaxParticles = int64_t(1) << 22;
// A tile holds kTile / 2 particles or more, but for the smaller tiles of a REF64 tracker, which number
// at most one a resident CTA (step_tile_size); a call whose tiles are more is refused.
constexpr int kMaxTiles = static_cast<int>(kMaxParticles / (kTile / 2));
constexpr int kMaxDevices = 64;
// tracker descriptor, state, frame and counters, then the per-tile descriptors and partials
constexpr size_t kScratchBytes = 8192 + (sizeof(LookbackDesc) + sizeof(TilePartial)) * size_t(kMaxTiles);

// The scratch array.  In host code its name is only a stand-in for the symbol; the
// device address comes from cudaGetSymbolAddress (per context).
static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

// Layout inside the scratch array.
struct ScratchLayout {
    size_t trk, state, frame, ticket, done, est, stat, look, part, end;
};

constexpr size_t align256(size_t v) { return (v + 255) & ~size_t(255); }

constexpr ScratchLayout layout() {
    ScratchLayout L{};
    L.trk = 0;
    L.state = align256(L.trk + sizeof(TrackerDev));
    L.frame = align256(L.state + sizeof(TrackerState));
    L.ticket = align256(L.frame + sizeof(FrameRef));
    L.done = L.ticket + 16;
    L.est = L.done + 16;
    L.stat = L.est + 16;
    L.look = align256(L.stat + 16);
    L.part = align256(L.look + sizeof(LookbackDesc) * kMaxTiles);
    L.end = L.part + sizeof(TilePartial) * kMaxTiles;
    return L;
}
static_assert(layout().end <= kScratchBytes, "scratch layout exceeds the array");

// What the step reads, laid out as in the scratch array, so that it is copied a word a thread:
// a structure assignment by one thread is a chain of constant-bank misses and stores.  Measured
// us a call, one thread -> a word a thread: F32 260001 particles 54.3 -> 46.9, BF16 2^21 81.2 ->
// 75.4, F16 8192 50.4 -> 46.6.  (Letting the step's blocks become resident during this launch as
// well: no gain, 47.3 and 76.8.)
struct SetupParams {
    alignas(256) TrackerDev trk;
    alignas(256) TrackerState state;
    alignas(256) FrameRef frame;
};
constexpr int kSetupWords = static_cast<int>((offsetof(SetupParams, frame) + sizeof(FrameRef)) / 8);
static_assert(offsetof(SetupParams, state) == layout().state && offsetof(SetupParams, frame) == layout().frame &&
              sizeof(FrameRef) % 8 == 0 && sizeof(SetupParams) < 4000, "the parameters mirror the scratch layout");
static_assert(kSetupWords <= 8 * 256, "a word a thread");

// Writes the tracker descriptor, its state and the frame reference into the scratch array
// and clears what every step must find at zero there (the ticket, the tile counter, the
// lookback descriptors and tile partials of the nt tiles).  The three structures travel as
// kernel parameters, so no host buffer has to outlive the call.
__global__ void noalloc_setup_kernel(const __grid_constant__ SetupParams p, unsigned char *scr, int nt) {
    constexpr ScratchLayout LY = layout();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int stride = gridDim.x * blockDim.x;
    if (i < kSetupWords) reinterpret_cast<uint64_t *>(scr + LY.trk)[i] = reinterpret_cast<const uint64_t *>(&p)[i];
    uint4 *z = reinterpret_cast<uint4 *>(scr + LY.ticket);
    for (int k = i; k < static_cast<int>((LY.est - LY.ticket) / 16); k += stride) z[k] = make_uint4(0u, 0u, 0u, 0u);
    uint4 *look = reinterpret_cast<uint4 *>(scr + LY.look);
    for (int k = i; k < nt * static_cast<int>(sizeof(LookbackDesc) / 16); k += stride) look[k] = make_uint4(0u, 0u, 0u, 0u);
    uint4 *part = reinterpret_cast<uint4 *>(scr + LY.part);
    for (int k = i; k < nt * static_cast<int>(sizeof(TilePartial) / 16); k += stride) part[k] = make_uint4(0u, 0u, 0u, 0u);
}
static_assert(sizeof(LookbackDesc) % 16 == 0 && sizeof(TilePartial) % 16 == 0, "16-byte clears");
static_assert(layout().ticket % 16 == 0 && layout().est % 16 == 0 && layout().look % 16 == 0 &&
              layout().part % 16 == 0, "16-byte aligned scratch regions");

// True if the byte ranges [a, a + n) and [b, b + n) overlap.
bool overlaps(const void *a, const void *b, size_t n) {
    const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
    return x < y + n && y < x + n;
}

// What a call needs looked up.  The scratch array is a device variable, of which every context has
// its own copy at its own address, and the step kernels' shared-memory limits are a context's
// as well; a context is known by its id, which the driver never gives out twice.
struct ContextEntry {
    unsigned long long id;
    unsigned char *scratch;   // null: the entry is free
    int grid[4];
};
std::mutex g_lock;
ContextEntry g_ctx[16] = {};   // (more contexts than this take turns and are looked up again)
int g_ctx_next = 0;

bool current_context_id(unsigned long long *id) {
    using GetId = CUresult (*)(CUcontext, unsigned long long *);
    static const GetId get = [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            f = nullptr;
        }
        return reinterpret_cast<GetId>(f);
    }();
    return get && get(nullptr, id) == CUDA_SUCCESS;
}

// Address of the scratch array in the current context and the step's grid there.
pf_status scratch_for_current_context(int precision, unsigned char **ptr_out, int *grid_out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return PF_ERR_CUDA; }
    if (dev < 0 || dev >= kMaxDevices) return PF_ERR_ARG;
    std::lock_guard<std::mutex> guard(g_lock);
    ContextEntry *e = nullptr, unknown = {};
    unsigned long long id = 0;
    if (!current_context_id(&id)) {
        e = &unknown;   // (looked up on every call)
    } else {
        for (ContextEntry &c : g_ctx)
            if (c.scratch && c.id == id) e = &c;
        if (!e) {
            e = &g_ctx[g_ctx_next];
            g_ctx_next = (g_ctx_next + 1) % static_cast<int>(sizeof(g_ctx) / sizeof(g_ctx[0]));
            *e = ContextEntry{};
            e->id = id;
        }
    }
    if (!e->scratch) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) {
            cudaGetLastError();
            return PF_ERR_CUDA;
        }
        e->scratch = static_cast<unsigned char *>(p);
    }
    if (!e->grid[precision]) {
        const int g = step_grid_size(precision, kMaxTiles);
        if (g < 1) return PF_ERR_CUDA;
        e->grid[precision] = g;
    }
    *ptr_out = e->scratch;
    *grid_out = e->grid[precision];
    return PF_OK;
}

}  // namespace

extern "C" pf_status pf_step_frame_noalloc(const pf_config *cfg, const pf_state_header *state_in,
                                           const void *x_in, const void *y_in, const void *l_in,
                                           const uint8_t *frame, int64_t pitch_bytes,
                                           void *x_out, void *y_out, void *l_out,
                                           pf_state_header *state_out, void *cuda_stream) {
    if (!cfg || !state_in || !frame || !x_out || !y_out || !l_out || !state_out) return PF_ERR_ARG;
    const pf_config &c = *cfg;
    if (c.width < 1 || c.width > 65535 || c.height < 1 || c.height > 65535) return PF_ERR_ARG;
    if (c.num_particles < 1 || c.num_particles > kMaxParticles) return PF_ERR_ARG;
    if (c.disk_radius < 0 || c.disk_radius > kMaxRadius) return PF_ERR_ARG;
    if (c.precision < PF_REF64 || c.precision > PF_BF16) return PF_ERR_ARG;
    if (!(c.sigma_x >= 0) || !(c.sigma_y >= 0) || !isfinite(c.sigma_x) || !isfinite(c.sigma_y)) return PF_ERR_ARG;
    if (!isfinite(c.init_x) || !isfinite(c.init_y) || fabs(c.init_x) > 1.0e6 || fabs(c.init_y) > 1.0e6) return PF_ERR_ARG;
    if (!isfinite(c.drift_x) || !isfinite(c.drift_y) || !isfinite(c.bg_level) || !isfinite(c.fg_level)) return PF_ERR_ARG;
    if (c.flags & ~PF_FLAG_ACCUM32) return PF_ERR_ARG;   // no debug arrays here
    if (c.resampler != PF_RESAMPLE_SYSTEMATIC && c.resampler != PF_RESAMPLE_STRATIFIED) return PF_ERR_ARG;
    if (c.resampler_steps != 0 || c.reserved != 0) return PF_ERR_ARG;
    if (pitch_bytes < c.width) return PF_ERR_ARG;
    const pf_state_header &h = *state_in;
    if (h.magic != 0x31534650u || h.precision != c.precision || h.num_particles != c.num_particles || h.t < 0)
        return PF_ERR_ARG;
    if (h.t > 0 && (!x_in || !y_in || !l_in || !(h.sum_e > 0) || !isfinite(h.max_l))) return PF_ERR_ARG;
    // the step moves particles in 16-byte vectors
    const auto misaligned = [](const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) != 0u; };
    if (misaligned(x_out) || misaligned(y_out) || misaligned(l_out)) return PF_ERR_ARG;
    if (h.t > 0 && (misaligned(x_in) || misaligned(y_in) || misaligned(l_in))) return PF_ERR_ARG;
    // the step gathers ancestors from the inputs while it writes the outputs: no buffer
    // may overlap another
    {
        const size_t nb = static_cast<size_t>(c.num_particles) * pos_bytes(c.precision);
        const void *bufs[6] = {x_out, y_out, l_out, x_in, y_in, l_in};
        const int nbuf = h.t > 0 ? 6 : 3;
        for (int a = 0; a < nbuf; ++a)
            for (int b = a + 1; b < nbuf; ++b)
                if (overlaps(bufs[a], bufs[b], nb)) return PF_ERR_ARG;
    }

    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    // the call waits for its step and reads the new state back: it cannot be captured
    {
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(stream, &cs) != cudaSuccess) { cudaGetLastError(); return PF_ERR_CUDA; }
        if (cs != cudaStreamCaptureStatusNone) return PF_ERR_ARG;
    }
    unsigned char *scr = nullptr;
    int grid = 0;
    pf_status s = scratch_for_current_context(c.precision, &scr, &grid);
    if (s != PF_OK) return s;
    constexpr ScratchLayout LY = layout();

    // descriptor of the tracker: the caller's buffers are the ping-pong slots of frame t
    const int64_t N = c.num_particles;
    const int tile = step_tile_size(c.precision, N);
    const int nt = static_cast<int>((N + tile - 1) / tile);
    if (nt > kMaxTiles) return PF_ERR_ARG;
    const int in = static_cast<int>((h.t + 1) & 1), out = static_cast<int>(h.t & 1);
    SetupParams sp;
    memset(&sp, 0, sizeof sp);
    TrackerDev &T = sp.trk;
    fill_tracker_constants(c, T);
    T.tile_begin = 0; T.ntiles = nt; T.tile = tile; T.est_cap = 1;
    T.px[in] = const_cast<void *>(x_in); T.py[in] = const_cast<void *>(y_in); T.pl[in] = const_cast<void *>(l_in);
    T.px[out] = x_out; T.py[out] = y_out; T.pl[out] = l_out;
    T.look = reinterpret_cast<LookbackDesc *>(scr + LY.look);
    T.part = reinterpret_cast<TilePartial *>(scr + LY.part);
    T.done = reinterpret_cast<uint32_t *>(scr + LY.done);
    T.state = reinterpret_cast<TrackerState *>(scr + LY.state);
    T.est_ring = reinterpret_cast<double *>(scr + LY.est);
    T.stat_ring = reinterpret_cast<double *>(scr + LY.stat);

    // the scalars the step reads (frame 0: every particle at the initial position)
    TrackerState &st = sp.state;
    st.t = h.t;
    st.epoch = 1;   // the lookback descriptors and tile partials are cleared below
    if (h.t == 0) {
        st.M = 0.0; st.S = 1.0;
        st.ax = st.nx = round_half_up(c.init_x);
        st.ay = st.ny = round_half_up(c.init_y);
        st.est_x = c.init_x; st.est_y = c.init_y;
    } else {
        st.M = h.max_l; st.S = h.sum_e;
        st.ax = h.anchor_x; st.ay = h.anchor_y; st.nx = h.next_anchor_x; st.ny = h.next_anchor_y;
        st.est_x = h.est_x; st.est_y = h.est_y;
    }
    st.invS = c.precision == PF_REF64 ? 1.0 / st.S : static_cast<double>(1.0f / static_cast<float>(st.S));
    bbox_unknown(st);   // (no tracker table here: every tile tabulates its own window)
    state_copies(st);
    FrameRef &fr = sp.frame;
    fr.base = frame; fr.pitch = pitch_bytes; fr.stride = 0; fr.active = 1;

    // Every call shares the scratch array and finds the previous call's contents in it:
    // the lookback descriptors, the tile partials (their words carry the launch counter,
    // which is 1 on every call), the tile counter and the ticket must start at zero.  One
    // small kernel writes the descriptor, state and frame reference (its parameters) and
    // clears those.
    noalloc_setup_kernel<<<8, 256, 0, stream>>>(sp, scr, nt);
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return PF_ERR_CUDA;
    if (grid > nt) grid = nt;
    StepLaunch L;
    L.trk = reinterpret_cast<const TrackerDev *>(scr + LY.trk);
    L.states = T.state;
    L.frames = reinterpret_cast<const FrameRef *>(scr + LY.frame);
    L.tile_trk = nullptr;   // one tracker: every tile belongs to it
    L.tile_prefix = nullptr;
    L.slot_of = nullptr;
    L.est_out = nullptr;
    L.ticket = reinterpret_cast<uint32_t *>(scr + LY.ticket);
    L.ntrk = 1;
    L.total_tiles = nt;
    L.frame_override = nullptr;
    L.pitch_override = 0;
    if (launch_step(c.precision, L, grid, stream) != 0) { cudaGetLastError(); return PF_ERR_CUDA; }

    // the new state header: read back once the step has run (the call waits for it), with
    // the device status a failed wait or a checked build's index test left there
    {
        TrackerState res;
        err = cudaMemcpyAsync(&res, scr + LY.state, sizeof res, cudaMemcpyDeviceToHost, stream);
        if (err == cudaSuccess) err = cudaStreamSynchronize(stream);
        if (err != cudaSuccess) { cudaGetLastError(); return PF_ERR_CUDA; }
        if (res.status & kStatusTimeout) return PF_ERR_TIMEOUT;
        if (res.status & kStatusBounds) return PF_ERR_STATE;   // checked builds
        pf_state_header o;
        memset(&o, 0, sizeof o);
        o.magic = 0x31534650u;
        o.precision = c.precision;
        o.num_particles = N;
        o.t = res.t;
        o.max_l = res.M;
        o.sum_e = res.S;
        o.anchor_x = res.ax; o.anchor_y = res.ay;
        o.next_anchor_x = res.nx; o.next_anchor_y = res.ny;
        o.est_x = res.est_x; o.est_y = res.est_y;
        *state_out = o;
    }
    return PF_OK;
}
