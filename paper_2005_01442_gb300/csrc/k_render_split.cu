// Split render (params.kernel 6, and 0 in vrc_render): two launches that bound the cost any
// one warp carries.
//
// One warp per 8 x 4 pixel tile renders a CT view's many short rays cheaply (air, rays that
// stop at a bone surface), but rays through regions of low opacity run for hundreds of
// samples, and a tile full of them keeps its warp busy for most of the frame while the rest of
// the device idles. So:
//
// 1. the per-ray body (k_ray_tile.cuh, SPLIT) sets every ray up with one lane, leaps over
//    empty bricks and composites samples 0 .. SPLIT_J0 - 1; rays that never reach a sample
//    in an occupied brick are written out, the others are appended to a queue with their
//    colour and transmittance so far and the index of that sample;
// 2. a grid sized to fill the device drains the queue, each group of SPLIT_G lanes claiming
//    one ray at a time and finishing it in blocks of SPLIT_G consecutive samples (march_block,
//    k_group.cuh) composited by a scan of the "over" operator.
//
// Each ray is composited in the same order whatever the other rays do, and with the same
// result with and without skipping (the hand-over index is fixed and blocks are aligned to
// SPLIT_G; skipped samples are exact identities in both phases).
#include "k_split.cuh"

namespace vrc {

template <bool ESL, bool CKPT>
__global__ void __launch_bounds__(32 * SPLIT_RAY_WARPS, 16 / SPLIT_RAY_WARPS)
    split_head_kernel(RenderLaunch L) {
    split_head_body<ESL, CKPT>(L);
}

// Four CTAs per SM (64 registers, a few spills): 32 resident warps hide the latency of dependent
// loads better than 24 at 80 registers (1024^2 frame of a 256^3 int16 CT / with soft tissue: 438 /
// 1290 us against 448 / 1311, with 16 at 128 registers 533 / 1515, with 40 at 48 registers, which
// spill, 461 / 1460).
// Float32 volumes with cubic taps: three, at 80 registers. Their taps take twice the registers of
// 16-bit ones, and cubic pre-classification spilled 480 bytes at 64. 640 x 512 frame of 253 x 187
// x 250, four CTAs / three: pre-classified 354 / 315 us (with soft tissue 1673 / 1376), shaded
// 178 / 179 (514 / 479), default 163 / 160 (396 / 373); at 1280 x 1024 the default takes 455 /
// 469 (1371 / 1322).
constexpr int tail_ctas_per_sm(int mode, int packed) {
    return packed == 0 && mode != MODE_LINEAR_POST && mode != MODE_LINEAR_PRE ? 3 : 4;
}
template <bool ESL, int MODE, bool CKPT, int PACKED>
__global__ void __launch_bounds__(32 * SPLIT_WARPS, tail_ctas_per_sm(MODE, PACKED))
    split_tail_kernel(RenderLaunch L) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // The counters of the stream's next render: the render before this one, which used them, has
    // ended, and the next one starts after this one. Whatever they hold, each frame starts clean.
    if (L.split.next && blockIdx.x == 0 && threadIdx.x < 3) L.split.next[threadIdx.x] = 0u;
    split_tail_body<ESL, MODE, CKPT, PACKED>(L);
}

namespace {
int sm_count(cudaError_t &e) {
    static int cached[64] = {0};
    int dev = 0;
    e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return 0;
    if (dev >= 0 && dev < 64 && cached[dev]) return cached[dev];
    int sms = 0;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return 0;
    if (dev >= 0 && dev < 64) cached[dev] = sms;
    return sms;
}
}  // namespace

template <int MODE, bool CKPT, int PACKED>
static cudaError_t launch_tail_of(const RenderLaunch &L, int sms, cudaStream_t st) {
    // launched while the first phase ends (programmatic dependent launch; it waits for that end
    // before it reads anything): a 128^2 preview takes 48.4 us instead of 51.1
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(sms * tail_ctas_per_sm(MODE, PACKED));
    cfg.blockDim = dim3(32 * SPLIT_WARPS);
    cfg.stream = st;
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return L.dist ? cudaLaunchKernelEx(&cfg, split_tail_kernel<true, MODE, CKPT, PACKED>, L)
                  : cudaLaunchKernelEx(&cfg, split_tail_kernel<false, MODE, CKPT, PACKED>, L);
}
template <int MODE, bool CKPT = false>
static cudaError_t launch_tail(const RenderLaunch &L, int sms, cudaStream_t st) {
    return L.rep.packed ? launch_tail_of<MODE, CKPT, 1>(L, sms, st)
                        : launch_tail_of<MODE, CKPT, 0>(L, sms, st);
}

cudaError_t launch_render_split(const RenderLaunch &L, cudaStream_t st) {
    cudaError_t e = cudaSuccess;
    const int sms = sm_count(e);
    if (e != cudaSuccess) return e;
    const long tiles = (long)((L.cam.width + 7) / 8) * ((L.cam.height + 3) / 4);
    const unsigned grid = (unsigned)((tiles + SPLIT_RAY_WARPS - 1) / SPLIT_RAY_WARPS);
    const bool ck = L.ckpt != nullptr;  // default variant only (checked by the caller)
    if (L.dist) {
        if (ck) split_head_kernel<true, true><<<grid, 32 * SPLIT_RAY_WARPS, 0, st>>>(L);
        else split_head_kernel<true, false><<<grid, 32 * SPLIT_RAY_WARPS, 0, st>>>(L);
    } else {
        if (ck) split_head_kernel<false, true><<<grid, 32 * SPLIT_RAY_WARPS, 0, st>>>(L);
        else split_head_kernel<false, false><<<grid, 32 * SPLIT_RAY_WARPS, 0, st>>>(L);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (ck) return launch_tail<MODE_CUBIC_POST, true>(L, sms, st);
    switch (L.mode) {
    case MODE_LINEAR_POST: return launch_tail<MODE_LINEAR_POST>(L, sms, st);
    case MODE_CUBIC_PRE: return launch_tail<MODE_CUBIC_PRE>(L, sms, st);
    case MODE_LINEAR_PRE: return launch_tail<MODE_LINEAR_PRE>(L, sms, st);
    case MODE_CUBIC_PHONG: return launch_tail<MODE_CUBIC_PHONG>(L, sms, st);
    default: return launch_tail<MODE_CUBIC_POST>(L, sms, st);
    }
}

}  // namespace vrc
