// The two phases of the split render as device functions, shared by the split render's own
// kernels (k_render_split.cu) and by the kernels that serving launches on the device
// (k_serve_dl.cu). The algorithm is described in k_render_split.cu.
#pragma once

#include "k_group.cuh"
#include "k_ray_tile.cuh"

namespace vrc {

constexpr int SPLIT_RAY_WARPS = 4;  // warps per CTA of the first phase (2: 0.3% slower)
constexpr int SPLIT_WARPS = 8;      // warps per CTA of the second phase
constexpr int SPLIT_CLAIM = 1;      // queued rays a group claims per atomic (more: the long
                                    // rays of a claim serialise and the frame waits on them)

// First phase: the calling CTA's SPLIT_RAY_WARPS tiles of 8 x 4 pixels.
template <bool ESL, bool CKPT>
__device__ __forceinline__ void split_head_body(const RenderLaunch &L) {
    render_ray_tile<ESL, true, MODE_CUBIC_POST, CKPT>(L, blockIdx.x * SPLIT_RAY_WARPS +
                                                             (threadIdx.x >> 5));
}

// Second phase: the calling CTA's groups of SPLIT_G lanes drain the queue.
template <bool ESL, int MODE, bool CKPT = false, int PACKED = -1>
__device__ __forceinline__ void split_tail_body(const RenderLaunch &L) {
    constexpr int G = SPLIT_G;
    // per group: the entry point and inverse direction that leaps use, kept out of registers
    __shared__ float s_leap[SPLIT_WARPS * 32 / G][8];
    const int lane = threadIdx.x & 31;
    const int q = lane & (G - 1);       // lane within the group
    const int gbase = lane & ~(G - 1);  // first lane of the group
    const unsigned gmask = G == 32 ? 0xffffffffu : (((1u << G) - 1u) << gbase);
    const float inv_step = 1.0f / L.grid.step;
    const long nbricks = ESL ? (long)L.bricks.nb[0] * L.bricks.nb[1] * L.bricks.nb[2] : 0;
    // final counts (the first phase has finished): front records 0 .. nf-1, then back
    // records cap-1 down to cap-nb
    const unsigned nf = __ldcg(&L.split.head[0]), nb = __ldcg(&L.split.head[2]);
    const unsigned total = min(nf + nb, L.split.cap);
    __shared__ unsigned long long s_count[SPLIT_WARPS * 32 / G][2];  // executed, resampled
    if (q == 0) s_count[threadIdx.x / G][0] = s_count[threadIdx.x / G][1] = 0;
    unsigned next = 0, end = 0;  // rays claimed by this group and not yet started
    while (true) {
        if (next == end) {  // claim SPLIT_CLAIM consecutive rays with one atomic
            unsigned qi = 0;
            if (q == 0) qi = atomicAdd(&L.split.head[1], (unsigned)SPLIT_CLAIM);
            next = __shfl_sync(gmask, qi, 0, G);
            end = min(next + SPLIT_CLAIM, total);
        }
        const unsigned c = next++;
        if (c >= total) break;
        const unsigned qi = c < nf ? c : L.split.cap - 1u - (c - nf);
        RayPos rp;
        int jlo, pix;
        float RC0, RC1, RC2, RT;
        split_load(L.split.rec + (long)qi * SPLIT_REC, rp, jlo, pix, RC0, RC1, RC2, RT);
        const float df[3] = {rp.d[0].hi, rp.d[1].hi, rp.d[2].hi};
        float *leap = s_leap[threadIdx.x / G];
        if (ESL) {
            __syncwarp(gmask);  // the ray before is done with it
            if (q == 0) {
                float Pf[3], d[3], inv_df[3];
                ray_float(rp, Pf, d, inv_df);
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    leap[k] = Pf[k];
                    leap[4 + k] = inv_df[k];
                }
            }
            __syncwarp(gmask);
        }
        const uint8_t *dist = nullptr;
        if (ESL) dist = L.dist + octant_of(df) * nbricks;
        unsigned executed = 0, resampled = 0;
        CkState ck;
        if constexpr (CKPT) ck = {L.ckpt + (long)pix * L.ckpt_K, -1, -1, -1};
        group_march<ESL, G, MODE, CKPT, PACKED>(L, rp, dist, leap, df, leap + 4, inv_step, jlo,
                                                gmask, q, gbase, RC0, RC1, RC2, RT, executed,
                                                resampled, &ck);
        if constexpr (CKPT) {
            if (q == 0) L.ckpt_head[pix] = make_int2(ck.first < 0 ? 0 : ck.first, ck.jlast);
        }
        if (q == 0) {
            s_count[threadIdx.x / G][0] += executed;
            s_count[threadIdx.x / G][1] += resampled;
            if (L.accum)  // ordered pass: T itself (a queued ray met a sample of the piece)
                L.accum[pix] = make_float4(RC0, RC1, RC2, RT);
            else
                L.out[pix] = make_float4(RC0, RC1, RC2, 1.0f - RT);
        }
    }
    if (L.counters && q == 0) {
        const unsigned long long ex = s_count[threadIdx.x / G][0], rs = s_count[threadIdx.x / G][1];
        if (ex) atomicAdd(&L.counters[1], ex);
        if (rs) atomicAdd(&L.counters[2], rs);
    }
}

}  // namespace vrc
