// Marching one ray with a group of G lanes (G = 4, 8, 16 or 32), shared by the lane-group kernels
// (k_render_warp.cu), serving (k_serve.cu) and the second phase of the split render (k_split.cuh).
//
// The ray is walked in blocks of G consecutive sample indices, lane q of the group taking
// sample G k + q. Every lane places its sample exactly from the double-float ray record,
// resamples the uniform cubic B-spline from the render layout (ReplView), classifies it
// through the transfer function and corrects its opacity to the segment length (paper, Sec.
// "Methodology": cubic interpolation, post-classification). The block is composited front to
// back by a group-wide inclusive scan of the "over" operator
// (C_a, T_a) o (C_b, T_b) = (C_a + T_a C_b, T_a T_b) on (alpha rgb, 1 - alpha) and prepended by
// what the ray has accumulated so far; early ray termination picks the first lane whose
// accumulated opacity exceeds the threshold (ballot). Samples known to have zero opacity (in
// an empty brick or a transparent cell) enter the scan as the identity (0, 1), which is
// exactly what computing them gives, so the result is bit-identical with and without
// skipping. Between blocks the group leaps over empty space (Sec. "Analysis", Pros (b)).
#pragma once

#include "vrc_internal.h"

namespace vrc {

// From sample j, a sample (or nseg) before which none has an opacity other than zero: the first
// that leaping cannot pass. Deterministic in its inputs, so every lane of a group gets the same
// answer. (The sample may still lie in an empty brick, next to a face: the block that starts
// there finds out from the exact position.)
__device__ __forceinline__ int advance_to_occupied(const RayPos &rp, const RenderLaunch &L,
                                                   const uint8_t *__restrict__ dist,
                                                   const float Pf[3], const float df[3],
                                                   const float inv_df[3], float inv_step, int j) {
    int cache_lin = -1, cache_r = 0;
    while (j < rp.nseg) {
        const int jn = leap_float(L.bricks, dist, Pf, df, inv_df, L.grid.step, inv_step, rp.nseg,
                                  j, cache_lin, cache_r);
        if (jn == j) break;
        j = jn;
    }
    return min(j, rp.nseg);
}

// What a ray's march accumulates.
struct March {
    float C0, C1, C2, T;           // colour and transmittance, equal in every lane of the group
    unsigned executed, resampled;  // samples in occupied bricks, and those resampled
};

// Composites the block of G samples blk * G .. + G - 1 of a ray onto m, lane q of the group (first
// lane gbase) taking one sample; those before jlo and after the ray's end are left out, and all
// of them where `on` is false. `mask`: the lanes that run this together, the group's or the
// warp's. occ_bits: the block's samples in occupied bricks. Returns true when the ray ends by
// early termination. cache_lin / cache_occ memoise the brick of this lane's last sample.
//
// CKPT (default variant, L.ckpt_seg a multiple of G, so a block lies in one segment): ck
// records the ray's reverse-mode checkpoints as render_ray_tile does -- the transmittance
// before the first block with a composited sample in each segment (-1 for segments without
// one), every segment from the first to the last such one (written by the group's lanes in
// turn), and the last composited sample.
template <bool ESL, int G, int MODE, bool CKPT>
__device__ __forceinline__ bool march_block(const RenderLaunch &L, const ReplView &rep,
                                            const RayPos &rp, const uint8_t *__restrict__ dist,
                                            const float df[3], bool on, int blk, int jlo,
                                            unsigned mask, int q, int gbase, int &cache_lin,
                                            bool &cache_occ, March &m, unsigned &occ_bits,
                                            CkState *ck) {
    constexpr unsigned low = G == 32 ? 0xffffffffu : ((1u << G) - 1u);
    const float step = L.grid.step, thr = L.grid.ert;
    const int j = blk * G + q;
    float e0 = 0.0f, e1 = 0.0f, e2 = 0.0f, eT = 1.0f;  // identity of "over"
    bool live = on && j >= jlo && j < rp.nseg;
    bool in_occ = live;  // sample in range and in an occupied brick
    if (live) {
        float delta;
        int ip[3];
        float f[3];
        place(rp, step, L.grid.n, j, ip, f, delta);
        if (ESL) {
            // both looked up at once: the word is worth a load even if the brick is empty
            const uint32_t word = L.cells ? cell_word(L.cells, L.grid.n, ip) : 0xffffffffu;
            const int lin = brick_of(L.bricks, ip);
            if (lin != cache_lin) {  // lane q's samples of successive blocks share bricks
                cache_lin = lin;
                cache_occ = dist[lin] == 0;
            }
            in_occ = cache_occ;
            live = in_occ && cell_bit(word, ip);
        }
        if (live) {
            const float4 rgba = sample_rgba<MODE>(rep, L.tf, ip, f, df, &L.phong);
            const float alpha = segment_alpha(rgba.w, delta);
            e0 = alpha * rgba.x;
            e1 = alpha * rgba.y;
            e2 = alpha * rgba.z;
            eT = 1.0f - alpha;
        }
    }
    occ_bits = (__ballot_sync(mask, in_occ) >> gbase) & low;
    const unsigned any = __ballot_sync(mask, live);
    const unsigned live_bits = (any >> gbase) & low;
    int last = G - 1;
    unsigned stop_bits = 0;
    if (any) {  // (a group of a warp without a live sample scans identities: m unchanged)
        if constexpr (CKPT) {
            const int k = (blk * G) / L.ckpt_seg;
            if (live_bits && k != ck->last) {
                for (int kk = (ck->first < 0 ? k : ck->last + 1) + q; kk <= k; kk += G)
                    ck->row[kk] = kk == k ? m.T : -1.0f;  // -1: no composited sample
                if (ck->first < 0) ck->first = k;
                ck->last = k;
            }
        }
        // inclusive scan of "over" across the group's block
#pragma unroll
        for (int o = 1; o < G; o <<= 1) {
            const float p0 = __shfl_up_sync(mask, e0, o, G);
            const float p1 = __shfl_up_sync(mask, e1, o, G);
            const float p2 = __shfl_up_sync(mask, e2, o, G);
            const float pT = __shfl_up_sync(mask, eT, o, G);
            if (q >= o) {
                e0 = fmaf(pT, e0, p0);
                e1 = fmaf(pT, e1, p1);
                e2 = fmaf(pT, e2, p2);
                eT = pT * eT;
            }
        }
        // prepend what the ray has accumulated before this block
        const float t0 = fmaf(m.T, e0, m.C0), t1 = fmaf(m.T, e1, m.C1), t2 = fmaf(m.T, e2, m.C2);
        const float tT = m.T * eT;
        stop_bits = (__ballot_sync(mask, live && (1.0f - tT > thr)) >> gbase) & low;
        if (stop_bits) last = __ffs(stop_bits) - 1;
        m.C0 = __shfl_sync(mask, t0, last, G);
        m.C1 = __shfl_sync(mask, t1, last, G);
        m.C2 = __shfl_sync(mask, t2, last, G);
        m.T = __shfl_sync(mask, tT, last, G);
        if constexpr (CKPT) {
            if (live_bits) ck->jlast = blk * G + (stop_bits ? last : 31 - __clz(live_bits));
        }
    }
    if (L.counters) {
        m.executed += __popc(occ_bits & (0xffffffffu >> (31 - last)));
        m.resampled += __popc(live_bits & (0xffffffffu >> (31 - last)));
    }
    return stop_bits != 0;
}

// A group of G lanes (mask gmask) marches the ray from sample jlo on by itself, whatever the rest
// of its warp does.
template <bool ESL, int G, int MODE = MODE_CUBIC_POST>
__device__ __forceinline__ void group_march(const RenderLaunch &L, const RayPos &rp,
                                            const uint8_t *__restrict__ dist, const float Pf[3],
                                            const float df[3], const float inv_df[3],
                                            float inv_step, int jlo, unsigned gmask, int q,
                                            int gbase, March &m) {
    int blk = jlo / G, cache_lin = -1;
    bool cache_occ = false;
    while (blk * G < rp.nseg) {
        unsigned occ_bits;
        if (march_block<ESL, G, MODE, false>(L, L.rep, rp, dist, df, true, blk, jlo, gmask, q,
                                             gbase, cache_lin, cache_occ, m, occ_bits, nullptr))
            break;
        ++blk;
        jlo = blk * G;
        // leap from the next block's first sample (uniform across the group) unless the block
        // ended inside an occupied brick
        if (ESL && !((occ_bits >> (G - 1)) & 1u) && jlo < rp.nseg) {
            jlo = advance_to_occupied(rp, L, dist, Pf, df, inv_df, inv_step, jlo);
            blk = jlo / G;
        }
    }
}

}  // namespace vrc
