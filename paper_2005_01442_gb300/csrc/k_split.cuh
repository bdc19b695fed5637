// The two phases of the split render as device functions, shared by the split render's own
// kernels (k_render_split.cu) and by the kernels that serving launches on the device
// (k_serve_dl.cu). The algorithm is described in k_render_split.cu.
#pragma once

#include "k_group.cuh"
#include "k_ray_tile.cuh"

namespace vrc {

constexpr int SPLIT_RAY_WARPS = 4;  // warps per CTA of the first phase (2: 0.3% slower)
constexpr int SPLIT_WARPS = 8;      // warps per CTA of the second phase

// First phase: the calling CTA's SPLIT_RAY_WARPS tiles of 8 x 4 pixels.
template <bool ESL, bool CKPT>
__device__ __forceinline__ void split_head_body(const RenderLaunch &L) {
    render_ray_tile<ESL, true, MODE_CUBIC_POST, CKPT>(L, blockIdx.x * SPLIT_RAY_WARPS +
                                                             (threadIdx.x >> 5));
}

// Second phase: the calling CTA's groups of SPLIT_G lanes drain the queue. The two groups of a
// warp take a ray each (mostly neighbours: their samples share lines in L1) and go through the
// steps of their marches -- leap, composite a block -- together, until both rays are done; a
// group that leapt while the other composited would run the warp at half width. Leaps go 16
// samples a lane ahead (0.75 million leap steps of a 1024^2 CT frame were 28% of its
// instructions when all lanes of a group took the same one).
// Bound: issue (78% of the slots), for dense views also the L1 data path. 1024^2 frame of a 512^2
// x 400 CT / with soft tissue: 274 / 1905 us; groups marching on their own 285 / 2034; each group
// taking its next ray as it gets free 315 / 2089 (the rays of a warp drift apart); together but
// with the same leap in every lane 284 / 2149.
template <bool ESL, int MODE, bool CKPT = false, int PACKED = -1>
__device__ __forceinline__ void split_tail_body(const RenderLaunch &L) {
    constexpr int G = SPLIT_G;
    constexpr unsigned FULL = 0xffffffffu, low = (1u << G) - 1u;
    static_assert(G < 32, "two groups a warp");
    // per group: the entry point and inverse direction that leaps use, kept out of registers, and
    // the samples counted
    __shared__ float s_leap[SPLIT_WARPS * 32 / G][8];
    __shared__ unsigned long long s_count[SPLIT_WARPS * 32 / G][2];
    const int lane = threadIdx.x & 31;
    const int q = lane & (G - 1);       // lane within the group
    const int gbase = lane & ~(G - 1);  // first lane of the group
    float *const leap = s_leap[threadIdx.x / G];
    unsigned long long *const count = s_count[threadIdx.x / G];
    if (q == 0) count[0] = count[1] = 0;
    const float step = L.grid.step, inv_step = 1.0f / step;
    const long nbricks = ESL ? (long)L.bricks.nb[0] * L.bricks.nb[1] * L.bricks.nb[2] : 0;
    ReplView rep = L.rep;
    if (PACKED >= 0) rep.packed = PACKED;
    // final counts (the first phase has finished): front records 0 .. nf-1, then back
    // records cap-1 down to cap-nb
    const unsigned nf = __ldcg(&L.split.head[0]), nb = __ldcg(&L.split.head[2]);
    const unsigned total = min(nf + nb, L.split.cap);

    bool has = false;    // the group has a ray in hand
    bool leaps = false;  // it leaps before its next block
    RayPos rp = {};
    int pix = 0, blk = 0, jlo = 0;
    const uint8_t *dist = nullptr;
    int cache_lin = -1;
    bool cache_occ = false;
    March m = {};
    CkState ck = {};
    while (true) {
        if (!__any_sync(FULL, has)) {
            unsigned c = 0;
            if (lane == 0) c = atomicAdd(&L.split.head[1], 2u);  // two rays
            c = __shfl_sync(FULL, c, 0);
            if (c >= total) break;
            c += lane / G;
            has = c < total;
            if (has) {
                const unsigned qi = c < nf ? c : L.split.cap - 1u - (c - nf);
                split_load(L.split.rec + (long)qi * SPLIT_REC, rp, jlo, pix, m.C0, m.C1, m.C2,
                           m.T);
                leaps = false;
                blk = jlo / G;
                cache_lin = -1;
                m.executed = m.resampled = 0;
                if constexpr (CKPT) ck = {L.ckpt + (long)pix * L.ckpt_K, -1, -1, -1};
                if (ESL) {
                    const float d[3] = {rp.d[0].hi, rp.d[1].hi, rp.d[2].hi};
                    dist = L.dist + octant_of(d) * nbricks;
                    if (q == 0) {
                        float Pf[3], df[3], inv_df[3];
                        ray_float(rp, Pf, df, inv_df);
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            leap[k] = Pf[k];
                            leap[4 + k] = inv_df[k];
                        }
                    }
                }
            }
            __syncwarp();
        }
        const float df[3] = {rp.d[0].hi, rp.d[1].hi, rp.d[2].hi};
        if (ESL) {
            // Leaps: lane q from sample jlo + G q, to where none before has an opacity other than
            // zero. The lanes that reach the next lane's sample join up from lane 0 on; the group
            // goes on from where the first other one got, until that one does not move.
            bool moving = has && leaps;
            while (__any_sync(FULL, moving)) {
                const int from = jlo + G * q;
                int to = from, lin = -1, r = 0;
                if (moving && from < rp.nseg)
                    to = leap_float(L.bricks, dist, leap, df, leap + 4, step, inv_step, rp.nseg,
                                    from, lin, r);
                const unsigned ends =
                    (__ballot_sync(FULL, to < min(from + G, rp.nseg)) >> gbase) & low;
                const int first = ends ? __ffs(ends) - 1 : G - 1;
                const int at = __shfl_sync(FULL, to, first, G);
                if (moving) {
                    moving = ends == 0 ? at < rp.nseg : at > jlo + G * first;
                    jlo = at;
                }
            }
            if (leaps) blk = jlo / G;
        }
        // (a ray whose leaps reached its end has no block)
        bool on = has && blk * G < rp.nseg;
        unsigned occ_bits;
        const bool stop =
            march_block<ESL, G, MODE, CKPT>(L, rep, rp, dist, df, on, blk, jlo, FULL, q, gbase,
                                            cache_lin, cache_occ, m, occ_bits, &ck);
        ++blk;
        jlo = blk * G;
        leaps = !((occ_bits >> (G - 1)) & 1u);
        if (has && (stop || jlo >= rp.nseg)) {
            has = false;
            if (q == 0) {
                count[0] += m.executed;
                count[1] += m.resampled;
                if constexpr (CKPT)
                    L.ckpt_head[pix] = make_int2(ck.first < 0 ? 0 : ck.first, ck.jlast);
                if (L.accum)  // ordered pass: T itself (a queued ray met a sample of the piece)
                    L.accum[pix] = make_float4(m.C0, m.C1, m.C2, m.T);
                else
                    L.out[pix] = make_float4(m.C0, m.C1, m.C2, 1.0f - m.T);
            }
        }
    }
    if (L.counters && q == 0) {
        if (count[0]) atomicAdd(&L.counters[1], count[0]);
        if (count[1]) atomicAdd(&L.counters[2], count[1]);
    }
}

}  // namespace vrc
