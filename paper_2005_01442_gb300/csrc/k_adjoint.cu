// Adjoint of the render: gradients of a loss on the image with respect to the 256-entry RGBA
// transfer function and the voxel values. The paper renders only; the reverse mode is built on
// its forward model (cubic B-spline resampling, post-classification, opacity correction,
// front-to-back compositing, early termination).
//
// It reads the checkpoints of a forward render (RenderLaunch::ckpt): the ray's last composited
// sample and, for each segment of `seg` samples up to it, the transmittance at the segment's
// start (-1 for segments without composited samples). One warp takes one ray and walks its
// segments back to front, a block of 32 consecutive samples at a time, a lane per sample:
//   1. forward over the segment's blocks: every lane resamples and classifies its sample, and a
//      prefix product from the checkpoint gives its transmittance T_j (never dividing by
//      1 - alpha);
//   2. back over the blocks: a suffix scan of the "over" operator gives each lane what lies
//      behind its sample -- the rest of the block, then the carry of the blocks before -- as
//      S = normalised colour behind, U = transmittance behind, and
//        dL/drgb_j   = T_j alpha_j g_rgb
//        dL/dalpha_j = T_j [ g_rgb . (rgb_j - S) + g_A U ]
//      chained through alpha = 1 - (1-a)^delta, the table interpolation (into the two entries)
//      and the 64 B-spline taps (into the voxels);
//   3. the lanes' contributions are summed in shared memory, sample by sample, the warp's lanes
//      being the taps (two each) and the table components: no two lanes meet at an address, so
//      plain adds do. Voxels collect in a box of up to ADJ_BOX floats around 16 consecutive
//      samples, which then goes to the volume as float4 atomics.
// Transfer-function gradients are kept per warp and added up per CTA (global float atomics at
// the end: the summation order, and so the last bits, vary from run to run). Samples in empty
// bricks or clear cells (opacity exactly zero, whose derivative is taken as zero at the clamp,
// so that every contribution of such a sample is exactly zero) are skipped exactly as in the
// forward.
//
// What bounds it: adding every tap to the volume on its own was bound by the vector atomics of
// L2 (16 rows a sample of one float4, two float2 or float + float2 + float, 2.25 atomics a row
// on average, at 192 G/s measured: 36 a sample), and eight shared-memory atomics a sample
// contended for the few table entries in use. Consecutive samples half a voxel apart share most
// of their taps, so a box of 16 gives some 4.9 atomic sectors a sample instead. 256^3 float32 at
// 512^2, soft tissue visible (17 M samples): 1.80 ms a view against 4.0 ms. What bounds it now is
// the chain of a warp's adds and the registers (16 warps an SM): 54% of the issue slots, 61% of
// the L1 and shared-memory data path. Eight warps a CTA share the long rays of a tile out better
// than four and halve the sums that go to the table: 256^3 at 512^2, bone and vessels visible, 298
// us against 398; with soft tissue 2.06 ms against 2.12.
#include "vrc_internal.h"

namespace vrc {

// Adds (v0, v1, v2, v3) to the voxel gradients of taps x0 .. x0+3 of a row, clamped to
// [0, nx-1], with the fewest aligned vector atomics (one float4, two float2 or float + float2
// + float away from the edges).
__device__ __forceinline__ void add_taps_x(float *row, int x0, int nx, float v0, float v1,
                                           float v2, float v3) {
    if (x0 >= 0 && x0 + 3 < nx) {
        float *a = row + x0;
        switch ((unsigned)((uintptr_t)a & 15u)) {
        case 0:
            atomicAdd((float4 *)a, make_float4(v0, v1, v2, v3));
            return;
        case 8:
            atomicAdd((float2 *)a, make_float2(v0, v1));
            atomicAdd((float2 *)(a + 2), make_float2(v2, v3));
            return;
        default:  // 4 or 12: a + 1 is 8-byte aligned
            atomicAdd(a, v0);
            atomicAdd((float2 *)(a + 1), make_float2(v1, v2));
            atomicAdd(a + 3, v3);
            return;
        }
    }
    atomicAdd(row + min(max(x0, 0), nx - 1), v0);
    atomicAdd(row + min(max(x0 + 1, 0), nx - 1), v1);
    atomicAdd(row + min(max(x0 + 2, 0), nx - 1), v2);
    atomicAdd(row + min(max(x0 + 3, 0), nx - 1), v3);
}

constexpr int ADJ_WARPS = 8;
constexpr int ADJ_BOX = 1152;    // floats of a warp's box of voxel gradients
constexpr int ADJ_CHUNK = 16;    // samples summed into one box
constexpr int ADJ_REC = 36;      // words of a sample's record (conflict-free 16-byte stores)
constexpr int ADJ_TILE = 64;     // pixels of a CTA at most

// A ray of the CTA's tile that composited something.
struct AdjRay {
    RayPos rp;
    float4 g;        // dL/d(pixel)
    int pix, k0, jlast;
};

struct alignas(16) AdjWarp {  // a warp's shared memory
    float box[ADJ_BOX];
    float tf[1024];
    // per sample of the chunk: 16 products wx[a] wy[b]; (ds wz[0], ds wz[2], box offset of the
    // first tap, table offset); the same with wz[1], wz[3]; the 8 table components
    float rec[(ADJ_CHUNK + 1) * ADJ_REC];
};

struct AdjShared {  // a CTA's (dynamic: above the 48 KB of static shared memory)
    AdjWarp warp[ADJ_WARPS];
    AdjRay ray[ADJ_TILE];
};

// NB: blocks of 32 samples that a segment spans at most.
template <bool ESL, bool VOLGRAD, int NB>
__global__ void __launch_bounds__(32 * ADJ_WARPS, 2) adjoint_kernel(AdjointLaunch A, int tw_shift,
                                                                    int th_shift) {
    extern __shared__ AdjShared s_adj[];
    AdjWarp *const s_warp = s_adj->warp;
    AdjRay *const s_ray = s_adj->ray;
    __shared__ int s_count, s_head;
    const RenderLaunch &L = A.L;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float step = L.grid.step;
    const int seg = A.seg;
    if (threadIdx.x == 0) s_count = s_head = 0;
    __syncthreads();

    // the tile's rays that have work, by the forward's record: first checkpointed segment, last
    // composited sample (read first: most rays of a CT view composite nothing and need no set-up)
    if (threadIdx.x < (1u << (tw_shift + th_shift))) {
        const int tiles_x = (L.cam.width + (1 << tw_shift) - 1) >> tw_shift;
        const int px = ((blockIdx.x % tiles_x) << tw_shift) + (threadIdx.x & ((1 << tw_shift) - 1));
        const int py = ((blockIdx.x / tiles_x) << th_shift) + (threadIdx.x >> tw_shift);
        if (px < L.cam.width && py < L.cam.height) {
            const int pix = py * L.cam.width + px;
            const float4 g = A.grad_out[pix];
            const int2 h = L.ckpt_head[pix];
            if (h.y >= 0 && (g.x != 0.0f || g.y != 0.0f || g.z != 0.0f || g.w != 0.0f)) {
                RaySetup ray;
                ray_setup(L.cam, L.grid, px, py, ray);
                if (ray.nseg > 0) {
                    AdjRay r;
                    ray_pos_init(ray, step, r.rp);
                    r.g = g;
                    r.pix = pix;
                    r.k0 = max(h.x, 0);
                    r.jlast = min(h.y, r.rp.nseg - 1);
                    s_ray[atomicAdd(&s_count, 1)] = r;
                }
            }
        }
    }
    __syncthreads();
    const int count = s_count;
    if (count == 0) return;

    AdjWarp &W = s_warp[warp];
    for (int i = lane; i < ADJ_BOX; i += 32) W.box[i] = 0.0f;
    for (int i = lane; i < 1024; i += 32) W.tf[i] = 0.0f;
    __syncwarp();
    const int nx = L.grid.n[0], ny = L.grid.n[1], nz = L.grid.n[2];
    // rows of the volume's gradient on 16-byte boundaries
    const bool aligned = VOLGRAD && (nx & 3) == 0 && ((uintptr_t)A.grad_vol & 15) == 0;
    const long nbricks = ESL ? (long)L.bricks.nb[0] * L.bricks.nb[1] * L.bricks.nb[2] : 0;

    while (true) {
        int qi = 0;
        if (lane == 0) qi = atomicAdd(&s_head, 1);
        qi = __shfl_sync(0xffffffffu, qi, 0);
        if (qi >= count) break;
        const RayPos rp = s_ray[qi].rp;
        const float4 g = s_ray[qi].g;
        const int k0 = s_ray[qi].k0, jlast = s_ray[qi].jlast;
        const float df[3] = {rp.d[0].hi, rp.d[1].hi, rp.d[2].hi};
        const uint8_t *dist = ESL ? L.dist + octant_of(df) * nbricks : nullptr;
        const float *ck_row = L.ckpt + (long)s_ray[qi].pix * L.ckpt_K;
        // what lies behind the current block: normalised colour and transmittance
        float cS0 = 0.0f, cS1 = 0.0f, cS2 = 0.0f, cU = 1.0f;
        const int klast = min(jlast / seg, L.ckpt_K - 1);
        float ck = -1.0f;  // 32 segments' checkpoints at a time, one a lane
        for (int k = klast; k >= k0; --k) {
            const int back = (klast - k) & 31;
            if (back == 0) ck = k - lane >= k0 ? ck_row[k - lane] : -1.0f;
            const float Tk = __shfl_sync(0xffffffffu, ck, back);
            if (!(Tk >= 0.0f)) continue;  // no composited sample in this segment
            const int j1 = min(k * seg + seg, jlast + 1);
            int chunk = ADJ_CHUNK;
            // forward: values, opacities and transmittances of the segment's samples
            int ip[NB][3];
            float f[NB][3], sv[NB], Tj[NB];
            unsigned live_bits[NB];
            float T = Tk;
            uint32_t word[NB];
            uint8_t empty[NB];
#pragma unroll
            for (int b = 0; b < NB; ++b) {  // the blocks' look-ups in flight together
                float delta;
                const int j = min(k * seg + 32 * b + lane, rp.nseg - 1);
                place(rp, step, L.grid.n, j, ip[b], f[b], delta);
                if (ESL) {
                    empty[b] = dist[brick_of(L.bricks, ip[b])];
                    word[b] = L.cells ? cell_word(L.cells, L.grid.n, ip[b]) : 0xffffffffu;
                }
            }
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const int j = k * seg + 32 * b + lane;
                bool live = j < j1;
                if (ESL) live = live && empty[b] == 0 && cell_bit(word[b], ip[b]);
                const float delta = j < rp.nseg - 1 ? step : rp.dlast;
                float eT = 1.0f;
                sv[b] = 0.0f;
                if (live) {
                    sv[b] = tricubic_rep(L.rep, ip[b], f[b]);
                    eT = 1.0f - segment_alpha(classify(L.tf, sv[b]).c.w, delta);
                }
                live_bits[b] = __ballot_sync(0xffffffffu, live);
                if (live_bits[b] == 0u) continue;
                float incl = eT;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const float p = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl = p * incl;
                }
                const float excl = __shfl_up_sync(0xffffffffu, incl, 1);
                Tj[b] = lane == 0 ? T : T * excl;
                T = T * __shfl_sync(0xffffffffu, incl, 31);
            }
            // back to front over the blocks
#pragma unroll
            for (int b = NB - 1; b >= 0; --b) {
                if (live_bits[b] == 0u) continue;
                const bool live = (live_bits[b] >> lane) & 1u;
                const int j = k * seg + 32 * b + lane;
                const float delta = j < rp.nseg - 1 ? step : rp.dlast;
                const Classified c = classify(L.tf, sv[b]);
                const float alpha = live ? segment_alpha(c.c.w, delta) : 0.0f;
                // behind the sample: suffix scan of v_j = P_j o ... o P_31 of the "over" operator
                // (C_a, T_a) o (C_b, T_b) = (C_a + T_a C_b, T_a T_b)
                float v0 = alpha * c.c.x, v1 = alpha * c.c.y, v2 = alpha * c.c.z, vT = 1.0f - alpha;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const float p0 = __shfl_down_sync(0xffffffffu, v0, o);
                    const float p1 = __shfl_down_sync(0xffffffffu, v1, o);
                    const float p2 = __shfl_down_sync(0xffffffffu, v2, o);
                    const float pT = __shfl_down_sync(0xffffffffu, vT, o);
                    if (lane + o < 32) {
                        v0 = fmaf(vT, p0, v0);
                        v1 = fmaf(vT, p1, v1);
                        v2 = fmaf(vT, p2, v2);
                        vT = vT * pT;
                    }
                }
                float S0 = __shfl_down_sync(0xffffffffu, v0, 1);
                float S1 = __shfl_down_sync(0xffffffffu, v1, 1);
                float S2 = __shfl_down_sync(0xffffffffu, v2, 1);
                float U = __shfl_down_sync(0xffffffffu, vT, 1);
                if (lane == 31) {
                    S0 = S1 = S2 = 0.0f;
                    U = 1.0f;
                }
                S0 = fmaf(U, cS0, S0);
                S1 = fmaf(U, cS1, S1);
                S2 = fmaf(U, cS2, S2);
                U = U * cU;
                {  // the next block lies in front of this one: carry = v_0 o carry
                    const float aT = __shfl_sync(0xffffffffu, vT, 0);
                    cS0 = fmaf(aT, cS0, __shfl_sync(0xffffffffu, v0, 0));
                    cS1 = fmaf(aT, cS1, __shfl_sync(0xffffffffu, v1, 0));
                    cS2 = fmaf(aT, cS2, __shfl_sync(0xffffffffu, v2, 0));
                    cU = aT * cU;
                }
                // compositing
                const float ta = Tj[b] * alpha;
                const float d_r = ta * g.x, d_g = ta * g.y, d_b = ta * g.z;
                const float dalpha = Tj[b] * (g.x * (c.c.x - S0) + g.y * (c.c.y - S1) +
                                              g.z * (c.c.z - S2) + g.w * U);
                // opacity correction (zero derivative at the clamp ends; from above at 0 when
                // asked)
                const float a = fminf(fmaxf(c.c.w, 0.0f), ALPHA_MAX);
                const bool up = c.c.w > 0.0f || (A.open_alpha && c.c.w == 0.0f);
                const float da = (up && c.c.w <= ALPHA_MAX)
                                     ? delta * ex2((delta - 1.0f) * lg2(1.0f - a))
                                     : 0.0f;
                const float d_a = dalpha * da;
                float ds = 0.0f;
                if (VOLGRAD && live && c.u_raw > 0.0f && c.u_raw < 255.0f)
                    ds = (d_r * c.dc.x + d_g * c.dc.y + d_b * c.dc.z + d_a * c.dc.w) * L.tf.du;
                const unsigned vox = VOLGRAD ? __ballot_sync(0xffffffffu, ds != 0.0f) : 0u;

                for (int l0 = 0; l0 < 32;) {
                    const unsigned span = (chunk == 32 ? 0xffffffffu : (1u << chunk) - 1u) << l0;
                    unsigned todo = live_bits[b] & span;
                    if (todo == 0u) {
                        l0 += chunk;
                        continue;
                    }
                    const bool mine = (todo >> lane) & 1u;
                    // box of the taps, from x0 (a multiple of 4), y0, z0
                    int x0 = 0, y0 = 0, z0 = 0, px = 0, ey = 0, ez = 0, plane = 0;
                    if (VOLGRAD && (vox & span)) {
                        const bool v = mine && ds != 0.0f;
                        const int big = 1 << 20;
                        x0 = (__reduce_min_sync(0xffffffffu, v ? ip[b][0] : big) - 1) & ~3;
                        y0 = __reduce_min_sync(0xffffffffu, v ? ip[b][1] : big) - 1;
                        z0 = __reduce_min_sync(0xffffffffu, v ? ip[b][2] : big) - 1;
                        px = (__reduce_max_sync(0xffffffffu, v ? ip[b][0] : -big) + 6 - x0) & ~3;
                        ey = __reduce_max_sync(0xffffffffu, v ? ip[b][1] : -big) + 3 - y0;
                        ez = __reduce_max_sync(0xffffffffu, v ? ip[b][2] : -big) + 3 - z0;
                        // rows and planes 4-float groups apart from each other in the banks
                        if (px == 16) px = 20;
                        plane = px * ey;
                        plane += ((px == 8 ? 4 : 16) - plane) & 31;
                        if (plane * ez > ADJ_BOX) {  // long steps: fewer samples a box (one
                            chunk >>= 1;             // sample takes 8 x 4 x 4 at most)
                            continue;
                        }
                    }
                    const bool boxed = plane != 0;
                    if (mine) {  // the chunk's records, without gaps
                        float *r = W.rec + __popc(todo & ((1u << lane) - 1u)) * ADJ_REC;
                        if (VOLGRAD && boxed) {
                            float wx[4], wy[4], wz[4];
                            bspline_w(f[b][0], wx);
                            bspline_w(f[b][1], wy);
                            bspline_w(f[b][2], wz);
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                *(float4 *)(r + 4 * i) = make_float4(wx[0] * wy[i], wx[1] * wy[i],
                                                                     wx[2] * wy[i], wx[3] * wy[i]);
                            // a sample without a voxel gradient adds zeros at the box's start
                            const float o = __int_as_float(
                                ds == 0.0f ? 0 : (ip[b][2] - 1 - z0) * plane +
                                                     (ip[b][1] - 1 - y0) * px + (ip[b][0] - 1 - x0));
                            *(float4 *)(r + 16) = make_float4(wz[0] * ds, wz[2] * ds, o, 0.0f);
                            *(float4 *)(r + 20) = make_float4(wz[1] * ds, wz[3] * ds, o, 0.0f);
                        }
                        r[19] = __int_as_float(4 * c.i0);
                        const float w1 = c.fu, w0 = 1.0f - c.fu;
                        *(float4 *)(r + 24) = make_float4(w0 * d_r, w0 * d_g, w0 * d_b, w0 * d_a);
                        *(float4 *)(r + 28) = make_float4(w1 * d_r, w1 * d_g, w1 * d_b, w1 * d_a);
                    }
                    __syncwarp();
                    // sample by sample: lane (a, b, h) adds the taps (a, b, h) and (a, b, h + 2),
                    // lanes 0 .. 7 the table components; the next record is read ahead
                    const int n = __popc(todo);
                    const float *r = W.rec;
                    if (VOLGRAD && boxed) {
                        float *t0 = W.box + (lane & 3) + ((lane >> 2) & 3) * px +
                                    (lane >> 4) * plane;
                        const float *rw = r + (lane & 15), *rz = r + 16 + 4 * (lane >> 4);
                        const float *re = r + 24 + (lane & 7);
                        float w = *rw, e = *re;
                        float4 z = *(const float4 *)rz;
#pragma unroll 2
                        for (int i = 1; i <= n; ++i) {
                            // (the record after the last is read too, and not used)
                            const float w2 = rw[i * ADJ_REC], e2 = re[i * ADJ_REC];
                            const float4 z2 = *(const float4 *)(rz + i * ADJ_REC);
                            float *t = t0 + __float_as_int(z.z);
                            const float u0 = t[0], u1 = t[2 * plane];
                            t[0] = fmaf(w, z.x, u0);
                            t[2 * plane] = fmaf(w, z.y, u1);
                            if (lane < 8) W.tf[__float_as_int(z.w) + lane] += e;
                            __syncwarp();
                            w = w2;
                            e = e2;
                            z = z2;
                        }
                    } else {
                        for (int i = 0; i < n; ++i) {
                            if (lane < 8)
                                W.tf[__float_as_int(r[i * ADJ_REC + 19]) + lane] +=
                                    r[i * ADJ_REC + 24 + lane];
                            __syncwarp();
                        }
                    }
                    if (VOLGRAD && boxed) {
                        // the box to the volume, 4 voxels along x a lane and a few rows a step,
                        // and back to zeros
                        const int pq = px >> 2, per = 32 / pq, q = lane % pq;
                        int yy = lane / pq, zz = 0;
                        if (yy >= per) yy = 1 << 20;
                        for (int row = yy; row < ey * ez; row += per, yy += per) {
                            while (yy >= ey) {
                                yy -= ey;
                                ++zz;
                            }
                            float4 *cell = (float4 *)(W.box + zz * plane + yy * px + 4 * q);
                            const float4 v = *cell;
                            if (v.x == 0.0f && v.y == 0.0f && v.z == 0.0f && v.w == 0.0f) continue;
                            *cell = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                            const int y = min(max(y0 + yy, 0), ny - 1);
                            const int z = min(max(z0 + zz, 0), nz - 1);
                            const int x = x0 + 4 * q;
                            float *to = A.grad_vol + ((long)z * ny + y) * nx;
                            if (aligned && x >= 0 && x + 3 < nx) atomicAdd((float4 *)(to + x), v);
                            else add_taps_x(to, x, nx, v.x, v.y, v.z, v.w);
                        }
                        __syncwarp();
                    }
                    l0 += chunk;
                }
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 1024; i += blockDim.x) {
        float v = 0.0f;
#pragma unroll
        for (int w = 0; w < ADJ_WARPS; ++w) v += s_warp[w].tf[i];
        if (v != 0.0f) atomicAdd(A.grad_tf + i, v);
    }
}

template <int NB>
static cudaError_t launch_adjoint_n(const AdjointLaunch &A, cudaStream_t st) {
    // Every CTA adds its table sums to the same 1024 floats, whose error grows with the number of
    // additions (4 x 2 pixels a CTA: 1.5 times the error of 4 x 4 for a 98 x 460 image), so larger
    // images take larger tiles: 64 pixels from 1.5 Mi on (error of the table gradient of 256^3 at
    // 2048^2 / 4096^2, random loss: 1.2e-6 / 2.8e-6, with 32 pixels 2.0e-6 / 5.4e-6), 32 from 64 Ki
    // on, 16 below. Small images want small tiles anyway, large ones large: 256^3 at 128^2 79 us
    // with 16 pixels, 106 with 32; at 256^2 126, 144 and 208 with 64; at 1024^2 893, 806, 888; at
    // 1448^2 1740, 1491, 1504 (table alone 1272, 1033, 932); at 2048^2 3650, 3031, 2750.
    const long pixels = (long)A.L.cam.width * A.L.cam.height;
    const int tw = pixels < 1536 * 1024 ? 2 : 3, th = pixels < 64 * 1024 ? 2 : 3;
    const unsigned grid = (unsigned)((((long)A.L.cam.width + (1 << tw) - 1) >> tw) *
                                     ((A.L.cam.height + (1 << th) - 1) >> th));
    const bool esl = A.L.dist != nullptr, vg = A.grad_vol != nullptr;
    auto kernel = esl ? (vg ? adjoint_kernel<true, true, NB> : adjoint_kernel<true, false, NB>)
                      : (vg ? adjoint_kernel<false, true, NB> : adjoint_kernel<false, false, NB>);
    const cudaError_t e = cudaFuncSetAttribute(
        kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(AdjShared));
    if (e != cudaSuccess) return e;
    kernel<<<grid, 32 * ADJ_WARPS, sizeof(AdjShared), st>>>(A, tw, th);
    return cudaGetLastError();
}

cudaError_t launch_adjoint(const AdjointLaunch &A, cudaStream_t st) {
    static_assert(ADJ_MAX_SEG <= 128, "a segment spans at most 4 blocks of 32 samples");
    if (A.seg <= 32) return launch_adjoint_n<1>(A, st);
    if (A.seg <= 64) return launch_adjoint_n<2>(A, st);
    return launch_adjoint_n<4>(A, st);
}

}  // namespace vrc
