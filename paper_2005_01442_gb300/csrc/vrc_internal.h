// Host-side declarations shared between the C-ABI layer (vrc_api.cu) and the kernel
// translation units. Not part of the public interface.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "vrc.h"
#include "vrc_device.cuh"

namespace vrc {

constexpr int PAD = 2;  // edge-replicated voxels on each side of a resident volume

enum Dtype { DT_U16 = 0, DT_I16 = 1, DT_F32 = 2 };

inline size_t dtype_size(int dt) { return dt == DT_F32 ? 4 : 2; }

// A resident volume in the padded layout: element (x, y, z) of the original volume lives at
// ((z + PAD) * pny + (y + PAD)) * pnx + (x + PAD); pnx is rounded up to a multiple of 8
// elements so every row starts on a 16-byte boundary. The pad replicates the edge voxels
// (clamp-to-edge), so taps at -2 .. n+1 need no clamping.
struct VolView {
    const void *base;  // padded buffer
    int dtype;
    int n[3];
    int pnx, pny, pnz;
};

// The render layout of a resident volume: each voxel in several entries of 16 bytes, so that a
// sample reads its 64 taps with few aligned wide loads. The entry (x', y', z') starts at voxel
// (x'-2, y'-2, z'-2), x' in [0, nx+2] and so on, indices clamped to the volume (clamp-to-edge)
// when the layout is written. The voxels lie in pairs along z with x fastest, as the packed
// float32 arithmetic of the resampling takes them.
//
// 16-bit: the 2^3 voxels, a pair one word (low half the lower z), each voxel plus `bias` as an
//   unsigned 16-bit value. A sample at base i reads the 8 entries (i0+1 + {0, 2}, i1+1 + {0, 2},
//   i2+1 + {0, 2}).
// float32: the 2^2 voxels along x and z (y' in [0, ny+3]); a sample reads 16 entries, i1+1 + {0,
//   1, 2, 3} along y.
//
// Entries lie in blocks of 2^3 (slot 4 (z' & 1) + 2 (y' & 1) + (x' & 1)), blocks in rows along x.
// The render is bound by the L1 data path, which serves a line at a time: the samples of a warp
// lie along rays, and a ray crosses fewer blocks than rows of entries.
// Second phase of a dense 1024^2 frame of a 512^2 x 400 int16 CT, 105 M samples: 2.50 ms and 637
// M wavefronts of the L1 data path in rows of entries, 2.36 ms and 563 M in blocks, 2.11 ms and
// 481 M (72% of its rate; 75% of the issue slots) with table lookups of 32 bytes and a kernel per
// voxel type as well.
// float32 entries of 2^3 voxels (8 loads of 32 bytes a sample) would take twice the memory and a
// third longer to write (256^3: 133 against 99 us). A dense 1280 x 1024 frame of 253 x 187 x 250
// takes 1.32 ms so and 1.31 ms with them, without bricks 2.75 and 2.40 ms; rays a lane each,
// whose warps spread over more lines, 2.37 and 2.79 ms (pre-integrated), and a training pass of
// 256^3 at 512^2 6.29 and 6.45 ms.
struct ReplView {
    const void *base;
    size_t row, slice;  // bytes from a block to the next along y and z
    int rnx, rny;       // blocks per row, rows of blocks per slice
    int packed;         // 16-bit voxels
    float magic;        // 16-bit: 2^23 + bias
};

// Brick table of size B (min/max arrays of the voxel dtype, ceil(n/B) per axis).
struct BrickView {
    int B, shift;
    int nb[3];
    const void *mn, *mx;
    float margin;  // leap and quick-skip margin in voxels (leap_margin)
};

// Device transfer function: table entry k at tab[2k], the forward difference to entry k + 1 (0 for
// the last) at tab[2k + 1], 256 of each; a lookup is one 32-byte load.
struct TfView {
    const float4 *tab;
    float lo, hi, du;     // du = 255 / (hi - lo) in float32
};

// ------------------------------------------------------------------------------------------
// Leaping (Sec. "Analysis", Pros (b): auxiliary structures to skip empty space). Decisions use
// float positions pa = fma(m, d, P): the entry point P (|P| <= C, the largest extent of the
// volume), the direction d and m = (j + 1/2) ds (<= the box diagonal, 1.8 C) each rounded once,
// and the fma once more, so |pa - p| <= 2^-24 (|P| + 2 m + |pa|) < 3.3e-7 C. A sample is leapt
// over only when it sits at least the margin inside a forward box of empty bricks, where its
// opacity is exactly zero; the margin is three times that bound (4.1e-3 voxel at C = 4096),
// and at least 2.5e-4 voxel.
inline float leap_margin(const int n[3]) {
    const int c = (n[0] > n[1] ? (n[0] > n[2] ? n[0] : n[2]) : (n[1] > n[2] ? n[1] : n[2])) + 4;
    const float m = 1.0e-6f * (float)c;
    return m > 2.5e-4f ? m : 2.5e-4f;
}

// Leap mode for sample j on the forward-box distance field `dist` of the ray's direction
// octant. Returns a value > j when sample j and every sample before the returned index lie
// the margin inside such a box, or j itself when sample j needs its exact position.
// cache_lin / cache_r memoise the last brick looked up (start with cache_lin = -1).
__device__ __forceinline__ int leap_float(const BrickView &bv, const uint8_t *__restrict__ dist,
                                          const float Pf[3], const float df[3],
                                          const float inv_df[3], float step, float inv_step,
                                          int nseg, int j, int &cache_lin, int &cache_r) {
    const float margin = bv.margin;
    if (j >= nseg - 1) return j;  // the last segment's midpoint is not (j + 1/2) ds
    const float m = ((float)j + 0.5f) * step;
    const float B = float_small(bv.B), inv_B = bv.shift == 4 ? 0.0625f : 0.125f;
    int b[3];
    float lo[3];
    bool near = false;  // sample j must sit the margin inside its own brick (interior faces only)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float pa = fmaf(m, df[k], Pf[k]);
        floor_small(pa * inv_B, b[k]);
        b[k] = min(max(b[k], 0), bv.nb[k] - 1);
        lo[k] = float_small(b[k]) * B;  // exact
        const float in = pa - lo[k];
        near |= (in < margin && b[k] > 0) || (in > B - margin && b[k] < bv.nb[k] - 1);
    }
    const int lin = (b[2] * bv.nb[1] + b[1]) * bv.nb[0] + b[0];
    if (lin != cache_lin) {
        cache_lin = lin;
        cache_r = dist[lin];
    }
    const int r = cache_r;
    if (r == 0 || near) return j;
    // exit of the empty forward box of extent r - 1 bricks, faces moved inward by the margin
    const float ahead = float_small(r) * B - margin;
    float texit = INFINITY;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const bool fwd = df[k] > 0.0f;
        const bool inside = fwd ? b[k] + r < bv.nb[k] : (df[k] < 0.0f && b[k] - r + 1 > 0);
        const float face = fwd ? lo[k] + ahead : lo[k] + B - ahead;
        if (inside) texit = fminf(texit, (face - Pf[k]) * inv_df[k]);
    }
    if (!(texit < INFINITY)) return nseg;
    // first sample whose midpoint may reach the moved face
    const float jf = ceilf(fmaf(texit, inv_step, -0.5f));
    const int jn = jf >= (float)nseg ? nseg : (int)jf;
    return max(jn, j + 1);
}

// Two float32 in one 64-bit register pair, with the packed arithmetic of sm_100 (each half
// rounded on its own, as the scalar operations).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// The two 16-bit values of a word as float32, exactly: 2^23 + u by byte insertion, minus 2^23 +
// bias (sub = the pair of -(2^23 + bias)).
__device__ __forceinline__ f32x2 voxels2(uint32_t w, f32x2 sub) {
    return add2(pack2(__uint_as_float(__byte_perm(w, 0x4b00u, 0x5410)),
                      __uint_as_float(__byte_perm(w, 0x4b00u, 0x5432))),
                sub);
}

// Entry (x', y', z') = (x + 2, y + 2, z + 2): the one that starts at voxel (x, y, z). Two entries
// on along an axis lies the same slot of the next block: 8 entries on along x, 8 rnx along y.
constexpr int ENTRY_BYTES = 16;
__device__ __forceinline__ unsigned entry_index(const ReplView &rp, int x, int y, int z) {
    const unsigned X = x + 2, Y = y + 2, Z = z + 2;
    return (((Z >> 1) * rp.rny + (Y >> 1)) * rp.rnx + (X >> 1)) * 8u +
           ((Z & 1) * 4u + (Y & 1) * 2u + (X & 1));
}

// 32 bytes from a 32-byte boundary, through the read-only path.
__device__ __forceinline__ void load32(const void *p, f32x2 v[4]) {
    asm("ld.global.nc.v4.b64 {%0, %1, %2, %3}, [%4];"
        : "=l"(v[0]), "=l"(v[1]), "=l"(v[2]), "=l"(v[3])
        : "l"(p));
}

// Two pairs of float32 from a 16-byte boundary, through the read-only path.
__device__ __forceinline__ void load16(const void *p, f32x2 v[2]) {
    asm("ld.global.nc.v2.b64 {%0, %1}, [%2];" : "=l"(v[0]), "=l"(v[1]) : "l"(p));
}

// The 2^3 voxels from (x, y, z) as they lie in memory: one 16-bit entry, or two of float32, the
// second one voxel on along y (next_y bytes further).
template <bool PACKED>
struct Entry {
    uint4 w;
    __device__ __forceinline__ void load(const char *p, int) { w = __ldg((const uint4 *)p); }
    // pair (x, y) = (k & 1, k >> 1) as float32
    __device__ __forceinline__ f32x2 pair(int k, f32x2 sub) const {
        return voxels2(k == 0 ? w.x : k == 1 ? w.y : k == 2 ? w.z : w.w, sub);
    }
};
template <>
struct Entry<false> {
    f32x2 v[4];
    __device__ __forceinline__ void load(const char *p, int next_y) {
        load16(p, v);
        load16(p + next_y, v + 2);
    }
    __device__ __forceinline__ f32x2 pair(int k, f32x2) const { return v[k]; }
};

// Bytes from an entry at voxel y to the next along y: two slots on in the block, or the same slots
// of the next block (blocks begin at even y).
__device__ __forceinline__ int next_entry_y(const ReplView &rp, int y) {
    return (y & 1) ? (int)rp.row - 2 * ENTRY_BYTES : 2 * ENTRY_BYTES;
}

// The entry at voxel (x, y, z); the first of the 2^3 sets of 2^3 voxels of a sample, and set (x,
// y, z) of them.
__device__ __forceinline__ const char *entry_ptr(const ReplView &rp, int x, int y, int z) {
    return (const char *)rp.base + ENTRY_BYTES * (size_t)entry_index(rp, x, y, z);
}
__device__ __forceinline__ const char *first_entry(const ReplView &rp, const int ip[3]) {
    return entry_ptr(rp, ip[0] - 1, ip[1] - 1, ip[2] - 1);
}
__device__ __forceinline__ const char *entry_at(const ReplView &rp, const char *p, int x, int y,
                                                int z) {
    if (z) p += rp.slice;
    if (y) p += rp.row;
    return x ? p + 8 * ENTRY_BYTES : p;
}

// Calls fn(c, b, v) for the 16 tap rows (y ip1-1+b, z ip2-1+c) of base ip, c outermost; v holds
// the voxels ip0-1 .. ip0+2 of the row.
template <bool PACKED, class Fn>
__device__ __forceinline__ void for_rows_of(const ReplView &rp, const int ip[3], Fn fn) {
    const f32x2 sub = pack2(-rp.magic, -rp.magic);
    const char *p = first_entry(rp, ip);
    const int ny = next_entry_y(rp, ip[1] - 1);
#pragma unroll
    for (int zh = 0; zh < 2; ++zh) {
        float4 v[2][4];  // rows of the lower and the upper z
#pragma unroll
        for (int yh = 0; yh < 2; ++yh) {
            Entry<PACKED> l, u;
            l.load(entry_at(rp, p, 0, yh, zh), ny);
            u.load(entry_at(rp, p, 1, yh, zh), ny);
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const float2 a = unpack2(l.pair(2 * k, sub)), b = unpack2(l.pair(2 * k + 1, sub));
                const float2 c = unpack2(u.pair(2 * k, sub)), d = unpack2(u.pair(2 * k + 1, sub));
                v[0][2 * yh + k] = make_float4(a.x, b.x, c.x, d.x);
                v[1][2 * yh + k] = make_float4(a.y, b.y, c.y, d.y);
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int b = 0; b < 4; ++b) fn(2 * zh + h, b, v[h][b]);
    }
}
template <class Fn>
__device__ __forceinline__ void for_rows(const ReplView &rp, const int ip[3], Fn fn) {
    if (rp.packed) for_rows_of<true>(rp, ip, fn);
    else for_rows_of<false>(rp, ip, fn);
}

// Cubic B-spline sample at integer base ip (taps ip-1 .. ip+2) with fractions f: sums along x,
// then y, then z, two z at a time.
template <bool PACKED>
__device__ __forceinline__ float tricubic_of(const ReplView &rp, const int ip[3],
                                             const float f[3]) {
    const f32x2 sub = pack2(-rp.magic, -rp.magic);
    const char *p = first_entry(rp, ip);
    const int ny = next_entry_y(rp, ip[1] - 1);
    // 16-bit: all loads in flight together; float32 takes twice the registers: z half by z half
    // (with checkpoints 904 -> 776 us for a 640 x 512 image of 253 x 187 x 250 without bricks)
    Entry<PACKED> e[2][2][2];
    auto load = [&](int zh) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            e[zh][k >> 1][k & 1].load(entry_at(rp, p, k & 1, k >> 1, zh), ny);
    };
    if (PACKED) load(0), load(1);
    float wx[4], wy[4], wz[4];
    bspline_w(f[0], wx);
    bspline_w(f[1], wy);
    bspline_w(f[2], wz);
    f32x2 wx2[4], wy2[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        wx2[k] = pack2(wx[k], wx[k]);
        wy2[k] = pack2(wy[k], wy[k]);
    }
    float s = 0.0f;
#pragma unroll
    for (int zh = 0; zh < 2; ++zh) {
        f32x2 plane = 0ull;
        if (!PACKED) load(zh);
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const Entry<PACKED> &l = e[zh][b >> 1][0], &u = e[zh][b >> 1][1];
            const int k = 2 * (b & 1);
            f32x2 r = mul2(wx2[0], l.pair(k, sub));
            r = fma2(wx2[1], l.pair(k + 1, sub), r);
            r = fma2(wx2[2], u.pair(k, sub), r);
            r = fma2(wx2[3], u.pair(k + 1, sub), r);
            plane = fma2(wy2[b], r, plane);
        }
        const float2 pl = unpack2(plane);
        s = fmaf(wz[2 * zh], pl.x, s);
        s = fmaf(wz[2 * zh + 1], pl.y, s);
    }
    return s;
}
__device__ __forceinline__ float tricubic_rep(const ReplView &rp, const int ip[3],
                                              const float f[3]) {
    return rp.packed ? tricubic_of<true>(rp, ip, f) : tricubic_of<false>(rp, ip, f);
}

// Pre-integrated classification: 256 x 256 table of slab (associated rgb, opacity), front
// entry major (preint_table_kernel); PREINT_K sub-steps per entry.
constexpr int PREINT_K = 32;
cudaError_t launch_preint_table(const float4 *tf_tab, float ds, float4 *tab, cudaStream_t st);

// Bilinear lookup at clamped table coordinates (uf, ub) in [0, 255].
__device__ __forceinline__ float4 preint_lookup(const float4 *__restrict__ tab, float uf,
                                                float ub) {
    int i0, k0;
    floor_small(uf, i0);
    floor_small(ub, k0);
    i0 = min(i0, 254);
    k0 = min(k0, 254);
    const float fi = uf - (float)i0, fk = ub - (float)k0;
    const float4 *r0 = tab + i0 * 256 + k0;
    const float4 a = __ldg(r0), b = __ldg(r0 + 1), c = __ldg(r0 + 256), d = __ldg(r0 + 257);
    const float gi = 1.0f - fi, gk = 1.0f - fk;
    float4 o;
    o.x = fmaf(fi, fmaf(fk, d.x, gk * c.x), gi * fmaf(fk, b.x, gk * a.x));
    o.y = fmaf(fi, fmaf(fk, d.y, gk * c.y), gi * fmaf(fk, b.y, gk * a.y));
    o.z = fmaf(fi, fmaf(fk, d.z, gk * c.z), gi * fmaf(fk, b.z, gk * a.z));
    o.w = fmaf(fi, fmaf(fk, d.w, gk * c.w), gi * fmaf(fk, b.w, gk * a.w));
    return o;
}

// The 8 voxels ip .. ip+1 (clamped), x fastest, then y, then z.
template <bool PACKED>
__device__ __forceinline__ void taps8_of(const ReplView &rp, const int ip[3], float v[8]) {
    const f32x2 sub = pack2(-rp.magic, -rp.magic);
    Entry<PACKED> e;
    e.load(entry_ptr(rp, ip[0], ip[1], ip[2]), next_entry_y(rp, ip[1]));
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float2 z = unpack2(e.pair(k, sub));
        v[k] = z.x;
        v[k + 4] = z.y;
    }
}
__device__ __forceinline__ void taps8(const ReplView &rp, const int ip[3], float v[8]) {
    if (rp.packed) taps8_of<true>(rp, ip, v);
    else taps8_of<false>(rp, ip, v);
}

// Trilinear sample at integer base ip with fractions f.
__device__ __forceinline__ float trilinear_rep(const ReplView &rp, const int ip[3],
                                               const float f[3]) {
    float v[8];
    taps8(rp, ip, v);
    const float gx = 1.0f - f[0], gy = 1.0f - f[1], gz = 1.0f - f[2];
    const float r0 = fmaf(f[0], v[1], gx * v[0]), r1 = fmaf(f[0], v[3], gx * v[2]);
    const float r2 = fmaf(f[0], v[5], gx * v[4]), r3 = fmaf(f[0], v[7], gx * v[6]);
    const float q0 = fmaf(f[1], r1, gy * r0), q1 = fmaf(f[1], r3, gy * r2);
    return fmaf(f[2], q1, gz * q0);
}

// Post-classification of value v: u = (v - lo) * du on [0, 255], linear between entries.
struct Classified {
    float u_raw, fu;  // index coordinate before clamping, weight of the upper entry
    int i0;           // lower entry
    float4 c, dc;     // interpolated entry, table difference at i0
};
__device__ __forceinline__ Classified classify(const TfView &tf, float v) {
    Classified k;
    k.u_raw = (v - tf.lo) * tf.du;
    const float u = fminf(fmaxf(k.u_raw, 0.0f), 255.0f);
    const float fl = fminf(floor_small(u, k.i0), 254.0f);
    k.i0 = min(k.i0, 254);
    k.fu = u - fl;
    f32x2 e[4];
    load32(tf.tab + 2 * k.i0, e);
    const float2 dxy = unpack2(e[2]), dzw = unpack2(e[3]);
    k.dc = make_float4(dxy.x, dxy.y, dzw.x, dzw.y);
    const f32x2 fu2 = pack2(k.fu, k.fu);
    const float2 xy = unpack2(fma2(fu2, e[2], e[0])), zw = unpack2(fma2(fu2, e[3], e[1]));
    k.c = make_float4(xy.x, xy.y, zw.x, zw.y);
    return k;
}
__device__ __forceinline__ float4 tf_classify(const TfView &tf, float v) {
    return classify(tf, v).c;
}

// Headlight Blinn-Phong coefficients (local lighting): rgb <- rgb (ka + kd n.L) +
// ks (n.L)^shininess with n.L = |g . d| / sqrt(|g|^2 + eps^2), g the field gradient.
struct Phong {
    float ka, kd, ks, shininess, eps;
};

// Value and gradient of the cubic B-spline at integer base ip with fractions f (derivative
// weights d/df of the weights, the same taps).
template <bool PACKED>
__device__ __forceinline__ float tricubic_grad_of(const ReplView &rp, const int ip[3],
                                                  const float f[3], float g[3]) {
    float wx[4], wy[4], wz[4], dx[4], dy[4], dz[4];
    bspline_w(f[0], wx);
    bspline_w(f[1], wy);
    bspline_w(f[2], wz);
    bspline_dw(f[0], dx);
    bspline_dw(f[1], dy);
    bspline_dw(f[2], dz);
    float s = 0.0f;
    g[0] = g[1] = g[2] = 0.0f;
    const f32x2 sub = pack2(-rp.magic, -rp.magic);
    f32x2 wx2[4], dx2[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        wx2[k] = pack2(wx[k], wx[k]);
        dx2[k] = pack2(dx[k], dx[k]);
    }
    const char *p = first_entry(rp, ip);
    const int ny = next_entry_y(rp, ip[1] - 1);
#pragma unroll
    for (int zh = 0; zh < 2; ++zh) {
        f32x2 ps = 0ull, pdx = 0ull, pdy = 0ull;
#pragma unroll
        for (int yh = 0; yh < 2; ++yh) {
            Entry<PACKED> l, u;
            l.load(entry_at(rp, p, 0, yh, zh), ny);
            u.load(entry_at(rp, p, 1, yh, zh), ny);
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int b = 2 * yh + k;
                const f32x2 v0 = l.pair(2 * k, sub), v1 = l.pair(2 * k + 1, sub);
                const f32x2 v2 = u.pair(2 * k, sub), v3 = u.pair(2 * k + 1, sub);
                const f32x2 r =
                    fma2(wx2[3], v3, fma2(wx2[2], v2, fma2(wx2[1], v1, mul2(wx2[0], v0))));
                const f32x2 rd =
                    fma2(dx2[3], v3, fma2(dx2[2], v2, fma2(dx2[1], v1, mul2(dx2[0], v0))));
                const f32x2 wyb = pack2(wy[b], wy[b]);
                ps = fma2(wyb, r, ps);
                pdx = fma2(wyb, rd, pdx);
                pdy = fma2(pack2(dy[b], dy[b]), r, pdy);
            }
        }
        const float2 p0 = unpack2(ps), p1 = unpack2(pdx), p2 = unpack2(pdy);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = 2 * zh + h;
            s = fmaf(wz[c], h ? p0.y : p0.x, s);
            g[0] = fmaf(wz[c], h ? p1.y : p1.x, g[0]);
            g[1] = fmaf(wz[c], h ? p2.y : p2.x, g[1]);
            g[2] = fmaf(dz[c], h ? p0.y : p0.x, g[2]);
        }
    }
    return s;
}
__device__ __forceinline__ float tricubic_grad_rep(const ReplView &rp, const int ip[3],
                                                   const float f[3], float g[3]) {
    return rp.packed ? tricubic_grad_of<true>(rp, ip, f, g)
                     : tricubic_grad_of<false>(rp, ip, f, g);
}

// Interpolation and classification variants (the paper's Fig. 4 comparison):
// MODE = interp + 2 * preclass. Post-classification classifies the interpolated value;
// pre-classification sums the taps' classified rgba with the interpolation weights.
// MODE_CUBIC_PHONG adds headlight shading to cubic post-classification (d: unit ray
// direction).
enum {
    MODE_CUBIC_POST = 0,
    MODE_LINEAR_POST = 1,
    MODE_CUBIC_PRE = 2,
    MODE_LINEAR_PRE = 3,
    MODE_CUBIC_PHONG = 4,
    MODE_PREINT = 5  // slabs through the pre-integration table (per-ray kernel, no skipping)
};

template <int MODE>
__device__ __forceinline__ float4 sample_rgba(const ReplView &rp, const TfView &tf,
                                              const int ip[3], const float f[3],
                                              const float d[3] = nullptr,
                                              const Phong *ph = nullptr) {
    if constexpr (MODE == MODE_CUBIC_POST) {
        return tf_classify(tf, tricubic_rep(rp, ip, f));
    } else if constexpr (MODE == MODE_CUBIC_PHONG) {
        float g[3];
        float4 c = tf_classify(tf, tricubic_grad_rep(rp, ip, f, g));
        const float gd = fmaf(g[0], d[0], fmaf(g[1], d[1], g[2] * d[2]));
        const float gg = fmaf(g[0], g[0], fmaf(g[1], g[1], fmaf(g[2], g[2], ph->eps * ph->eps)));
        const float nl = fabsf(gd) / sqrtf(gg);
        const float diff = fmaf(ph->kd, nl, ph->ka);
        const float spec = ph->ks * exp2f(ph->shininess * log2f(nl));
        c.x = fmaf(c.x, diff, spec);
        c.y = fmaf(c.y, diff, spec);
        c.z = fmaf(c.z, diff, spec);
        return c;
    } else if constexpr (MODE == MODE_LINEAR_POST) {
        return tf_classify(tf, trilinear_rep(rp, ip, f));
    } else if constexpr (MODE == MODE_CUBIC_PRE) {
        float wx[4], wy[4], wz[4];
        bspline_w(f[0], wx);
        bspline_w(f[1], wy);
        bspline_w(f[2], wz);
        float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        for_rows(rp, ip, [&](int c, int b, const float4 &v) {
            const float vals[4] = {v.x, v.y, v.z, v.w};
            const float wyz = wy[b] * wz[c];
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const float4 t = tf_classify(tf, vals[a]);
                const float w = wx[a] * wyz;
                acc.x = fmaf(w, t.x, acc.x);
                acc.y = fmaf(w, t.y, acc.y);
                acc.z = fmaf(w, t.z, acc.z);
                acc.w = fmaf(w, t.w, acc.w);
            }
        });
        return acc;
    } else {
        float v[8];
        taps8(rp, ip, v);
        float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
        for (int k = 0; k < 4; ++k) {  // the rows (y, z) of the taps
            const float wyz = ((k & 1) ? f[1] : 1.0f - f[1]) * ((k >> 1) ? f[2] : 1.0f - f[2]);
            const float4 t0 = tf_classify(tf, v[2 * k]), t1 = tf_classify(tf, v[2 * k + 1]);
            const float wa = (1.0f - f[0]) * wyz, wb = f[0] * wyz;
            acc.x = fmaf(wb, t1.x, fmaf(wa, t0.x, acc.x));
            acc.y = fmaf(wb, t1.y, fmaf(wa, t0.y, acc.y));
            acc.z = fmaf(wb, t1.z, fmaf(wa, t0.z, acc.z));
            acc.w = fmaf(wb, t1.w, fmaf(wa, t0.w, acc.w));
        }
        return acc;
    }
}

__device__ __forceinline__ int brick_of(const BrickView &bv, const int ip[3]) {
    return ((max(ip[2], 0) >> bv.shift) * bv.nb[1] + (max(ip[1], 0) >> bv.shift)) * bv.nb[0] +
           (max(ip[0], 0) >> bv.shift);
}

__device__ __forceinline__ int octant_of(const float df[3]) {
    return (df[0] < 0.0f) | ((df[1] < 0.0f) << 1) | ((df[2] < 0.0f) << 2);
}

// Split render (k_render_split.cu): the first phase composites samples 0 .. SPLIT_J0 - 1 of
// every ray with one lane and hands rays that go on to a queue; the second phase finishes
// each queued ray with SPLIT_G lanes (blocks of SPLIT_G consecutive samples composited by a
// scan), so no ray's cost rests on one lane. With SPLIT_J0 = 0 (the measured best on the
// 512^2 x 400 CT) the first phase only sets rays up and leaps each to its first sample in an
// occupied brick. SPLIT_G = 16 at four CTAs per SM measured best on that CT (8 lanes: 1.4%
// slower, 32 lanes 12% slower, 4 lanes 25% slower).
constexpr int SPLIT_G = 16;
constexpr int SPLIT_J0 = 0;  // a multiple of SPLIT_G
struct RaySplit {
    unsigned *head;     // [records at the front, records claimed, records at the back]
    unsigned *next;     // NULL, or the counters of the next render, which the second phase clears
    float4 *rec;        // SPLIT_REC float4 per queued ray (split_store)
    unsigned cap;       // records the queue holds (>= the image's pixels)
    unsigned long_len;  // rays with more samples left go to the front (claimed first)
};
constexpr int SPLIT_REC = 7;

// A queued ray: its sample placement record, the next sample index, the colour and
// transmittance composited so far and its pixel.
__device__ __forceinline__ void split_store(float4 *r, const RayPos &rp, int j, int pix, float C0,
                                            float C1, float C2, float T) {
    r[0] = make_float4(__int_as_float(rp.I0[0]), __int_as_float(rp.I0[1]),
                       __int_as_float(rp.I0[2]), __int_as_float(rp.nseg));
    r[1] = make_float4(rp.r0[0].hi, rp.r0[0].lo, rp.r0[1].hi, rp.r0[1].lo);
    r[2] = make_float4(rp.r0[2].hi, rp.r0[2].lo, rp.d[0].hi, rp.d[0].lo);
    r[3] = make_float4(rp.d[1].hi, rp.d[1].lo, rp.d[2].hi, rp.d[2].lo);
    r[4] = make_float4(rp.mlast.hi, rp.mlast.lo, rp.dlast, __int_as_float(j));
    r[5] = make_float4(C0, C1, C2, T);
    r[6] = make_float4(__int_as_float(pix), 0.0f, 0.0f, 0.0f);
}

__device__ __forceinline__ void split_load(const float4 *r, RayPos &rp, int &j, int &pix,
                                           float &C0, float &C1, float &C2, float &T) {
    const float4 a = __ldcg(r), b = __ldcg(r + 1), c = __ldcg(r + 2), d = __ldcg(r + 3);
    const float4 e = __ldcg(r + 4), f = __ldcg(r + 5), g = __ldcg(r + 6);
    rp.I0[0] = __float_as_int(a.x);
    rp.I0[1] = __float_as_int(a.y);
    rp.I0[2] = __float_as_int(a.z);
    rp.nseg = __float_as_int(a.w);
    rp.r0[0] = {b.x, b.y};
    rp.r0[1] = {b.z, b.w};
    rp.r0[2] = {c.x, c.y};
    rp.d[0] = {c.z, c.w};
    rp.d[1] = {d.x, d.y};
    rp.d[2] = {d.z, d.w};
    rp.mlast = {e.x, e.y};
    rp.dlast = e.z;
    j = __float_as_int(e.w);
    C0 = f.x;
    C1 = f.y;
    C2 = f.z;
    T = f.w;
    pix = __float_as_int(g.x);
}

struct RenderLaunch {
    VolView vol;
    ReplView rep;
    TfView tf;
    CamDev cam;
    RayGrid grid;
    const uint8_t *dist;  // NULL: no leaping; else 8 x nbricks forward-box distances
    BrickView bricks;
    float4 *out;
    unsigned long long *counters;  // NULL or [nominal, executed]
    int *err;                      // device error word
    RaySplit split;                // used by the split render only
    const uint32_t *cells;         // NULL, or the cell transparency mask (with dist)
    int mode;                      // interpolation / classification variant (MODE_*)
    Phong phong;                   // MODE_CUBIC_PHONG only
    const float4 *preint;          // MODE_PREINT only: the table for slabs of length step
    float4 *accum;                 // NULL, or the running (C, T) image of an ordered pass
    int accum_pitch;               // its pixels per row (the full image's width)
    // checkpoints for the reverse mode (NULL: none): per pixel (first checkpointed segment,
    // last composited sample) in ckpt_head, and ckpt_K floats from ckpt + pixel * ckpt_K: the
    // transmittance at the start of segments of ckpt_seg samples
    int2 *ckpt_head;
    float *ckpt;
    int ckpt_K, ckpt_seg;
    const void *tma_map;  // host address of the volume's tensor map (kernel 7; launcher only)
    // serving by device-side launches (k_serve_dl.cu): the second phase's grid, and where its
    // CTAs count themselves and the last one announces the request's completion (NULL: none)
    int tail_ctas;
    int *done_ctr;
    int *done_flag;
    int done_seq;
};

// Checkpoint state of one ray while it is composited (reverse-mode checkpoints).
struct CkState {
    float *row;  // the ray's ckpt_K floats
    int first;   // first segment written (-1: none yet)
    int last;    // last segment written
    int jlast;   // last composited sample (-1: none)
};

// Segments that the longest ray of a volume box can hold at `step` in segments of `seg`.
inline int ckpt_segments(const int n[3], float step, int seg) {
    const double d = __builtin_sqrt((double)n[0] * n[0] + (double)n[1] * n[1] + (double)n[2] * n[2]);
    const double samples = __builtin_ceil(d / (double)step) + 2.0;
    return (int)__builtin_ceil(samples / (double)seg);
}

// Cell transparency mask: cells c = -1 .. n-1 per axis in blocks of 4^3, cell c in block
// (c + 4) >> 2 (blocks do not straddle bricks; block 0 holds the cells -1), block
// (bz * cell_blocks(ny) + by) * cell_blocks(nx) + bx, two 32-bit words per block (c_z & 2 picks
// the word), bit 16 (c_z & 1) + 4 (c_y & 3) + (c_x & 3). A ray's next samples mostly fall into
// the word it read last, and 32 bytes hold a run of 4 blocks. A tile is 2^3 blocks: cell c in
// tile (c + 8) >> 3.
VRC_HD int cell_blocks(int n) { return ((n + 3) >> 2) + 1; }
VRC_HD int cell_tiles(int n) { return ((n + 7) >> 3) + 1; }

// The word and the bit in it of the cell holding sample base ip (ip in [-1, n-1]).
__device__ __forceinline__ uint32_t cell_word(const uint32_t *__restrict__ cells, const int n[3],
                                              const int ip[3]) {
    const int cx = ip[0] + 4, cy = ip[1] + 4, cz = ip[2] + 4;
    const int blk = ((cz >> 2) * cell_blocks(n[1]) + (cy >> 2)) * cell_blocks(n[0]) + (cx >> 2);
    return __ldg(cells + 2 * blk + ((cz >> 1) & 1));
}
__device__ __forceinline__ bool cell_bit(uint32_t w, const int ip[3]) {
    return (w >> (((ip[2] & 1) << 4) | ((ip[1] & 3) << 2) | (ip[0] & 3))) & 1u;
}

// 0: the opacity of samples at base ip is zero.
__device__ __forceinline__ bool cell_open(const uint32_t *__restrict__ cells, const int n[3],
                                          const int ip[3]) {
    return cell_bit(cell_word(cells, n, ip), ip);
}

// Quick skip test of sample j < nseg - 1 from its float position (the leap path's, within a
// third of the margin of the exact one). Away from cell faces (by the margin) the float cell
// is the exact cell, so the brick and cell tests need no exact
// placement: QS_EMPTY_BRICK and QS_CLEAR_CELL mean opacity zero (skip), QS_OPEN means the
// sample must be resampled; QS_EXACT (near a face) means take the exact position first.
// Without a cell mask (cells == NULL) only the brick is tested.
enum { QS_EXACT = 0, QS_EMPTY_BRICK = 1, QS_CLEAR_CELL = 2, QS_OPEN = 3 };
__device__ __forceinline__ int quick_skip(const BrickView &bv, const uint8_t *__restrict__ dist,
                                          const uint32_t *__restrict__ cells, const int n[3],
                                          const float Pf[3], const float df[3], float step,
                                          int j, int &cache_lin, int &cache_empty) {
    const float m = ((float)j + 0.5f) * step;
    int c[3];
    bool near = false;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float pk = fmaf(m, df[k], Pf[k]);
        const float fl = floorf(pk);
        const float fr = pk - fl;
        near |= !(fr >= bv.margin && fr <= 1.0f - bv.margin);
        c[k] = min(max((int)fl, -1), n[k] - 1);
    }
    if (near) return QS_EXACT;
    const int lin = ((max(c[2], 0) >> bv.shift) * bv.nb[1] + (max(c[1], 0) >> bv.shift)) *
                        bv.nb[0] + (max(c[0], 0) >> bv.shift);
    if (lin != cache_lin) {
        cache_lin = lin;
        cache_empty = dist[lin] != 0;
    }
    if (cache_empty) return QS_EMPTY_BRICK;
    if (!cells) return QS_OPEN;
    return cell_open(cells, n, c) ? QS_OPEN : QS_CLEAR_CELL;
}

// Launchers (return cudaSuccess or the launch error).
// Writes a volume's resident copies: the padded one (VolView) and the render layout (rep_view
// gives its extents; rep_bytes its size).
ReplView rep_view(const void *base, int dtype, const int n[3]);
size_t rep_bytes(int dtype, const int n[3]);
cudaError_t launch_volume_layouts(const void *src, int dtype, const int n[3], void *pad, int pnx,
                                  void *rep, cudaStream_t st);
cudaError_t launch_brick_minmax(const VolView &v, int B, void *mn, void *mx, cudaStream_t st);
cudaError_t launch_occupancy(const void *mn, const void *mx, int dtype, long nbricks,
                             const int *prefix_dev, float lo, float du, uint8_t *occ,
                             cudaStream_t st);
// Cell transparency mask of a padded volume for a transfer function (layout: cell_open), given
// its occupancy with bricks of size B and the run id of each zero-opacity table entry (1, 2,
// ... per maximal run of zero entries; 0 for entries of non-zero opacity).
size_t cellmask_bytes(const int n[3]);
cudaError_t launch_cellmask(const VolView &v, int B, const int nb[3], const uint8_t *occ,
                            const uint8_t *zrun_dev, float lo, float du, uint32_t *cells,
                            cudaStream_t st);
// Occupancy bytes of the 8^3 tiles (cells 8t .. 8t + 7 per axis, tile 0 also the cells -1; nt =
// ceil(n / 8) of them): 1 where the mask has an open cell.
cudaError_t launch_tile_occupancy(const uint32_t *cells, const int n[3], const int nt[3],
                                  uint8_t *tiles, cudaStream_t st);
// The mask as rows of 32-cell words along x, the layout vrc_cellmask_get returns.
long cellmask_row_words(const int n[3]);
cudaError_t launch_cellmask_rows(const uint32_t *cells, const int n[3], uint32_t *out,
                                 cudaStream_t st);
size_t box_dist_scratch_bytes(const int nb[3]);
// dist: 8 x nbricks bytes (one forward-box distance field per direction octant)
cudaError_t launch_box_dist(const uint8_t *occ, const int nb[3], uint8_t *scratch, uint8_t *dist,
                             cudaStream_t st);
// Object-order pieces and sort-last compositing (k_pieces.cu).
constexpr int MAX_PIECES = 64;
// Partials listed front to back; partial k covers the image pixels [rect[k][0], +rect[k][2])
// x [rect[k][1], +rect[k][3]), rect[k][2] pixels per row.
struct CompositeArgs {
    int K, width, height;
    const float4 *part[MAX_PIECES];
    int rect[MAX_PIECES][4];
};
// out: 6 int16 per brick (tight visible box, half-open cell coordinates, zeros when empty)
cudaError_t launch_brick_aabbs(const uint32_t *cells, const int n[3], int B, const int nb[3],
                               const uint8_t *occ, int16_t *out,
                               cudaStream_t st);
cudaError_t launch_piece_mask(const uint8_t *occ, const int nb[3], const int blo[3],
                              const int bhi[3], uint8_t *out, cudaStream_t st);
// bricks_k: K x 6 ints (device; brick lo, hi of each piece); out: K x 6 ints (device)
cudaError_t launch_piece_boxes(const int16_t *aabb, const int nb[3], const int *bricks_k, int K,
                               int *out, cudaStream_t st);
cudaError_t launch_composite(const CompositeArgs &a, float4 *out, cudaStream_t st);
// ordered pass: accum = (0, 0, 0, 1) everywhere; out = (C, 1 - T) of accum
cudaError_t launch_accum_init(float4 *accum, long n, cudaStream_t st);
cudaError_t launch_accum_finish(const float4 *accum, float4 *out, long n, cudaStream_t st);
cudaError_t launch_render_ray(const RenderLaunch &L, cudaStream_t st);
// TMA-staged render (k_render_tma.cu): a float32 copy of the padded volume (same layout as
// VolView, element type float) and a tensor map of it (tma_map_bytes() bytes, 64-byte
// aligned) are built once per volume; L.tma_map points at the map.
cudaError_t launch_padded_to_float(const VolView &v, float *dst, cudaStream_t st);
size_t tma_map_bytes();
cudaError_t encode_tma_map(void *map_out, const float *base, int pnx, int pny, int pnz);
cudaError_t launch_render_tma(const void *map, const RenderLaunch &L, cudaStream_t st);
cudaError_t launch_render_warp(const RenderLaunch &L, int lanes_per_ray, cudaStream_t st);
// Both phases of the split render; L.split.head must be zero. L.split.next, if given, is zero at
// the end.
cudaError_t launch_render_split(const RenderLaunch &L, cudaStream_t st);

// Reverse mode of one render: grad_out is the loss gradient per pixel (H x W x RGBA);
// grad_tf (256 x 4) and grad_vol (nx*ny*nz, x fastest, may be NULL) are accumulated.
constexpr int ADJ_MAX_SEG = 128;   // largest checkpoint interval (samples)
struct AdjointLaunch {
    RenderLaunch L;
    const float4 *grad_out;
    float *grad_tf;
    float *grad_vol;
    int seg;
    int open_alpha;  // derivative from above at table opacity 0
};
cudaError_t launch_adjoint(const AdjointLaunch &A, cudaStream_t st);

// Microbenchmarks of the stencil's roofs (k_microbench.cu): FP32 fused multiply-adds, 16-byte
// loads that hit in L1, 16-byte loads from shared memory, 16-byte float atomics to global.
enum { MB_FMA = 0, MB_L1 = 1, MB_LDS = 2, MB_RED = 3 };
size_t microbench_scratch_bytes();
size_t microbench_red_bytes();
cudaError_t launch_microbench(int kind, int ctas, int iters, void *scratch, void *red_buf,
                              cudaStream_t st);
double microbench_work(int kind, int ctas, int iters);  // flops (MB_FMA) or bytes per launch

// Persistent serving (k_serve.cu). A slot holds one request; the queue holds (slot, seq)
// entries in arrival order; ctl holds the device-side front and the host-published tail.
// The persistent serving kernel: warps per CTA and CTAs per SM (64 registers per thread, the
// occupancy of the split render's second phase: the bodies are bound by the latency of
// dependent loads, so every SM keeps as many warps resident as it can).
constexpr int SERVE_WARPS = 8;
constexpr int SERVE_CTAS_PER_SM = 4;
struct ServeSlot {
    RenderLaunch L;          // the request's render (L.split.head != NULL: split render, with
                             // the request's own ray queue)
    int seq;                 // the request in the slot (sequence number)
    int state;               // 0 phase 1, 1 queued rays open, 2 every item claimed or none left
    int p1_rem;              // tiles not yet claimed (claims subtract; <= 0: none)
    int p2_rem;              // queued rays not yet claimed (opened by the end of phase 1)
    int ntiles;              // 8 x 4 pixel tiles of its image
    int stride;              // tile order: k -> k * stride mod ntiles (stride coprime to ntiles)
    int p1_done;             // tiles finished (device atomics)
    int p2_total;            // rays phase 1 queued (set when phase 1 finishes)
    int p2_nf;               // of them, records at the queue's front
    int p2_done;             // queued rays finished (device atomics)
    unsigned qhead[4];       // the split request's ray-queue counters (front, -, back)
    int pad[2];
};
struct ServeEntry {
    int slot;
    int seq;
};
struct ServeCtl {
    unsigned long long front;   // oldest queue entry that may still have queued rays to claim
    unsigned long long tail;    // entries published by the host
    int stop;                   // host request to leave
    int leaving;                // set by the first warp that times out; no new claims after it
    unsigned long long front1;  // oldest entry that may still have tiles to claim (>= front)
    unsigned long long epoch;   // bumped whenever queued rays open for claiming
};
// front_mirror: host-mapped copy of ctl->front (a lower bound of it) that the host reads
// before it publishes a new entry into the ring of `cap` entries; sms: the device's SM count
cudaError_t launch_serve(ServeSlot *slots, const ServeEntry *queue, int cap, ServeCtl *ctl,
                         int *done_flags, unsigned long long *front_mirror,
                         unsigned long long budget_ns, unsigned long long idle_ns, int sms,
                         cudaStream_t st);
// Serving by device-side launches: one scheduler thread launches each request's split render
// (both phases, plain kernels whose launch record is a kernel parameter) as it arrives.
cudaError_t launch_serve_dl(ServeSlot *slots, const ServeEntry *queue, int cap, ServeCtl *ctl,
                            unsigned long long *front_mirror, unsigned long long budget_ns,
                            unsigned long long idle_ns, cudaStream_t stream);
// CTAs of a device-launched second phase (fills the device; cached per device).
int serve_dl_tail_ctas(cudaError_t &e);

}  // namespace vrc
