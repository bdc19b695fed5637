// Volume layouts, brick min/max tables and transfer-function occupancy.
//
// Brick tables are the auxiliary structures of the paper's block decomposition
// (Sec. "Methodology", Fig. 3; Sec. "Analysis", Pros (b)): brick b covers voxels [bB, bB+B)
// per axis and stores min/max over its apron box [bB-1, bB+B+1] clamped to the volume, the
// overlap a cubic kernel reads. The occupancy of a brick under a transfer function is the
// integer decision "is any table opacity > 0 on the brick's value range", taken in float32.
#include <string.h>

#include "vrc_internal.h"

namespace vrc {

// ------------------------------------------------------------------ volume layouts ------
// One warp per 2 x 2 rows (y', z') of the padded copy: it writes those rows and the row of blocks
// of render entries (ReplView) at the same place. The 3 x 3 rows it needs go through shared
// memory, VL_SPAN words of each at a time (each source voxel comes from HBM once, the rest from
// L2), from where consecutive lanes write consecutive 32-byte pieces of the blocks, past L2 (the
// padded copy, which the brick table reads next, may stay). Words of a row lie VL_Y and VL_Z
// apart, so that the four rows read at once fall on different banks.
// Bound: HBM, 2 (or 4) bytes read, as many padded and 16 of render layout written per voxel.
// 512^2 x 400 int16 (2.1 GB): 356 us, 5.9 TB/s; a warp per row that read its four source rows
// element by element, which the L1 data path bound: 388 us.
constexpr int VL_WARPS = 8, VL_SPAN = 128, VL_Y = 136, VL_Z = 432;

// 32 bytes to a 32-byte boundary, not kept in L2.
__device__ __forceinline__ void store32_streaming(void *p, const uint32_t v[8]) {
    asm volatile("st.global.cs.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(v[0]),
                 "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}

template <typename T>
__global__ void __launch_bounds__(32 * VL_WARPS)
    volume_layouts_kernel(const T *__restrict__ src, int nx, int ny, int nz, T *__restrict__ pad,
                          int pnx, char *__restrict__ rep, int rnx, int rny, int rnz) {
    constexpr int PER = 4 / (int)sizeof(T), SPAN = VL_SPAN * PER;  // voxels a word, a span
    constexpr int BLOCK = 8 * ENTRY_BYTES;
    __shared__ __align__(16) uint32_t s_rows[VL_WARPS][3 * VL_Z];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t *rows = s_rows[warp];
    const unsigned unit = blockIdx.x * VL_WARPS + warp;
    const int pny = ny + 2 * PAD, pnz = nz + 2 * PAD;
    const unsigned ny2 = (unsigned)(pny + 1) >> 1;
    const int by = (int)(unit % ny2), bz = (int)(unit / ny2);
    if (2 * bz >= pnz) return;
    const T *from[9];  // source rows of the padded rows (2 by + r % 3, 2 bz + r / 3)
    uintptr_t low = 0;
#pragma unroll
    for (int r = 0; r < 9; ++r) {
        from[r] = src + ((size_t)min(max(2 * bz + r / 3 - PAD, 0), nz - 1) * ny +
                         min(max(2 * by + r % 3 - PAD, 0), ny - 1)) * nx;
        low |= (uintptr_t)from[r];
    }
    const bool words = (low & 3) == 0;  // 16-bit voxels 2i, 2i + 1 in one load
    const bool blocks = by < rny && bz < rnz;
    char *out = rep + ((size_t)bz * rny + by) * rnx * BLOCK;
    for (int x0 = 0; x0 < max(pnx, 2 * rnx); x0 += SPAN) {
        __syncwarp();  // the span before has been read
        // padded elements x0 .. x0 + SPAN + 3
        for (int i = lane; i < VL_SPAN + 4 / PER; i += 32) {
            const int x = x0 + i * PER - PAD;
            uint32_t w[9];
            if (sizeof(T) == 4 || (words && x >= 0 && x + 1 < nx)) {
                const int xc = sizeof(T) == 4 ? min(max(x, 0), nx - 1) : x;
#pragma unroll
                for (int r = 0; r < 9; ++r) w[r] = *(const uint32_t *)(from[r] + xc);
            } else {
                const int xa = min(max(x, 0), nx - 1), xb = min(max(x + 1, 0), nx - 1);
#pragma unroll
                for (int r = 0; r < 9; ++r)
                    w[r] = (uint32_t)(uint16_t)from[r][xa] | (uint32_t)(uint16_t)from[r][xb] << 16;
            }
#pragma unroll
            for (int r = 0; r < 9; ++r) rows[(r % 3) * VL_Y + (r / 3) * VL_Z + i] = w[r];
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < 4; ++r) {  // padded rows, 4 elements per lane (pnx is a multiple of 8)
            const int y = 2 * by + (r & 1), z = 2 * bz + (r >> 1);
            const uint32_t *s0 = rows + (r & 1) * VL_Y + (r >> 1) * VL_Z;
            if (y >= pny || z >= pnz) continue;
            T *to = pad + ((size_t)z * pny + y) * pnx;
            for (int x = x0 + 4 * lane; x < min(pnx, x0 + SPAN); x += 128) {
                if constexpr (sizeof(T) == 2)
                    *(uint2 *)(to + x) = *(const uint2 *)(s0 + (x - x0) / 2);
                else *(uint4 *)(to + x) = *(const uint4 *)(s0 + (x - x0));
            }
        }
        if (!blocks) continue;
        const int kend = min(rnx - x0 / 2, SPAN / 2);
        // lane: the entries x' = 2k, 2k + 1 of (y', z') = (2 by + g, 2 bz + h) in block k
        const int g = lane & 1, h = (lane >> 1) & 1;
        const uint32_t *s0 = rows + g * VL_Y + h * VL_Z;
        char *to = out + (size_t)(x0 / 2) * BLOCK + 2 * ENTRY_BYTES * (lane & 3);
        if constexpr (sizeof(T) == 2) {
            // int16: bias 32768, i.e. the sign bit flipped
            const uint32_t flip = (T)-1 < (T)0 ? 0x80008000u : 0u;
            for (int k = lane >> 2; k < kend; k += 8) {
                uint32_t e[3][2];  // pairs of voxel 2k - 2 + i of row y
#pragma unroll
                for (int y = 0; y < 2; ++y) {
                    const uint32_t *a = s0 + y * VL_Y + k, *b = a + VL_Z;
                    e[0][y] = __byte_perm(a[0], b[0], 0x5410) ^ flip;
                    e[1][y] = __byte_perm(a[0], b[0], 0x7632) ^ flip;
                    e[2][y] = __byte_perm(a[1], b[1], 0x5410) ^ flip;
                }
                const uint32_t v[8] = {e[0][0], e[1][0], e[0][1], e[1][1],
                                       e[1][0], e[2][0], e[1][1], e[2][1]};
                store32_streaming(to + k * BLOCK, v);
            }
        } else {
            for (int k = lane >> 2; k < kend; k += 8) {
                const uint32_t *a = s0 + 2 * k, *b = a + VL_Z;
                const uint32_t v[8] = {a[0], b[0], a[1], b[1], a[1], b[1], a[2], b[2]};
                store32_streaming(to + k * BLOCK, v);
            }
        }
    }
}

ReplView rep_view(const void *base, int dtype, const int n[3]) {
    ReplView r;
    r.base = base;
    r.packed = dtype != DT_F32;
    r.rnx = (n[0] + 4) / 2;
    r.rny = (n[1] + (r.packed ? 4 : 5)) / 2;
    r.row = 8 * ENTRY_BYTES * (size_t)r.rnx;
    r.slice = r.row * r.rny;
    r.magic = 8388608.0f + (dtype == DT_I16 ? 32768.0f : 0.0f);
    return r;
}

size_t rep_bytes(int dtype, const int n[3]) {
    const ReplView r = rep_view(nullptr, dtype, n);
    return r.slice * ((n[2] + 4) / 2);
}

cudaError_t launch_volume_layouts(const void *src, int dtype, const int n[3], void *pad, int pnx,
                                  void *rep, cudaStream_t st) {
    const ReplView r = rep_view(rep, dtype, n);
    const int rnz = (n[2] + 4) / 2;
    const long units = (long)((n[1] + 2 * PAD + 1) / 2) * ((n[2] + 2 * PAD + 1) / 2);
    const unsigned blocks = (unsigned)((units + VL_WARPS - 1) / VL_WARPS);
    switch (dtype) {
    case DT_U16:
        volume_layouts_kernel<uint16_t><<<blocks, 32 * VL_WARPS, 0, st>>>(
            (const uint16_t *)src, n[0], n[1], n[2], (uint16_t *)pad, pnx, (char *)rep, r.rnx,
            r.rny, rnz);
        break;
    case DT_I16:
        volume_layouts_kernel<int16_t><<<blocks, 32 * VL_WARPS, 0, st>>>(
            (const int16_t *)src, n[0], n[1], n[2], (int16_t *)pad, pnx, (char *)rep, r.rnx,
            r.rny, rnz);
        break;
    default:
        volume_layouts_kernel<float><<<blocks, 32 * VL_WARPS, 0, st>>>(
            (const float *)src, n[0], n[1], n[2], (float *)pad, pnx, (char *)rep, r.rnx, r.rny,
            rnz);
    }
    return cudaGetLastError();
}

// ------------------------------------------------------------------ brick min/max ------
template <typename T>
struct Lim;
template <>
struct Lim<uint16_t> {
    __device__ static uint16_t lo() { return 0; }
    __device__ static uint16_t hi() { return 0xFFFF; }
};
template <>
struct Lim<int16_t> {
    __device__ static int16_t lo() { return -32768; }
    __device__ static int16_t hi() { return 32767; }
};
template <>
struct Lim<float> {
    __device__ static float lo() { return -INFINITY; }
    __device__ static float hi() { return INFINITY; }
};

// Two 16-bit values at a time.
template <typename T>
__device__ __forceinline__ uint32_t min2(uint32_t a, uint32_t b) {
    uint32_t r;
    if constexpr ((T)-1 < (T)0) asm("min.s16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    else asm("min.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
template <typename T>
__device__ __forceinline__ uint32_t max2(uint32_t a, uint32_t b) {
    uint32_t r;
    if constexpr ((T)-1 < (T)0) asm("max.s16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    else asm("max.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

template <typename T>
__device__ __forceinline__ T tmin(T a, T b) { return a < b ? a : b; }
template <typename T>
__device__ __forceinline__ T tmax(T a, T b) { return a > b ? a : b; }

// Min/max over rows of brick bx's apron, x in [bx*B - 1, bx*B + B + 1]: the padded row's elements
// bx*B + 1 .. bx*B + B + 3, i.e. the brick's own span but for its first element, and the first 4
// elements of the next span. 16-bit: a lane takes the span of one brick, 16 bytes a load, and keeps
// the two extremes apart; the next lane's first-4 extreme is fetched once, after the last row. The
// pad replicates the edge voxels (also in the rounding of pnx, a multiple of 8), so what lies
// past a row's end adds nothing. 16-bit voxels are compared two at a time.
template <typename T>
struct Pair16 {  // 8 elements in 4 words
    using V = uint32_t;
    __device__ static V none_lo() { return (uint32_t)(uint16_t)Lim<T>::hi() * 0x10001u; }
    __device__ static V none_hi() { return (uint32_t)(uint16_t)Lim<T>::lo() * 0x10001u; }
    __device__ static V least(V a, V b) { return min2<T>(a, b); }
    __device__ static V most(V a, V b) { return max2<T>(a, b); }
    __device__ static V skip_first(V a) { return __byte_perm(a, 0u, 0x3232); }
    __device__ static T low(V a) { return tmin((T)a, (T)(a >> 16)); }
    __device__ static T high(V a) { return tmax((T)a, (T)(a >> 16)); }
};
// The whole apron span of a row by one thread (float32).
template <int B>
__device__ __forceinline__ void apron_row(const float *__restrict__ r, int bx, int pnx, float &lo,
                                          float &hi) {
    float v[B + 4];
    const int i0 = bx * B;
    if (i0 + B + 4 <= pnx) {
        const float4 *p = reinterpret_cast<const float4 *>(r + i0);
#pragma unroll
        for (int k = 0; k < (B + 4) / 4; ++k) {
            const float4 w = __ldg(p + k);
            memcpy(&v[k * 4], &w, 16);
        }
    } else {
#pragma unroll
        for (int e = 0; e < B + 4; ++e) v[e] = r[min(i0 + e, pnx - 1)];
    }
#pragma unroll
    for (int e = 1; e < B + 4; ++e) {
        lo = tmin(lo, v[e]);
        hi = tmax(hi, v[e]);
    }
}

// One CTA per brick row (by, bz): thread x handles brick bx (64 at a time) and sweeps the
// rows of the (y, z) apron, thread y interleaves those rows; partial min/max are combined
// through shared memory. Each voxel is read from HBM about once (neighbouring rows of bricks
// re-read the overlap through L2). Exact for every dtype.
// Bound: latency of the loads. 512^2 x 400 int16, B = 8: 53 us (217 MB read, 4.1 TB/s); with three
// 8-byte loads of the overlapping 12 elements a brick and row 82 us. Float32 spans are 32 bytes or
// more and keep overlapping loads, row by row over the threads y: 36 us for 256^3 (41 us by the
// lanes' own spans, 56 us slice by slice).
constexpr int BM_TX = 64, BM_TY = 4;

template <typename T, int B>
__global__ void __launch_bounds__(BM_TX *BM_TY) brick_minmax_kernel(VolView v, int nbx, int nby,
                                                                     int nbz, T *__restrict__ mn,
                                                                     T *__restrict__ mx) {
    __shared__ T s_lo[BM_TY][BM_TX], s_hi[BM_TY][BM_TX];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int by = blockIdx.x % nby, bz = blockIdx.x / nby;
    if (bz >= nbz) return;
    const int y0 = max(by * B - 1, 0), y1 = min(by * B + B + 1, v.n[1] - 1);
    const int z0 = max(bz * B - 1, 0), z1 = min(bz * B + B + 1, v.n[2] - 1);
    const T *base = (const T *)v.base;
    for (int bx0 = 0; bx0 < nbx; bx0 += BM_TX) {
        const int bx = bx0 + tx;
        T least = Lim<T>::hi(), most = Lim<T>::lo();
        if constexpr (sizeof(T) == 4) {
            if (bx < nbx) {
                const int wy = y1 - y0 + 1, rows = wy * (z1 - z0 + 1);
                for (int r = ty; r < rows; r += BM_TY) {
                    const int y = y0 + r % wy, z = z0 + r / wy;
                    apron_row<B>(base + ((long)(z + PAD) * v.pny + (y + PAD)) * v.pnx, bx, v.pnx,
                                 least, most);
                }
            }
        } else {
            using X = Pair16<T>;
            using V = typename X::V;
            V lo = X::none_lo(), hi = X::none_hi();    // own span without its first element
            V flo = X::none_lo(), fhi = X::none_hi();  // first 4 elements of the span
            V nlo = X::none_lo(), nhi = X::none_hi();  // lane 31: of the next lane's span
            // spans (of whole 8-element pieces) inside the row; lanes past the last brick read
            // theirs for the lane before
            const bool last = (tx & 31) == 31 && (bx + 1) * B < v.pnx;
            for (int z = z0 + ty; z <= z1; z += BM_TY) {
                const T *row = base + ((long)(z + PAD) * v.pny + (y0 + PAD)) * v.pnx + bx * B;
#pragma unroll 6
                for (int y = y0; y <= y1; ++y, row += v.pnx) {
#pragma unroll
                    for (int k = 0; k < B / 8; ++k) {
                        if (bx * B + k * 8 >= v.pnx) break;
                        V w[4];
                        const uint4 q = __ldg(reinterpret_cast<const uint4 *>(row) + k);
                        memcpy(w, &q, 16);
                        if (k == 0) {
#pragma unroll
                            for (int i = 0; i < 2; ++i) {
                                flo = X::least(flo, w[i]);
                                fhi = X::most(fhi, w[i]);
                            }
                            w[0] = X::skip_first(w[0]);
                        }
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            lo = X::least(lo, w[i]);
                            hi = X::most(hi, w[i]);
                        }
                    }
                    if (last) {
                        const uint2 q = __ldg(reinterpret_cast<const uint2 *>(row + B));
                        nlo = X::least(nlo, X::least(q.x, q.y));
                        nhi = X::most(nhi, X::most(q.x, q.y));
                    }
                }
            }
            const V dlo = __shfl_down_sync(0xffffffffu, flo, 1);
            const V dhi = __shfl_down_sync(0xffffffffu, fhi, 1);
            least = X::low(X::least(lo, (tx & 31) == 31 ? nlo : dlo));
            most = X::high(X::most(hi, (tx & 31) == 31 ? nhi : dhi));
        }
        s_lo[ty][tx] = least;
        s_hi[ty][tx] = most;
        __syncthreads();
        if (ty == 0 && bx < nbx) {
            T l = s_lo[0][tx], h = s_hi[0][tx];
#pragma unroll
            for (int k = 1; k < BM_TY; ++k) {
                l = tmin(l, s_lo[k][tx]);
                h = tmax(h, s_hi[k][tx]);
            }
            const long o = ((long)bz * nby + by) * nbx + bx;
            mn[o] = l;
            mx[o] = h;
        }
        __syncthreads();
    }
}

template <typename T>
void launch_minmax_t(const VolView &v, int B, const int nb[3], void *mn, void *mx,
                     cudaStream_t st) {
    const unsigned blocks = (unsigned)nb[1] * (unsigned)nb[2];
    const dim3 threads(BM_TX, BM_TY);
    if (B == 16)
        brick_minmax_kernel<T, 16><<<blocks, threads, 0, st>>>(v, nb[0], nb[1], nb[2], (T *)mn,
                                                                (T *)mx);
    else
        brick_minmax_kernel<T, 8><<<blocks, threads, 0, st>>>(v, nb[0], nb[1], nb[2], (T *)mn,
                                                               (T *)mx);
}

cudaError_t launch_brick_minmax(const VolView &v, int B, void *mn, void *mx, cudaStream_t st) {
    int nb[3];
    for (int k = 0; k < 3; ++k) nb[k] = (v.n[k] + B - 1) / B;
    switch (v.dtype) {
    case DT_U16: launch_minmax_t<uint16_t>(v, B, nb, mn, mx, st); break;
    case DT_I16: launch_minmax_t<int16_t>(v, B, nb, mn, mx, st); break;
    default: launch_minmax_t<float>(v, B, nb, mn, mx, st);
    }
    return cudaGetLastError();
}

// ------------------------------------------------------------------ occupancy ----------
template <typename T>
__device__ __forceinline__ float as_f32(T v) { return (float)v; }

// u(v) = (v - lo) * du in float32, clamped to [0, 255] (each operation rounded on its own).
__device__ __forceinline__ float u_index(float v, float lo, float du) {
    float u = __fmul_rn(__fsub_rn(v, lo), du);
    return fminf(fmaxf(u, 0.0f), 255.0f);
}

// prefix[k] = number of table entries i < k with opacity > 0 (257 ints).
template <typename T>
__global__ void occupancy_kernel(const T *__restrict__ mn, const T *__restrict__ mx, long n,
                                 const int *__restrict__ prefix, float lo, float du,
                                 uint8_t *__restrict__ occ) {
    __shared__ int pre[257];
    for (int i = threadIdx.x; i < 257; i += blockDim.x) pre[i] = prefix[i];
    __syncthreads();
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n;
         i += (long)gridDim.x * blockDim.x) {
        float ulo = u_index(as_f32(mn[i]), lo, du);
        float uhi = u_index(as_f32(mx[i]), lo, du);
        int k0 = max((int)floorf(ulo) - 1, 0);
        int k1 = min((int)ceilf(uhi) + 1, 255);
        occ[i] = (pre[k1 + 1] - pre[k0]) > 0 ? 1 : 0;
    }
}

cudaError_t launch_occupancy(const void *mn, const void *mx, int dtype, long nbricks,
                             const int *prefix_dev, float lo, float du, uint8_t *occ,
                             cudaStream_t st) {
    int threads = 256;
    long blocks = (nbricks + threads - 1) / threads;
    if (blocks > 152L * 16) blocks = 152L * 16;
    if (blocks < 1) blocks = 1;
    switch (dtype) {
    case DT_U16:
        occupancy_kernel<uint16_t><<<(unsigned)blocks, threads, 0, st>>>(
            (const uint16_t *)mn, (const uint16_t *)mx, nbricks, prefix_dev, lo, du, occ);
        break;
    case DT_I16:
        occupancy_kernel<int16_t><<<(unsigned)blocks, threads, 0, st>>>(
            (const int16_t *)mn, (const int16_t *)mx, nbricks, prefix_dev, lo, du, occ);
        break;
    default:
        occupancy_kernel<float><<<(unsigned)blocks, threads, 0, st>>>(
            (const float *)mn, (const float *)mx, nbricks, prefix_dev, lo, du, occ);
    }
    return cudaGetLastError();
}

// ------------------------------------------------------------- cell transparency mask ----
// Cell c (per axis c = -1 .. n-1, index c' = c + 1) holds the samples with floor(p) = c; their
// 64 cubic taps are voxels c-1 .. c+2, i.e. padded indices c' .. c'+3. The B-spline weights are
// non-negative and sum to one, so such a sample lies in [min, max] of the taps (up to float
// rounding, which the +-1 index margin covers). A cell is open when an entry of non-zero
// opacity lies in [floor(u(min)) - 1, ceil(u(max)) + 1] (the occupancy rule); a sample in a
// clear cell has opacity exactly zero. Layout of the mask: cell_open (vrc_internal.h).
//
// The rule is evaluated without a min/max: u is monotone in the value, so the range is the
// union of the taps' own index intervals [floor(u_i) - 1, ceil(u_i) + 1], and it holds no
// non-zero entry exactly when all those intervals lie in one run of zero-opacity entries.
// Each tap is therefore reduced to a byte, the id of the zero run holding its interval (0
// when none does), and a cell is clear exactly when its 64 bytes are equal and non-zero,
// i.e. when their bitwise OR equals their bitwise AND and is non-zero.
//
// Only cells of occupied bricks are worked out: a brick's [min, max] covers the taps of all its
// cells (the apron), so the cells of an empty brick are clear, by the same rule. The unit of
// work is a tile of 8^3 cells, 8t - 8 .. 8t - 1 per axis, which lies in one brick (tile 0 holds
// the cells -1). A warp looks at 4 tiles in a row along x and writes zeros for those whose brick is
// empty; the warps of a CTA share out the others, one at a time: the tile's 11 x 11 rows of 11 voxels are read
// with vector loads (8t - 8 is a 16-byte boundary of the padded row), reduced to run ids and
// ORed / ANDed along x in registers, the y and z windows are taken from shared memory, and the
// bits of a 4^3 block are gathered by a warp reduction.
// Bound: latency and issue of the occupied tiles (about 15 ALU operations a voxel). 512^2 x 400
// int16 with bone and vessels visible: 40 us (46 us with each warp working through its own tiles),
// against 240 us for two passes over the whole volume (run ids of every voxel to memory, then
// every cell's windows).
constexpr int CM_TILES = 4, CM_WARPS = 4;  // tiles a warp, warps a CTA
constexpr int CM_W = 11;  // voxels per axis that the cells of a tile read

// Table of the run id of a voxel's index interval: entry f for u = f exactly, entry 256 + f for
// u in (f, f + 1); zero when no single zero run holds the interval.
__device__ __forceinline__ void zero_run_table(const uint8_t *__restrict__ zrun, uint8_t *tab,
                                               int nthreads) {
    for (int i = threadIdx.x; i < 512; i += nthreads) {
        const int f = i & 255;
        const int k0 = max(f - 1, 0), k1 = min(f + 1 + (i >> 8), 255);
        tab[i] = zrun[k0] == zrun[k1] ? zrun[k0] : (uint8_t)0;
    }
}

__device__ __forceinline__ uint32_t zero_run_of(const uint8_t *tab, float v, float lo, float du) {
    const float u = u_index(v, lo, du);
    int f;
    const float fl = floor_small(u, f);
    return tab[f + (u > fl ? 256 : 0)];
}

// The run ids of padded elements x0 + 1 .. x0 + 11 of a row (x0 a multiple of 8), as bytes of
// w[0 .. 2]; elements outside the row (x0 = -8, and past its end) are read by no cell.
template <typename T>
__device__ __forceinline__ void run_id_row(const T *__restrict__ row, int x0, int pnx,
                                           const uint8_t *tab, float lo, float du,
                                           uint32_t w[3]) {
    T v[12] = {};
    if constexpr (sizeof(T) == 2) {
        if (x0 >= 0) {
            const uint4 a = __ldg((const uint4 *)(row + x0));
            memcpy(v, &a, 16);
        }
        if (x0 + 8 < pnx) {
            const uint2 b = __ldg((const uint2 *)(row + x0 + 8));
            memcpy(v + 8, &b, 8);
        }
    } else {
        if (x0 >= 0) {
            const float4 a = __ldg((const float4 *)(row + x0));
            const float4 b = __ldg((const float4 *)(row + x0) + 1);
            memcpy(v, &a, 16);
            memcpy(v + 4, &b, 16);
        }
        if (x0 + 8 < pnx) {
            const float4 c = __ldg((const float4 *)(row + x0 + 8));
            memcpy(v + 8, &c, 16);
        }
    }
    w[0] = w[1] = w[2] = 0u;
#pragma unroll
    for (int e = 0; e < CM_W; ++e)
        w[e >> 2] |= zero_run_of(tab, (float)v[e + 1], lo, du) << (8 * (e & 3));
}

// Bits of the bytes i of (o, a) whose cell is open: o != a or o == 0.
__device__ __forceinline__ uint32_t open_nibble(uint32_t o, uint32_t a) {
    auto nz = [](uint32_t v) { return (((v & 0x7f7f7f7fu) + 0x7f7f7f7fu) | v) & 0x80808080u; };
    const uint32_t m = (nz(o ^ a) | (nz(o) ^ 0x80808080u)) >> 7;
    return (m | (m >> 7) | (m >> 14) | (m >> 21)) & 0xfu;
}

template <typename T>
__global__ void __launch_bounds__(32 * CM_WARPS)
    cellmask_kernel(VolView v, const uint8_t *__restrict__ occ, int shift, int nbx, int nby,
                    const uint8_t *__restrict__ zrun, float lo, float du,
                    uint32_t *__restrict__ cells) {
    __shared__ uint8_t tab[512];
    __shared__ uint4 s_rows[CM_WARPS][CM_W * CM_W];
    __shared__ int s_tiles[CM_WARPS * CM_TILES], s_count;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint4 *rows = s_rows[warp];
    const int nfx = cell_blocks(v.n[0]), nfy = cell_blocks(v.n[1]), nfz = cell_blocks(v.n[2]);
    const int ntx = cell_tiles(v.n[0]), nty = cell_tiles(v.n[1]), ntz = cell_tiles(v.n[2]);
    const unsigned gx = (unsigned)(ntx + CM_TILES - 1) / CM_TILES;
    const unsigned unit = blockIdx.x * CM_WARPS + warp;
    const int t0 = (int)(unit % gx) * CM_TILES;
    int ty = (int)((unit / gx) % nty), tz = (int)(unit / (gx * nty));

    // the tiles with an occupied brick; zeros for the others (lane: row of blocks, tile)
    unsigned met = 0;
    if (tz < ntz) {
        const int tile = lane & 3, tx = t0 + tile;
        const int to_brick = shift - 3;
        bool any = false;
        if (tx < ntx)
            any = occ[((long)(max(tz - 1, 0) >> to_brick) * nby + (max(ty - 1, 0) >> to_brick)) *
                          nbx + (max(tx - 1, 0) >> to_brick)] != 0;
        met = __ballot_sync(0xffffffffu, any) & ((1u << CM_TILES) - 1u);
        const int by = 2 * ty - 1 + ((lane >> 2) & 1), bz = 2 * tz - 1 + ((lane >> 3) & 1);
        if (lane < 16 && tx < ntx && !any && (unsigned)by < (unsigned)nfy &&
            (unsigned)bz < (unsigned)nfz) {
            uint2 *o = (uint2 *)cells + ((long)bz * nfy + by) * nfx + 2 * tx;
            if (tx > 0) o[-1] = make_uint2(0u, 0u);
            if (2 * tx < nfx) o[0] = make_uint2(0u, 0u);
        }
    }
    // the tiles of all the CTA's warps in one list, which they share out
    if (threadIdx.x == 0) s_count = 0;
    if (!__syncthreads_or(met != 0)) return;
    if (lane < CM_TILES && ((met >> lane) & 1u))
        s_tiles[atomicAdd(&s_count, 1)] = (tz * nty + ty) * ntx + t0 + lane;
    zero_run_table(zrun, tab, 32 * CM_WARPS);
    __syncthreads();
    const T *base = (const T *)v.base;
    for (int k = warp; k < s_count; k += CM_WARPS) {
        const int tile = s_tiles[k], tx = tile % ntx;
        ty = (tile / ntx) % nty;
        tz = tile / (ntx * nty);
        __syncwarp();  // the rows of the tile before have been read
        for (int r = lane; r < CM_W * CM_W; r += 32) {
            const int y = min(max(8 * ty - 7 + r % CM_W, 0), v.pny - 1);
            const int z = min(max(8 * tz - 7 + r / CM_W, 0), v.pnz - 1);
            uint32_t w[3];
            run_id_row<T>(base + ((long)z * v.pny + y) * v.pnx, 8 * tx - 8, v.pnx, tab, lo, du, w);
            // byte i of o / a: OR / AND over the columns i .. i+3 of cell i
            uint32_t o[2], a[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t w1 = __funnelshift_r(w[h], w[h + 1], 8);
                const uint32_t w2 = __funnelshift_r(w[h], w[h + 1], 16);
                const uint32_t w3 = __funnelshift_r(w[h], w[h + 1], 24);
                o[h] = (w[h] | w1) | (w2 | w3);
                a[h] = (w[h] & w1) & (w2 & w3);
            }
            rows[r] = make_uint4(o[0], o[1], a[0], a[1]);
        }
        __syncwarp();
        const int y = lane & 7, cy = 8 * ty - 8 + y;
        const int cx = 8 * tx - 8;
        // cells of the tile inside the volume, -1 .. n-1, as bits
        const unsigned inx = (tx == 0 ? 0x80u : 0xffu) & ((2u << min(v.n[0] - 1 - cx, 7)) - 1u);
#pragma unroll
        for (int h = 0; h < 2; ++h) {  // cells of the lower, then the upper 4^3 blocks in z
            const int z = 4 * h + (lane >> 3), cz = 8 * tz - 8 + z;
            uint32_t o0 = 0u, o1 = 0u, a0 = 0xffffffffu, a1 = 0xffffffffu;
#pragma unroll
            for (int dz = 0; dz < 4; ++dz) {
#pragma unroll
                for (int dy = 0; dy < 4; ++dy) {
                    const uint4 q = rows[(z + dz) * CM_W + y + dy];
                    o0 |= q.x;
                    o1 |= q.y;
                    a0 &= q.z;
                    a1 &= q.w;
                }
            }
            const bool yz = cy >= -1 && cy < v.n[1] && cz >= -1 && cz < v.n[2];
            const uint32_t n0 = yz ? open_nibble(o0, a0) & inx : 0u;
            const uint32_t n1 = yz ? open_nibble(o1, a1) & (inx >> 4) : 0u;
            // one 32-bit half block per 8 lanes: 4 rows y x 2 slices z
            const unsigned mask = 0x0f0fu << (4 * ((lane >> 2) & 1) + 16 * (lane >> 4));
            const int sh = 16 * ((lane >> 3) & 1) + 4 * (lane & 3);
            const uint32_t w0 = __reduce_or_sync(mask, n0 << sh);
            const uint32_t w1 = __reduce_or_sync(mask, n1 << sh);
            const int by = 2 * ty - 1 + ((lane >> 2) & 1), bz = 2 * tz - 1 + h;
            if ((lane & 11) == 0 && (unsigned)by < (unsigned)nfy && (unsigned)bz < (unsigned)nfz) {
                uint32_t *out = cells + 2 * (((long)bz * nfy + by) * nfx + 2 * tx) + (lane >> 4);
                if (tx > 0) out[-2] = w0;
                if (2 * tx < nfx) out[0] = w1;
            }
        }
    }
}

size_t cellmask_bytes(const int n[3]) {
    return 8 * (size_t)cell_blocks(n[0]) * cell_blocks(n[1]) * cell_blocks(n[2]);
}

cudaError_t launch_cellmask(const VolView &v, int B, const int nb[3], const uint8_t *occ,
                            const uint8_t *zrun_dev, float lo, float du, uint32_t *cells,
                            cudaStream_t st) {
    const long units = (long)((cell_tiles(v.n[0]) + CM_TILES - 1) / CM_TILES) *
                       cell_tiles(v.n[1]) * cell_tiles(v.n[2]);
    const unsigned blocks = (unsigned)((units + CM_WARPS - 1) / CM_WARPS);
    const int shift = B == 16 ? 4 : 3;
    switch (v.dtype) {
    case DT_U16:
        cellmask_kernel<uint16_t><<<blocks, 32 * CM_WARPS, 0, st>>>(v, occ, shift, nb[0], nb[1],
                                                                    zrun_dev, lo, du, cells);
        break;
    case DT_I16:
        cellmask_kernel<int16_t><<<blocks, 32 * CM_WARPS, 0, st>>>(v, occ, shift, nb[0], nb[1],
                                                                   zrun_dev, lo, du, cells);
        break;
    default:
        cellmask_kernel<float><<<blocks, 32 * CM_WARPS, 0, st>>>(v, occ, shift, nb[0], nb[1],
                                                                 zrun_dev, lo, du, cells);
    }
    return cudaGetLastError();
}

// One thread per tile: the cells 8t .. 8t + 7 are the blocks 2t + 1 and 2t + 2 (cell_open), those
// of tile 0 and the cell -1 the blocks 0 .. 2.
__global__ void __launch_bounds__(256) tile_occupancy_kernel(const uint2 *__restrict__ cells,
                                                             int nfx, int nfy, int nfz, int ntx,
                                                             int nty, int ntz,
                                                             uint8_t *__restrict__ tiles) {
    const long i = (long)blockIdx.x * 256 + threadIdx.x;
    if (i >= (long)ntx * nty * ntz) return;
    const int tx = (int)(i % ntx), ty = (int)((i / ntx) % nty), tz = (int)(i / ((long)ntx * nty));
    uint32_t any = 0u;
    for (int z = tz ? 2 * tz + 1 : 0; z < min(2 * tz + 3, nfz); ++z)
        for (int y = ty ? 2 * ty + 1 : 0; y < min(2 * ty + 3, nfy); ++y)
            for (int x = tx ? 2 * tx + 1 : 0; x < min(2 * tx + 3, nfx); ++x) {
                const uint2 w = __ldg(cells + ((long)z * nfy + y) * nfx + x);
                any |= w.x | w.y;
            }
    tiles[i] = any ? 1 : 0;
}

cudaError_t launch_tile_occupancy(const uint32_t *cells, const int n[3], const int nt[3],
                                  uint8_t *tiles, cudaStream_t st) {
    const long count = (long)nt[0] * nt[1] * nt[2];
    tile_occupancy_kernel<<<(unsigned)((count + 255) / 256), 256, 0, st>>>(
        (const uint2 *)cells, cell_blocks(n[0]), cell_blocks(n[1]), cell_blocks(n[2]), nt[0],
        nt[1], nt[2], tiles);
    return cudaGetLastError();
}

// The mask as rows of 32 cells along x (vrc_cellmask_get): word (c'_z (ny + 1) + c'_y) cwx +
// c'_x / 32, bit c'_x % 32, c' = c + 1. One thread per word.
__global__ void cellmask_rows_kernel(const uint32_t *__restrict__ cells, int nx, int ny, int nz,
                                     int cwx, uint32_t *__restrict__ out) {
    const long total = (long)cwx * (ny + 1) * (nz + 1);
    const int nfx = cell_blocks(nx), nfy = cell_blocks(ny);
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < total;
         i += (long)gridDim.x * blockDim.x) {
        const int wx = (int)(i % cwx), y = (int)((i / cwx) % (ny + 1)) + 3;
        const int z = (int)(i / ((long)cwx * (ny + 1))) + 3;
        // cells c' = 32 wx .. + 31 are bits 3 .. 34 of the 9 nibbles from block 8 wx
        const uint32_t *row = cells + 2 * (((long)(z >> 2) * nfy + (y >> 2)) * nfx) + ((z >> 1) & 1);
        unsigned long long w = 0ull;
        for (int k = 0; k < 9 && 8 * wx + k < nfx; ++k)
            w |= (unsigned long long)((row[2 * (8 * wx + k)] >> (16 * (z & 1) + 4 * (y & 3))) & 0xfu)
                 << (4 * k);
        out[i] = (uint32_t)(w >> 3);
    }
}

long cellmask_row_words(const int n[3]) {
    return (long)((n[0] + 1 + 31) / 32) * (n[1] + 1) * (n[2] + 1);
}

cudaError_t launch_cellmask_rows(const uint32_t *cells, const int n[3], uint32_t *out,
                                 cudaStream_t st) {
    const long words = cellmask_row_words(n);
    const long blocks = (words + 255) / 256;
    cellmask_rows_kernel<<<(unsigned)(blocks > 152L * 32 ? 152L * 32 : blocks), 256, 0, st>>>(
        cells, n[0], n[1], n[2], (n[0] + 1 + 31) / 32, out);
    return cudaGetLastError();
}

// ---------------------------------------------------------- pre-integration table ------
// Entry (i, k) for slabs of length ds: the table composited along the linear ramp of the index
// from i (front sample) to k (back sample) by PREINT_K equal sub-steps (midpoint rule, each
// with the opacity correction alpha = 1 - (1 - a)^(ds / PREINT_K)); (associated rgb, opacity).
// Computed in double (65536 entries, 32 sub-steps: negligible), stored as float4.
__global__ void preint_table_kernel(const float4 *__restrict__ tf_tab, float ds,
                                    float4 *__restrict__ tab) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= 256 * 256) return;
    const int i = e >> 8, k = e & 255;
    double c0 = 0.0, c1 = 0.0, c2 = 0.0, T = 1.0;
    const double amax = 1.0 - 5.9604644775390625e-08;
    for (int n = 0; n < PREINT_K; ++n) {
        const double u = i + (k - i) * (n + 0.5) / PREINT_K;
        int i0 = (int)floor(u);
        i0 = i0 > 254 ? 254 : i0;
        const double f = u - i0;
        const float4 a = tf_tab[2 * i0], b = tf_tab[2 * i0 + 2];
        const double r = (1.0 - f) * a.x + f * b.x, g = (1.0 - f) * a.y + f * b.y;
        const double bl = (1.0 - f) * a.z + f * b.z;
        double al = (1.0 - f) * a.w + f * b.w;
        al = al < 0.0 ? 0.0 : (al > amax ? amax : al);
        const double alpha = -expm1((double)ds / PREINT_K * log1p(-al));
        c0 += T * alpha * r;
        c1 += T * alpha * g;
        c2 += T * alpha * bl;
        T *= 1.0 - alpha;
    }
    tab[e] = make_float4((float)c0, (float)c1, (float)c2, (float)(1.0 - T));
}

cudaError_t launch_preint_table(const float4 *tf_tab, float ds, float4 *tab, cudaStream_t st) {
    preint_table_kernel<<<256, 256, 0, st>>>(tf_tab, ds, tab);
    return cudaGetLastError();
}

// ------------------------------------------------------- empty-box distance (leaping) ----
// For each of the 8 direction octants s = (sx, sy, sz) in {+1, -1}^3 and each brick b:
// dist[oct][b] = 0 for an occupied brick, else the smallest r >= 1 such that the forward box
// of bricks {b + t : t_k between 0 and r s_k} holds an occupied brick (capped at 255). Every
// brick of the forward box of extent r - 1 is empty, so a ray whose direction lies in that
// octant may leap from b to the exit of that box. Octant index = (sx < 0) | (sy < 0) << 1 |
// (sz < 0) << 2.
//
// That is the distance to the nearest occupied brick ahead in the maximum norm, which separates
// by axis: with g the distances along x alone, f(y) = min over d >= 0 of max(d, g(y + d sy)),
// and the same again along z. Pass x finds the next set bit of the row's occupancy bits (2
// fields), passes y and z search forward until d reaches the best value (4, then 8 fields); a
// step reads consecutive bytes across a warp. Latency-bound (a field of 64 x 64 x 50 bricks is
// 0.2 MB): 28 us for the three passes, against 108 us for a summed-volume table by serial
// prefix sums and a binary search per brick and octant.
constexpr int DX_WARPS = 4;

// One warp per row (y, z) of bricks, 32 at a time, once in each direction.
__global__ void __launch_bounds__(32 * DX_WARPS) dist_x_kernel(const uint8_t *__restrict__ occ,
                                                               int nbx, long rows,
                                                               uint8_t *__restrict__ out) {
    const int lane = threadIdx.x & 31;
    const long row = (long)blockIdx.x * DX_WARPS + (threadIdx.x >> 5);
    if (row >= rows) return;
    const uint8_t *o = occ + row * nbx;
    uint8_t *fwd = out + row * nbx, *bwd = fwd + rows * nbx;
    // carry: distance from the last brick handled to the nearest occupied one at or before it
    int carry = 255;
    for (int x0 = 0; x0 < nbx; x0 += 32) {
        const int x = x0 + lane;
        const unsigned bits = __ballot_sync(0xffffffffu, x < nbx && o[x] != 0);
        const unsigned at = bits & (0xffffffffu >> (31 - lane));  // bricks x0 .. x
        const int d = at ? lane - (31 - __clz(at)) : min(carry + lane + 1, 255);
        if (x < nbx) bwd[x] = (uint8_t)d;
        carry = __shfl_sync(0xffffffffu, d, 31);
    }
    carry = 255;
    for (int x0 = (nbx - 1) & ~31; x0 >= 0; x0 -= 32) {
        const int x = x0 + lane;
        const unsigned bits = __ballot_sync(0xffffffffu, x < nbx && o[x] != 0);
        const unsigned at = bits & (0xffffffffu << lane);  // bricks x .. x0 + 31
        // past the row's end there is nothing: a full carry
        const int d = at ? __ffs(at) - 1 - lane : min(carry + 32 - lane, 255);
        if (x < nbx) fwd[x] = (uint8_t)d;
        carry = __shfl_sync(0xffffffffu, d, 0);
    }
}

// Pass along an axis of `len` bricks spaced `stride` apart, one field per blockIdx.y: fields NIN
// in, 2 NIN out, field f + NIN h from field f searching towards +(h = 0) or -(h = 1).
template <int NIN>
__global__ void __launch_bounds__(256) dist_axis_kernel(const uint8_t *__restrict__ in, unsigned n,
                                                        unsigned len, unsigned stride,
                                                        uint8_t *__restrict__ out) {
    const int h = blockIdx.y / NIN;
    const uint8_t *f = in + (size_t)(blockIdx.y % NIN) * n;
    uint8_t *o = out + (size_t)blockIdx.y * n;
    const int s = h ? -(int)stride : (int)stride;
    for (unsigned i = blockIdx.x * 256u + threadIdx.x; i < n; i += gridDim.x * 256u) {
        const uint8_t *p = f + i;
        const int pos = (int)((i / stride) % len);
        const int room = h ? pos : (int)len - 1 - pos;  // bricks ahead
        int best = p[0];
        for (int d = 1; d < best && d <= room; d += 4) {
            int g[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) g[k] = p[(long)min(d + k, room) * s];
#pragma unroll
            for (int k = 0; k < 4; ++k) best = min(best, max(d + k, g[k]));
        }
        o[i] = (uint8_t)best;
    }
}

// The same for rows of a multiple of 4 bricks, 4 bricks of a row a thread, as the byte pairs (0,
// 2) and (1, 3) in 16-bit halves.
template <int NIN>
__global__ void __launch_bounds__(256) dist_axis4_kernel(const uint32_t *__restrict__ in,
                                                         unsigned n4, unsigned len,
                                                         unsigned stride4,
                                                         uint32_t *__restrict__ out) {
    constexpr int U = 8;  // loads in flight
    const int h = blockIdx.y / NIN;
    const uint32_t *f = in + (size_t)(blockIdx.y % NIN) * n4;
    uint32_t *o = out + (size_t)blockIdx.y * n4;
    const int s = h ? -(int)stride4 : (int)stride4;
    for (unsigned i = blockIdx.x * 256u + threadIdx.x; i < n4; i += gridDim.x * 256u) {
        const uint32_t *p = f + i;
        const int pos = (int)((i / stride4) % len);
        const int room = h ? pos : (int)len - 1 - pos;
        const uint32_t w = p[0];
        uint32_t b0 = w & 0x00ff00ffu, b1 = (w >> 8) & 0x00ff00ffu;
        for (int d = 1; d <= room; d += U) {
            const uint32_t m = max2<uint16_t>(b0, b1);
            if ((int)max(m & 0xffffu, m >> 16) <= d) break;
            uint32_t g[U];
#pragma unroll
            for (int k = 0; k < U; ++k) g[k] = p[(long)min(d + k, room) * s];
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const uint32_t dd = (uint32_t)(d + k) * 0x10001u;
                b0 = min2<uint16_t>(b0, max2<uint16_t>(dd, g[k] & 0x00ff00ffu));
                b1 = min2<uint16_t>(b1, max2<uint16_t>(dd, (g[k] >> 8) & 0x00ff00ffu));
            }
        }
        o[i] = b0 | (b1 << 8);
    }
}

size_t box_dist_scratch_bytes(const int nb[3]) { return 4 * (size_t)nb[0] * nb[1] * nb[2]; }

// The x fields go through the first quarter of `dist`, the y fields (4 bytes a brick) through
// `scratch`.
cudaError_t launch_box_dist(const uint8_t *occ, const int nb[3], uint8_t *scratch, uint8_t *dist,
                             cudaStream_t st) {
    const long n = (long)nb[0] * nb[1] * nb[2], rows = (long)nb[1] * nb[2];
    uint8_t *yf = scratch;
    dist_x_kernel<<<(unsigned)((rows + DX_WARPS - 1) / DX_WARPS), 32 * DX_WARPS, 0, st>>>(
        occ, nb[0], rows, dist);
    auto blocks = [](long k) { return (unsigned)((k + 255) / 256 > 152L * 64 ? 152L * 64
                                                                             : (k + 255) / 256); };
    if (nb[0] % 4 == 0) {
        const unsigned n4 = (unsigned)(n / 4), sy = nb[0] / 4, sz = sy * nb[1];
        dist_axis4_kernel<2><<<dim3(blocks(n4), 4), 256, 0, st>>>((const uint32_t *)dist, n4, nb[1],
                                                                  sy, (uint32_t *)yf);
        dist_axis4_kernel<4><<<dim3(blocks(n4), 8), 256, 0, st>>>((const uint32_t *)yf, n4, nb[2],
                                                                  sz, (uint32_t *)dist);
        return cudaGetLastError();
    }
    dist_axis_kernel<2><<<dim3(blocks(n), 4), 256, 0, st>>>(dist, (unsigned)n, nb[1], nb[0], yf);
    dist_axis_kernel<4><<<dim3(blocks(n), 8), 256, 0, st>>>(yf, (unsigned)n, nb[2], nb[0] * nb[1],
                                                            dist);
    return cudaGetLastError();
}

}  // namespace vrc
