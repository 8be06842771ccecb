// mi_hard.cu -- hard-binned mutual information on sm_103a.
//
// Per transform T and fixed voxel i: the 16.16 moving index U = A i + b
// (exact integers), the overlap test, an 8-neighbour integer trilinear
// resample of the moving volume, the moving bin, and one increment of the
// joint histogram h[fixed bin][moving bin] (the paper's full, all-voxel
// histogram, Discussion).  The entropies of Eq. (1) and the MI of Eq. (2)
// (and Tsallis entropies for every q from the same histogram) are reduced in
// FP64 from the exact counts.
//
// Kernels:
//   k_bin_fixed       fixed volume -> uint8 bins, once per context
//   k_batched<...>    persistent CTAs pull work items from an atomic ticket.  An
//                     item is a whole (pair, transform), whose histogram one CTA
//                     builds in shared memory and reduces in place, or one of
//                     several interleaved parts of it, whose histogram is added
//                     to the transform's slot in global memory
//   k_entropy_slots   reduces the slots' histograms, several CTAs per slot
//   k_resample        v(T(x)) on the fixed grid
//
// Row clipping: along a fixed row (j, k) the moving index is linear in i, so
// the overlap is one interval [lo, hi] of i, found per row (float estimate,
// then exact 64-bit checks).  Inside it every U_a lies in [0, (n_a-1) 2^16],
// so the per-voxel arithmetic is exact in 32 bits.
#include <cuda_runtime.h>
#include <math.h>
#include <stddef.h>
#include <stdint.h>

#include "mi_internal.h"

namespace mi {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr uint32_t kEmptyKey = 0xffffffffu;

// ---------------------------------------------------------------------------
// Small kernels run once per context
// ---------------------------------------------------------------------------

__global__ void k_f32_to_u16(const float *__restrict__ in, long long n, uint16_t *__restrict__ out) {
    for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < n; x += (long long)gridDim.x * blockDim.x) {
        double v = (double)in[x];
        if (!(v == v)) v = 0.0;
        double s = rint(v * 65535.0);  // round half to even
        s = s < 0.0 ? 0.0 : (s > 65535.0 ? 65535.0 : s);
        out[x] = (uint16_t)s;
    }
}

// Eight elements of a volume, loaded and stored at once where both are aligned to it.
template <typename T>
struct alignas(8 * sizeof(T)) Eight {
    T v[8];
};

template <typename T>
bool aligned8(const void *p) {
    return (uintptr_t)p % (8 * sizeof(T)) == 0;
}

template <typename T>
__global__ void k_copy_clamp(const T *__restrict__ in, long long n, uint32_t vmax, bool vec, T *__restrict__ out) {
    const long long first = blockIdx.x * (long long)blockDim.x + threadIdx.x, step = (long long)gridDim.x * blockDim.x;
    const long long groups = vec ? n / 8 : 0;
    for (long long g = first; g < groups; g += step) {
        Eight<T> e = ((const Eight<T> *)in)[g];
#pragma unroll
        for (int k = 0; k < 8; ++k) e.v[k] = (T)min((uint32_t)e.v[k], vmax);
        ((Eight<T> *)out)[g] = e;
    }
    for (long long x = 8 * groups + first; x < n; x += step) out[x] = (T)min((uint32_t)in[x], vmax);
}

// bin(v) = (min(v, 2^d - 1) * bins) >> d, and the voxels per bin (in shared memory, then one addition per
// CTA and bin).
template <typename T>
__global__ void __launch_bounds__(256)
    k_bin_fixed(const T *__restrict__ in, long long n, int depth, int bins, bool vec, uint8_t *__restrict__ out,
                unsigned long long *__restrict__ counts) {
    __shared__ unsigned int h[4][256];  // a copy per two warps
    for (int c = threadIdx.x; c < 4 * 256; c += blockDim.x) (&h[0][0])[c] = 0;
    __syncthreads();
    unsigned int *mine = h[threadIdx.x >> 6];
    const uint32_t vmax = (uint32_t)((1ull << depth) - 1ull);
    auto bin = [&](uint32_t v) {
        const uint32_t b = (min(v, vmax) * (uint32_t)bins) >> depth;  // at most 65535 x 256
        atomicAdd(&mine[b], 1u);
        return (uint8_t)b;
    };
    const long long first = blockIdx.x * (long long)blockDim.x + threadIdx.x, step = (long long)gridDim.x * blockDim.x;
    const long long groups = vec ? n / 8 : 0;
    for (long long g = first; g < groups; g += step) {
        const Eight<T> e = ((const Eight<T> *)in)[g];
        Eight<uint8_t> o;
#pragma unroll
        for (int k = 0; k < 8; ++k) o.v[k] = bin(e.v[k]);
        ((Eight<uint8_t> *)out)[g] = o;
    }
    for (long long x = 8 * groups + first; x < n; x += step) out[x] = bin(in[x]);
    __syncthreads();
    for (int c = threadIdx.x; c < bins; c += blockDim.x) {
        const unsigned int v = h[0][c] + h[1][c] + h[2][c] + h[3][c];
        if (v) atomicAdd(counts + c, (unsigned long long)v);
    }
}

// tab[c] = c ln c (q == 1) or c^q, FP64, c < kTab; tab[0] = 0.
__global__ void k_table(double *__restrict__ tab, float qf) {
    const double q = (double)qf;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < kTab; c += gridDim.x * blockDim.x) {
        double d = (double)c;
        tab[c] = c == 0 ? 0.0 : (qf == 1.0f ? d * log(d) : pow(d, q));
    }
}

// ---------------------------------------------------------------------------
// Per-voxel sampling
// ---------------------------------------------------------------------------

// Stage lerp with an 8-bit weight: (a (256 - f) + b f + 128) >> 8 written as
// a + floor(((b - a) f + 128) / 256), identical for integers (arithmetic shift).
__device__ __forceinline__ int lerp8(int a, int b, int f) { return a + (((b - a) * f + 128) >> 8); }

template <typename MovT>
__device__ __forceinline__ int sample_hard(const MovT *__restrict__ mov, int n0, int n1, int n2, int ux, int uy,
                                           int uz) {
    const int ix = ux >> 16, iy = uy >> 16, iz = uz >> 16;
    const int fx = (ux >> 8) & 255, fy = (uy >> 8) & 255, fz = (uz >> 8) & 255;
    // the upper neighbour is clamped on the last plane, where its weight is 0
    const int sx = ix < n0 - 1 ? 1 : 0;
    const int sy = iy < n1 - 1 ? n0 : 0;
    const int sz = iz < n2 - 1 ? n0 * n1 : 0;
    const MovT *p = mov + (ix + n0 * (iy + n1 * iz));
    const int v000 = __ldg(p), v001 = __ldg(p + sx), v010 = __ldg(p + sy), v011 = __ldg(p + sy + sx);
    const int v100 = __ldg(p + sz), v101 = __ldg(p + sz + sx), v110 = __ldg(p + sz + sy),
              v111 = __ldg(p + sz + sy + sx);
    const int e00 = lerp8(v000, v001, fx), e01 = lerp8(v010, v011, fx);
    const int e10 = lerp8(v100, v101, fx), e11 = lerp8(v110, v111, fx);
    const int g0 = lerp8(e00, e01, fy), g1 = lerp8(e10, e11, fy);
    return lerp8(g0, g1, fz);
}

// The same resample from the padded x-paired moving volume: element (x, y, z)
// holds v[x] in its low half and v[min(x + 1, n0 - 1)] in its high half
// (uint16 pairs of a uint8 volume, uint32 pairs of a uint16 volume), and the
// volume carries one extra y row and one extra z plane repeating the last
// ones, so the three neighbour offsets are constants (n0, n0 (n1 + 1)) and a
// voxel takes 4 loads.  On the last plane of an axis the weight of the upper
// neighbour is 0, so the repeated values change nothing.
// Each stage lerp is (a (256 - f) + b f + 128) >> 8.
__device__ __forceinline__ int lerp8g(int a, int b, int f, int g) { return (a * g + b * f + 128) >> 8; }

template <typename PairT>
__device__ __forceinline__ int sample_hard_pair(const PairT *__restrict__ movp, int sy, int sz, int n0, int n01p,
                                                int ux, int uy, int uz) {
    constexpr int HB = (int)sizeof(PairT) * 4;  // bits per half
    constexpr uint32_t LO = (1u << HB) - 1u;
    const int fx = (int)__byte_perm((unsigned)ux, 0u, 0x4441), fy = (int)__byte_perm((unsigned)uy, 0u, 0x4441),
              fz = (int)__byte_perm((unsigned)uz, 0u, 0x4441);
    const int gx = 256 - fx, gy = 256 - fy, gz = 256 - fz;
    const int idx = (ux >> 16) + n0 * (uy >> 16) + n01p * (uz >> 16);
    const PairT *p = movp + idx;
    const uint32_t a = __ldg(p), b = __ldg(p + sy), c = __ldg(p + sz), d = __ldg(p + sz + sy);
    const int e00 = lerp8g((int)(a & LO), (int)(a >> HB), fx, gx), e01 = lerp8g((int)(b & LO), (int)(b >> HB), fx, gx);
    const int e10 = lerp8g((int)(c & LO), (int)(c >> HB), fx, gx), e11 = lerp8g((int)(d & LO), (int)(d >> HB), fx, gx);
    const int g0 = lerp8g(e00, e01, fy, gy), g1 = lerp8g(e10, e11, fy, gy);
    return lerp8g(g0, g1, fz, gz);
}

// The same resample with the four x-pairs fetched through the texture path
// from a 3D array of pairs (block-linear layout, point sampling at texel
// centres, clamped addressing: exact integer texels).
template <typename PairT>
__device__ __forceinline__ int sample_hard_tex(unsigned long long tex, int ux, int uy, int uz) {
    constexpr int HB = (int)sizeof(PairT) * 4;
    constexpr uint32_t LO = (1u << HB) - 1u;
    const int fx = (int)__byte_perm((unsigned)ux, 0u, 0x4441), fy = (int)__byte_perm((unsigned)uy, 0u, 0x4441),
              fz = (int)__byte_perm((unsigned)uz, 0u, 0x4441);
    const int gx = 256 - fx, gy = 256 - fy, gz = 256 - fz;
    const float x = (float)(ux >> 16) + 0.5f, y = (float)(uy >> 16) + 0.5f, z = (float)(uz >> 16) + 0.5f;
    const uint32_t a = tex3D<PairT>(tex, x, y, z), b = tex3D<PairT>(tex, x, y + 1.0f, z);
    const uint32_t c = tex3D<PairT>(tex, x, y, z + 1.0f), d = tex3D<PairT>(tex, x, y + 1.0f, z + 1.0f);
    const int e00 = lerp8g((int)(a & LO), (int)(a >> HB), fx, gx), e01 = lerp8g((int)(b & LO), (int)(b >> HB), fx, gx);
    const int e10 = lerp8g((int)(c & LO), (int)(c >> HB), fx, gx), e11 = lerp8g((int)(d & LO), (int)(d >> HB), fx, gx);
    const int g0 = lerp8g(e00, e01, fy, gy), g1 = lerp8g(e10, e11, fy, gy);
    return lerp8g(g0, g1, fz, gz);
}

// The same resample from 2 x 2 (y, z) quads through the texture path.  A fetch
// at integer texel coordinates (ix, iy, iz) returns v(ix, iy, iz),
// v(ix, iy + 1, iz), v(ix, iy, iz + 1), v(ix, iy + 1, iz + 1) in four
// registers, already unpacked, so a voxel takes two fetches (columns ix and
// ix + 1).  Column ix + 1 lies past the volume only when ix = nx - 1, which
// inside the overlap means a fraction of 0: the clamped texel's weight is 0.
// Neighbouring lanes of a warp step along x, so the column one lane fetches
// second is, under most transforms, the one the next lane fetches first: the
// two requests of a warp step touch about one texel per voxel, and each texel
// is wanted within one step (with (x, y) quads each texel is also wanted as
// the upper plane of the next fixed slice, long after the L1 has evicted it).
__device__ __forceinline__ void tex_quad(unsigned long long tex, int x, int y, int z, uint32_t &a, uint32_t &b,
                                         uint32_t &c, uint32_t &d) {
    asm("tex.3d.v4.u32.s32 {%0, %1, %2, %3}, [%4, {%5, %6, %7, %7}];"
        : "=r"(a), "=r"(b), "=r"(c), "=r"(d)
        : "l"(tex), "r"(x), "r"(y), "r"(z));
}

// The 8 neighbours of the sample at 16.16 index (ux, uy, uz) in quad_lerp's order: t[0..3] =
// (x, y), (x + 1, y), (x, y + 1), (x + 1, y + 1) of plane iz, t[4..7] the same of plane iz + 1.
__device__ __forceinline__ void quad_fetch(unsigned long long tex, unsigned ux, unsigned uy, unsigned uz,
                                           uint32_t (&t)[8]) {
    const int ix = (int)(ux >> 16), iy = (int)(uy >> 16), iz = (int)(uz >> 16);
    tex_quad(tex, ix, iy, iz, t[0], t[2], t[4], t[6]);
    tex_quad(tex, ix + 1, iy, iz, t[1], t[3], t[5], t[7]);
}

// Trilinear value from the 8 neighbours: x, then y, then z stages.
__device__ __forceinline__ int quad_lerp(unsigned ux, unsigned uy, unsigned uz, const uint32_t (&t)[8]) {
    const int fx = (int)__byte_perm(ux, 0u, 0x4441), fy = (int)__byte_perm(uy, 0u, 0x4441),
              fz = (int)__byte_perm(uz, 0u, 0x4441);
    const int gx = 256 - fx, gy = 256 - fy, gz = 256 - fz;
    const int e00 = lerp8g((int)t[0], (int)t[1], fx, gx), e01 = lerp8g((int)t[2], (int)t[3], fx, gx);
    const int e10 = lerp8g((int)t[4], (int)t[5], fx, gx), e11 = lerp8g((int)t[6], (int)t[7], fx, gx);
    const int g0 = lerp8g(e00, e01, fy, gy), g1 = lerp8g(e10, e11, fy, gy);
    return lerp8g(g0, g1, fz, gz);
}

// The 8 neighbours of the sample at 16.16 index (ux, uy, uz) in one gather from the z-pair atlas:
// the float coordinates ix + 1 + ox, iy + 1 + oy (exact integers, so the gather's 2 x 2 footprint
// starts at texel (ix, iy) of plane iz's tile) are formed from the bit pattern 2^23 + ix plus the
// plane's stored offset ox + 1 - 2^23.  The gather returns (ix, iy + 1), (ix + 1, iy + 1),
// (ix + 1, iy), (ix, iy), each holding v(x, y, z) in bits 0..11 and v(x, y, z + 1) in bits 20..31
// (moving depth <= 12); unpacked, the eight values take quad_lerp's stages.  (Lerping both planes at
// once in 20-bit fields of 64-bit products took fewer instructions but measured 6 % slower.)  On the
// last plane of an axis the upper neighbour's weight is 0, so the texel beyond the tile edge (the next
// tile, or a clamped one) changes nothing.
__device__ __forceinline__ int gather_value(unsigned long long tex, const float2 *zoff, unsigned ux, unsigned uy,
                                            unsigned uz) {
    const float2 o = zoff[uz >> 16];
    const float u = __int_as_float((int)__funnelshift_r(ux, 0x4B00u, 16)) + o.x;
    const float v = __int_as_float((int)__funnelshift_r(uy, 0x4B00u, 16)) + o.y;
    const uint4 t = tex2Dgather<uint4>((cudaTextureObject_t)tex, u, v, 0);
    const uint32_t n[8] = {t.w & 0xFFFu, t.z & 0xFFFu, t.x & 0xFFFu, t.y & 0xFFFu,
                           t.w >> 20, t.z >> 20, t.x >> 20, t.y >> 20};
    return quad_lerp(ux, uy, uz, n);
}

// The stage lerps of an 8-bit volume, two at a time: a value times a weight takes 16 bits (255 x 256 + 128),
// so the planes z and z + 1 share a register in the x and y stages, low and high half.  x0 and x1: the pair
// at columns x and x + 1, of rows y and y + 1.  400 transforms of a 192 x 192 x 128 byte pair at 64 bins, four
// rows a step: 3106 -> 3028 us through quads, 256^3 at 256 bins 11.3 -> 11.1 ms (14.5 -> 12.9 through gathers).
__device__ __forceinline__ int pair_lerp(unsigned ux, unsigned uy, unsigned uz, const uint32_t (&x0)[2],
                                         const uint32_t (&x1)[2]) {
    const uint32_t fx = __byte_perm(ux, 0u, 0x4441), fy = __byte_perm(uy, 0u, 0x4441), fz = __byte_perm(uz, 0u, 0x4441);
    const uint32_t gx = 256u - fx, gy = 256u - fy, gz = 256u - fz;
    constexpr uint32_t half = 0x00800080u;
    const uint32_t e0 = __byte_perm(x0[0] * gx + x1[0] * fx + half, 0u, 0x4341);
    const uint32_t e1 = __byte_perm(x0[1] * gx + x1[1] * fx + half, 0u, 0x4341);
    const uint32_t g = e0 * gy + e1 * fy + half;
    return (int)((__byte_perm(g, 0u, 0x4441) * gz + (g >> 24) * fz + 128u) >> 8);
}

// gather_value for an 8-bit volume, whose atlas holds v(x, y, z + 1) at bit 16: the four texels are pair_lerp's
// operands as they come (14 instructions after the gather instead of 29).
__device__ __forceinline__ int gather_value8(unsigned long long tex, const float2 *zoff, unsigned ux, unsigned uy,
                                             unsigned uz) {
    const float2 o = zoff[uz >> 16];
    const float u = __int_as_float((int)__funnelshift_r(ux, 0x4B00u, 16)) + o.x;
    const float v = __int_as_float((int)__funnelshift_r(uy, 0x4B00u, 16)) + o.y;
    const uint4 t = tex2Dgather<uint4>((cudaTextureObject_t)tex, u, v, 0);
    const uint32_t x0[2] = {t.w, t.x}, x1[2] = {t.z, t.y};
    return pair_lerp(ux, uy, uz, x0, x1);
}

// quad_fetch and quad_lerp for an 8-bit volume, whose quads are the four bytes of one 32-bit texel: two
// registers come back through the texture path instead of eight.
__device__ __forceinline__ int quad_value8(unsigned long long tex, unsigned ux, unsigned uy, unsigned uz) {
    const int ix = (int)(ux >> 16), iy = (int)(uy >> 16), iz = (int)(uz >> 16);
    uint32_t a, b, unused[3];
    tex_quad(tex, ix, iy, iz, a, unused[0], unused[1], unused[2]);
    tex_quad(tex, ix + 1, iy, iz, b, unused[0], unused[1], unused[2]);
    const uint32_t x0[2] = {__byte_perm(a, 0u, 0x4240), __byte_perm(a, 0u, 0x4341)};
    const uint32_t x1[2] = {__byte_perm(b, 0u, 0x4240), __byte_perm(b, 0u, 0x4341)};
    return pair_lerp(ux, uy, uz, x0, x1);
}

// The layouts of the moving volume, written straight into their arrays (blocks of 32 x 8 voxels of a plane).
template <typename T>
__global__ void __launch_bounds__(256)
    k_make_zpairs(const T *__restrict__ in, int n0, int n1, int n2, int ph, cudaSurfaceObject_t out) {
    const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 8 + threadIdx.y, z = blockIdx.z;
    if (x >= n0 || y >= n1) return;
    const long long plane = (long long)n0 * n1, at = (long long)y * n0 + x;
    const uint32_t a = in[plane * z + at], b = in[plane * min(z + 1, n2 - 1) + at];
    surf2Dwrite(a | b << (sizeof(T) == 1 ? 16 : 20), out, ((z / ph) * n0 + x) * 4, (z % ph) * n1 + y);
}

template <typename T>
__global__ void __launch_bounds__(256)
    k_make_quads(const T *__restrict__ in, int n0, int n1, int n2, cudaSurfaceObject_t out) {
    const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 8 + threadIdx.y, z = blockIdx.z;
    if (x >= n0 || y >= n1) return;
    const T *p0 = in + (long long)n0 * n1 * z + x, *p1 = in + (long long)n0 * n1 * min(z + 1, n2 - 1) + x;
    const long long r0 = (long long)n0 * y, r1 = (long long)n0 * min(y + 1, n1 - 1);
    const uint32_t a = p0[r0], b = p0[r1], c = p1[r0], d = p1[r1];
    if (sizeof(T) == 1)
        surf3Dwrite(a | b << 8 | c << 16 | d << 24, out, x * 4, y, z);
    else
        surf3Dwrite(make_ushort4((unsigned short)a, (unsigned short)b, (unsigned short)c, (unsigned short)d), out, x * 8, y, z);
}

// Builds the padded x-paired volume: out has dims (n0, n1 + 1, n2 + 1).
template <typename T, typename PairT>
__global__ void k_make_pairs(const T *__restrict__ in, int n0, int n1, int n2, PairT *__restrict__ out) {
    constexpr int HB = (int)sizeof(PairT) * 4;
    const long long n = (long long)n0 * (n1 + 1) * (n2 + 1);
    for (long long o = blockIdx.x * (long long)blockDim.x + threadIdx.x; o < n; o += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(o % n0);
        const int y = min((int)((o / n0) % (n1 + 1)), n1 - 1);
        const int z = min((int)(o / ((long long)n0 * (n1 + 1))), n2 - 1);
        const long long src = x + (long long)n0 * (y + (long long)n1 * z);
        out[o] = (PairT)((uint32_t)in[src] | ((uint32_t)in[x < n0 - 1 ? src + 1 : src] << HB));
    }
}

// Overlap interval [lo, hi] of fixed row (j, k) and the 16.16 moving index at i = lo.
struct RowClip {
    int lo, hi, u0, u1, u2;
};

__device__ __forceinline__ bool inside_at(const long long base[3], const int st[3], const long long umax[3], int i) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        long long U = base[a] + (long long)st[a] * i;
        if (U < 0 || U > umax[a]) return false;
    }
    return true;
}

__device__ RowClip clip_row(const int *q, int j, int k, int nf0, const int nm[3]) {
    long long base[3], umax[3];
    int st[3];
    int lo = 0, hi = nf0 - 1;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        base[a] = (long long)q[4 * a + 1] * j + (long long)q[4 * a + 2] * k + (long long)q[4 * a + 3];
        umax[a] = (long long)(nm[a] - 1) << 16;
        st[a] = q[4 * a];
        if (st[a] == 0) {
            if (base[a] < 0 || base[a] > umax[a]) { lo = nf0; hi = -1; }
        } else {
            // estimate of the real interval {i : 0 <= base + st i <= umax}; within one voxel of the truth
            const float fb = (float)base[a], fs = (float)st[a], fm = (float)umax[a];
            float e0 = -fb / fs, e1 = (fm - fb) / fs;
            float a0 = fminf(e0, e1), a1 = fmaxf(e0, e1);
            a0 = fminf(fmaxf(a0, -2.0f), (float)nf0 + 1.0f);
            a1 = fminf(fmaxf(a1, -2.0f), (float)nf0 + 1.0f);
            lo = max(lo, (int)ceilf(a0));
            hi = min(hi, (int)floorf(a1));
        }
    }
    // exact fix-up: the interval of a linear function is contiguous
    while (lo <= hi && !inside_at(base, st, umax, lo)) ++lo;
    while (lo > 0 && lo <= nf0 && inside_at(base, st, umax, lo - 1)) --lo;
    while (hi >= lo && !inside_at(base, st, umax, hi)) --hi;
    while (hi >= lo && hi < nf0 - 1 && inside_at(base, st, umax, hi + 1)) ++hi;
    if (hi < lo && lo < nf0 && inside_at(base, st, umax, lo)) {
        hi = lo;
        while (hi < nf0 - 1 && inside_at(base, st, umax, hi + 1)) ++hi;
    }
    RowClip r;
    r.lo = lo;
    r.hi = hi;
    r.u0 = r.u1 = r.u2 = 0;
    if (lo <= hi) {
        r.u0 = (int)(base[0] + (long long)st[0] * lo);
        r.u1 = (int)(base[1] + (long long)st[1] * lo);
        r.u2 = (int)(base[2] + (long long)st[2] * lo);
    }
    return r;
}

// ---------------------------------------------------------------------------
// Shared-memory histogram policies
// ---------------------------------------------------------------------------

// Shared histograms address cell (bf, bm) through rows padded by one word:
// with a row stride of S = B + 1 words the bank is (row + column) mod 32,
// so cells clustered in a few moving bins (the Rician background occupies
// bins 0..15 of both volumes) still spread over the banks.

// 32-bit counters: one shared atomic per voxel (or per group of equal cells in a warp).
template <bool MATCH>
struct HistU32 {
    uint32_t *h;
    int B, S;  // bins, padded row stride in words
    __device__ void load_info(const uint32_t *) {}
    __device__ void zero() {
        for (int c = threadIdx.x; c < B * S; c += blockDim.x) h[c] = 0;
    }
    __device__ __forceinline__ void add(int bf, int bm, bool valid) {
        const int idx = bf * S + bm;
        if (!MATCH) {
            if (valid) atomicAdd(&h[idx], 1u);
        } else {
            const unsigned vm = __ballot_sync(kFull, valid);
            if (valid) {
                const unsigned peers = __match_any_sync(vm, idx);
                if ((int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&h[idx], (unsigned)__popc(peers));
            }
        }
    }
    __device__ __forceinline__ uint32_t count(int bf, int bm) const { return h[bf * S + bm]; }
};

// 16-bit counters, two per word: the word at (row r, column bm) holds cell
// (r, bm) in its low half and cell (r + H, bm) in its high half, H = ceil(B/2),
// so the two halves of a word belong to fixed bins far apart and rarely
// collide.  A counter whose value reaches kDrainT is drained whole into a
// shared hash table of 32-bit overflow counts by a compare-and-swap; the
// adder that observed it does the drain, so a counter never exceeds
// kDrainT + (threads x 32) < 2^16.  The true count is the 16-bit value plus
// the overflow entry (flagged in a bitmap).  Overflow entries are keyed by
// the cell id bf * B + bm.
// Iteration cap of the drain's compare-and-swap loop (a failure-handling test hook lowers it; at 0
// every drain gives up at once and flags the error).
__device__ int g_drain_cap = 1 << 16;

template <bool MATCH>
struct HistU16 {
    uint32_t *w;      // H x S words
    uint32_t *okey;   // kOvfSlots keys
    uint32_t *ocnt;   // kOvfSlots counts
    uint32_t *bmap;   // (B^2 + 31) / 32 words
    int *flags;
    int B, S, H;
    __device__ void load_info(const uint32_t *) {}
    __device__ void zero() {
        const int nw = H * S, nb = (B * B + 31) >> 5;
        for (int c = threadIdx.x; c < nw; c += blockDim.x) w[c] = 0;
        for (int c = threadIdx.x; c < kOvfSlots; c += blockDim.x) {
            okey[c] = kEmptyKey;
            ocnt[c] = 0;
        }
        for (int c = threadIdx.x; c < nb; c += blockDim.x) bmap[c] = 0;
    }
    __device__ __forceinline__ static uint32_t slot_of(uint32_t key) { return (key * 2654435761u) >> 20; }
    __device__ void ovf_add(uint32_t key, uint32_t amount) {
        uint32_t s = slot_of(key) & (kOvfSlots - 1);
        for (int probe = 0; probe < kOvfSlots; ++probe) {
            const uint32_t k = ((volatile uint32_t *)okey)[s];
            if (k == key) {
                atomicAdd(&ocnt[s], amount);
                return;
            }
            if (k == kEmptyKey) {
                const uint32_t prev = atomicCAS(&okey[s], kEmptyKey, key);
                if (prev == kEmptyKey || prev == key) {
                    atomicAdd(&ocnt[s], amount);
                    if (prev == kEmptyKey) atomicOr(&bmap[key >> 5], 1u << (key & 31));
                    return;
                }
            }
            s = (s + 1) & (kOvfSlots - 1);
        }
        atomicOr(&flags[1], 1);  // cannot happen while N <= kOvfSlots / 2 * kDrainT
    }
    __device__ void drain(uint32_t idx, uint32_t sh, uint32_t key) {
        volatile uint32_t *vw = w;
        const int cap = g_drain_cap;
        // each failed attempt means another update of this word succeeded; bounded for safety
        for (int it = 0; it < cap; ++it) {
            const uint32_t cur = vw[idx];
            const uint32_t hv = (cur >> sh) & 0xffffu;
            if (hv < (uint32_t)kDrainT) return;
            if (atomicCAS(&w[idx], cur, cur - (hv << sh)) == cur) {
                ovf_add(key, hv);
                return;
            }
        }
        atomicOr(&flags[1], 2);
    }
    __device__ __forceinline__ void inc(int bf, int bm, uint32_t n) {
        const bool hi = bf >= H;
        const uint32_t idx = (uint32_t)((hi ? bf - H : bf) * S + bm), sh = hi ? 16u : 0u;
        const uint32_t old = atomicAdd(&w[idx], n << sh);
        if (((old >> sh) & 0xffffu) + n >= (uint32_t)kDrainT) drain(idx, sh, (uint32_t)(bf * B + bm));
    }
    __device__ __forceinline__ void add(int bf, int bm, bool valid) {
        if (!MATCH) {
            if (valid) inc(bf, bm, 1u);
        } else {
            const unsigned vm = __ballot_sync(kFull, valid);
            if (valid) {
                const unsigned peers = __match_any_sync(vm, bf * B + bm);
                if ((int)(threadIdx.x & 31) == __ffs(peers) - 1) inc(bf, bm, (unsigned)__popc(peers));
            }
        }
    }
    __device__ __forceinline__ uint32_t count(int bf, int bm) const {
        const bool hi = bf >= H;
        uint32_t v = (w[(hi ? bf - H : bf) * S + bm] >> (hi ? 16 : 0)) & 0xffffu;
        const int c = bf * B + bm;
        if (bmap[c >> 5] & (1u << (c & 31))) {
            uint32_t s = slot_of((uint32_t)c) & (kOvfSlots - 1);
            for (int probe = 0; probe < kOvfSlots; ++probe) {
                const uint32_t k = okey[s];
                if (k == (uint32_t)c) return v + ocnt[s];
                if (k == kEmptyKey) break;
                s = (s + 1) & (kOvfSlots - 1);
            }
        }
        return v;
    }
};

// Row-bound layout.  A cell count can never exceed the number of fixed voxels
// in its row's bin, F[r] (each fixed voxel contributes at most once per
// transform), and F is known when the context is built.  Rows with
// F[r] <= 65535 ("narrow") share words two at a time as 16-bit halves; the
// others ("wide") get 32-bit words.  No counter can overflow, so increments
// are fire-and-forget atomics with no return value and no drain.  rowinfo[r]
// = word offset of row r << 6 | wide << 5 | shift (0 or 16: the half of a
// narrow row); rows are padded to S = B + 1 words.
struct HistRows {
    uint32_t *w;
    uint32_t *info;  // B entries, copied into shared memory per item
    int B, S, nwords;
    __device__ void load_info(const uint32_t *rowinfo) {
        for (int r = threadIdx.x; r < B; r += blockDim.x) info[r] = __ldg(rowinfo + r);
    }
    __device__ void zero() {
        for (int c = threadIdx.x; c < nwords; c += blockDim.x) w[c] = 0;
    }
    __device__ __forceinline__ void add(int bf, int bm, bool valid) {
        if (valid) {
            const uint32_t inf = info[bf];
            // 1 << (inf & 31): the funnel shift takes its count modulo 32
            atomicAdd(&w[(inf >> 6) + bm], __funnelshift_l(0u, 1u, inf));
        }
    }
    __device__ __forceinline__ uint32_t count(int bf, int bm) const {
        const uint32_t inf = info[bf];
        const uint32_t v = w[(inf >> 6) + bm] >> (inf & 31u);
        return (inf & 32u) ? v : (v & 0xffffu);
    }
};

// Shared-memory layout of a CTA: [histogram words][ovf keys][ovf counts][bitmap] [rows][cols] [FP64 scratch].
__host__ __device__ inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

struct SmemLayout {
    size_t hist, okey, ocnt, bmap, rinfo, rows, cols, red, zoff, small, total;
    bool has_small;  // the count table of reduce_entropies fits
};
constexpr int kReduceWords = 1024;

// zmax: planes of the largest moving volume (gathers keep one float2 offset per plane).  The host, which sizes
// the allocation, and the kernels, which address it, have to pass the same counter kind and fetch.
__host__ __device__ inline SmemLayout smem_layout(int kind, int fetch, int bins, int rows_words, int zmax) {
    SmemLayout L;
    const size_t B2 = (size_t)bins * bins;
    const bool u16 = kind == HV_U16 || kind == HV_U16_MATCH;
    const size_t S = (size_t)bins + 1, H = ((size_t)bins + 1) / 2;
    size_t o = 0;
    L.hist = o;
    if (kind == HV_ROWS)
        o += (size_t)rows_words * 4;
    else
        o += u16 ? H * S * 4 : (size_t)bins * S * 4;
    L.okey = o;
    if (u16) o += (size_t)kOvfSlots * 4;
    L.ocnt = o;
    if (u16) o += (size_t)kOvfSlots * 4;
    L.bmap = o;
    if (u16) o += ((B2 + 31) / 32) * 4;
    L.rinfo = o;
    if (kind == HV_ROWS) o += (size_t)bins * 4;
    L.rows = o;
    o += (size_t)bins * 4;
    L.cols = o;
    o += (size_t)bins * 4;
    o = align_up(o, 16);
    L.red = o;
    o += (size_t)(3 * 32 + 3 * kMaxQ + 1) * 8;
    L.zoff = o;
    if (fetch == FM_GATHER) o += (size_t)zmax * 8;
    L.small = o;
    L.has_small = o + kReduceWords * 4 <= kMaxCtaSmem;
    if (L.has_small) o += kReduceWords * 4;
    L.total = o;
    return L;
}

template <int HV>
struct HistOf;
template <>
struct HistOf<HV_U32> { using T = HistU32<false>; };
template <>
struct HistOf<HV_U32_MATCH> { using T = HistU32<true>; };
template <>
struct HistOf<HV_U16> { using T = HistU16<false>; };
template <>
struct HistOf<HV_U16_MATCH> { using T = HistU16<true>; };
template <>
struct HistOf<HV_ROWS> { using T = HistRows; };

template <int HV>
__device__ typename HistOf<HV>::T make_hist(unsigned char *smem, const SmemLayout &L, int B, int *flags,
                                            int rows_words = 0) {
    typename HistOf<HV>::T H;
    H.B = B;
    H.S = B + 1;
    if constexpr (HV == HV_U16 || HV == HV_U16_MATCH) {
        H.H = (B + 1) / 2;
        H.w = (uint32_t *)(smem + L.hist);
        H.okey = (uint32_t *)(smem + L.okey);
        H.ocnt = (uint32_t *)(smem + L.ocnt);
        H.bmap = (uint32_t *)(smem + L.bmap);
        H.flags = flags;
    } else if constexpr (HV == HV_ROWS) {
        H.w = (uint32_t *)(smem + L.hist);
        H.info = (uint32_t *)(smem + L.rinfo);
        H.nwords = rows_words;
        (void)flags;
    } else {
        H.h = (uint32_t *)(smem + L.hist);
        (void)flags;
        (void)rows_words;
    }
    return H;
}

// ---------------------------------------------------------------------------
// Voxel loops: warps take batches of 32 fixed rows; lane l clips the l-th,
// then the warp walks the clipped rows.  The row blocks first_block +
// n * block_stride, n = 0, 1, ..., below n_end are visited.
// ---------------------------------------------------------------------------

// The interpolated moving value at a 16.16 index, through the variant's fetch path (PairT: uint16_t for an
// 8-bit moving volume, uint32_t for a 16-bit one).
template <int FM, typename PairT>
__device__ __forceinline__ int sample_value(const PairDev &P, const float2 *zoff, unsigned U0, unsigned U1,
                                            unsigned U2) {
    constexpr bool bytes = sizeof(PairT) == 2;
    if constexpr (FM == FM_GATHER && bytes) {
        return gather_value8(P.texg, zoff, U0, U1, U2);
    } else if constexpr (FM == FM_QUAD && bytes) {
        return quad_value8(P.texq, U0, U1, U2);
    } else if constexpr (FM == FM_GATHER) {
        return gather_value(P.texg, zoff, U0, U1, U2);
    } else if constexpr (FM == FM_QUAD) {
        uint32_t t[8];
        quad_fetch(P.texq, U0, U1, U2, t);
        return quad_lerp(U0, U1, U2, t);
    } else if constexpr (FM == FM_TEX) {
        return sample_hard_tex<PairT>(P.texp, (int)U0, (int)U1, (int)U2);
    } else {
        const int n0 = P.nm[0], sz = n0 * (P.nm[1] + 1);
        return sample_hard_pair<PairT>((const PairT *)P.movp, n0, sz, n0, sz, (int)U0, (int)U1, (int)U2);
    }
}

// Random sampling: the sampled voxels of each clipped row [lo, hi]; U at an entry's x index i is
// u_lo + st (i - lo), exact inside the interval.  A warp works on kSampledRows neighbouring rows at once: at
// 192 voxels and a quarter of them a row's entries are six steps of 8 lanes where they were two of 32, one
// broadcast serves all the rows, and the lanes that clip the rows load where their entries lie, so that no
// step waits for its row's offsets first.  Blocks are nwarps x kSampledRows rows.  400 transforms, a quarter of
// 192 x 192 x 128 at 64 bins: 2687 us one row at a time, 1982 with two rows, 1845 with four.
template <typename PairT, int FM, class Hist>
__device__ void accumulate_sampled(const PairDev &P, const int *q, const float2 *zoff, long long first_block,
                                   long long block_stride, long long n_end, Hist &H) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int nf0 = P.nf[0], nf1 = P.nf[1];
    const long long R = (long long)nf1 * P.nf[2];
    const int st0 = q[0], st1 = q[4], st2 = q[8];
    const int bins = P.bins, mdepth = P.mdepth;
    constexpr int G = kSampledRows, L = 32 / G;  // rows a step, lanes a row
    const int sub = lane / L, pos = lane % L;
    for (long long n0b = 0;; n0b += L) {
        if (first_block + n0b * block_stride >= n_end) break;
        RowClip mine;
        mine.lo = 0;
        mine.hi = -1;
        mine.u0 = mine.u1 = mine.u2 = 0;
        uint32_t k0 = 0, k1 = 0;  // the row's entries, none for an empty interval
        const long long nl = first_block + (n0b + lane / G) * block_stride;
        if (nl < n_end) {
            const long long rl = (nl * nwarps + warp) * G + lane % G;
            if (rl < R) {
                k0 = __ldg(P.srow + rl);
                k1 = __ldg(P.srow + rl + 1);
                mine = clip_row(q, (int)rl % nf1, (int)rl / nf1, nf0, P.nm);
                if (mine.lo > mine.hi) k1 = k0;
            }
        }
        for (int s0 = 0; s0 < 32; s0 += G) {
            if (first_block + (n0b + s0 / G) * block_stride >= n_end) break;  // warp-uniform
            const int s = s0 + sub;
            const uint32_t e0 = __shfl_sync(kFull, k0, s), e1 = __shfl_sync(kFull, k1, s);
            const int steps = (int)__reduce_max_sync(kFull, (e1 - e0 + L - 1) / L);
            if (steps == 0) continue;
            const int lo = __shfl_sync(kFull, mine.lo, s), hi = __shfl_sync(kFull, mine.hi, s);
            const unsigned ub0 = (unsigned)__shfl_sync(kFull, mine.u0, s), ub1 = (unsigned)__shfl_sync(kFull, mine.u1, s),
                           ub2 = (unsigned)__shfl_sync(kFull, mine.u2, s);
            uint32_t k = e0 + pos;
#pragma unroll 2
            for (int step = 0; step < steps; ++step, k += L) {
                int i = -1, bf = 0, bm = 0;
                if (k < e1) {
                    i = (int)__ldg(P.scol + k);
                    bf = (int)__ldg(P.sbin + k);
                }
                const bool valid = i >= lo && i <= hi && k < e1;
                if (valid) {
                    const unsigned d = (unsigned)(i - lo);
                    bm = (sample_value<FM, PairT>(P, zoff, ub0 + (unsigned)st0 * d, ub1 + (unsigned)st1 * d,
                                                  ub2 + (unsigned)st2 * d) * bins) >> mdepth;
                }
                H.add(bf, bm, valid);
            }
        }
    }
}

// Row walk (x-pair fetches): the CTA walks blocks of nwarps adjacent fixed rows (block blk
// holds rows blk * nwarps + w) and warp w takes row w of each block, so at any
// time the warps of a CTA sample neighbouring moving lines (row j's upper y
// neighbours are row j + 1's samples).  A warp clips its next 32 rows at once (lane l
// takes the warp's l-th upcoming row, exactly in 64 bits), then walks them one
// by one, 32 voxels at a time, with each row's interval broadcast by shuffles.
template <typename PairT, int FM, class Hist>
__device__ void accumulate_rows(const PairDev &P, const int *q, long long first_block, long long block_stride,
                                long long n_end, Hist &H) {
    static_assert(FM == FM_LDG || FM == FM_TEX, "quads and gathers take the group and stream walks");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int nf0 = P.nf[0], nf1 = P.nf[1];
    const long long R = (long long)nf1 * P.nf[2];
    const int n0 = P.nm[0], sy = n0, sz = n0 * (P.nm[1] + 1);
    const int st0 = q[0], st1 = q[4], st2 = q[8];
    const int bins = P.bins, mdepth = P.mdepth;
    const PairT *__restrict__ movp = (const PairT *)P.movp;
    for (long long n0b = 0;; n0b += 32) {
        // blocks of this group: lane l gets block first_block + (n0b + l) * block_stride
        if (first_block + n0b * block_stride >= n_end) break;
        RowClip mine;
        mine.lo = 0;
        mine.hi = -1;
        mine.u0 = mine.u1 = mine.u2 = 0;
        const long long nl = first_block + (n0b + lane) * block_stride;
        if (nl < n_end) {
            const long long rl = nl * nwarps + warp;
            if (rl < R) mine = clip_row(q, (int)rl % nf1, (int)rl / nf1, nf0, P.nm);
        }
        for (int s = 0; s < 32; ++s) {
            const long long n = first_block + (n0b + s) * block_stride;
            if (n >= n_end) break;  // warp-uniform
            const long long r = n * nwarps + warp;
            if (r >= R) break;  // warp-uniform: only the last block may be partial
            const int lo = __shfl_sync(kFull, mine.lo, s), hi = __shfl_sync(kFull, mine.hi, s);
            if (lo > hi) continue;
            const unsigned ub0 = (unsigned)__shfl_sync(kFull, mine.u0, s), ub1 = (unsigned)__shfl_sync(kFull, mine.u1, s),
                           ub2 = (unsigned)__shfl_sync(kFull, mine.u2, s);
            // unsigned: lanes past the row end may step outside the int range; only in-range lanes use them
            unsigned U0 = ub0 + (unsigned)st0 * lane, U1 = ub1 + (unsigned)st1 * lane, U2 = ub2 + (unsigned)st2 * lane;
            const uint8_t *__restrict__ frow = P.fbins + (size_t)r * nf0;
            for (int i = lo + lane; i - lane <= hi; i += 32) {
                const bool valid = i <= hi;
                int bf = 0, bm = 0;
                if (valid) {
                    int v;
                    if constexpr (FM == FM_TEX)
                        v = sample_hard_tex<PairT>(P.texp, (int)U0, (int)U1, (int)U2);
                    else
                        v = sample_hard_pair<PairT>(movp, sy, sz, n0, sz, (int)U0, (int)U1, (int)U2);
                    bm = (v * bins) >> mdepth;
                    bf = (int)__ldg(frow + i);
                }
                H.add(bf, bm, valid);
                U0 += 32u * (unsigned)st0;
                U1 += 32u * (unsigned)st1;
                U2 += 32u * (unsigned)st2;
            }
        }
    }
}

// Row-group walk (quad and gather fetches, every fixed voxel).  A block is nwarps * G adjacent fixed rows,
// G = 32 >> lpr_log2 of them to each warp, and each warp step covers the warp's G rows of a block with
// L = 1 << lpr_log2 lanes each (lane = row-in-group * L + column), so a row whose overlap is not a
// multiple of 32 wastes at most L - 1 lanes in its last step, and one clip broadcast serves G rows.  Rows
// are clipped 32 at a time (32 / G blocks).  The rows of a step being neighbours, they end together and
// their fetches share texels; as rows nwarps apart 4096 transforms of 256^3 took 163.6 ms, now 152,
// and 768 on twelve pairs 13.4, now 12.0.
// Steps in which every lane of every row is inside its interval run without predicates; the last
// ones (up to the longest row of the group) are predicated.  The fixed bin of the next full step is
// loaded one step ahead.
template <typename PairT, int FM, class Hist>
__device__ void accumulate_groups(const PairDev &P, const int *q, const float2 *zoff, long long first_block,
                                  long long block_stride, long long n_end, int lpr_log2, Hist &H) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int nf0 = P.nf[0], nf1 = P.nf[1];
    const long long R = (long long)nf1 * P.nf[2];
    const int st0 = q[0], st1 = q[4], st2 = q[8];
    const int bins = P.bins, mdepth = P.mdepth;
    const int lpr = 1 << lpr_log2, gsz = 32 >> lpr_log2;
    const int sub = lane >> lpr_log2, col = lane & (lpr - 1);
    const unsigned d0 = (unsigned)st0 << lpr_log2, d1 = (unsigned)st1 << lpr_log2, d2 = (unsigned)st2 << lpr_log2;
    for (long long n0b = 0;; n0b += 32 / gsz) {
        if (first_block + n0b * block_stride >= n_end) break;
        RowClip mine;
        mine.lo = 0;
        mine.hi = -1;
        mine.u0 = mine.u1 = mine.u2 = 0;
        const long long nl = first_block + (n0b + lane / gsz) * block_stride;
        if (nl < n_end) {
            const long long rl = (nl * nwarps + warp) * gsz + lane % gsz;
            if (rl < R) mine = clip_row(q, (int)rl % nf1, (int)rl / nf1, nf0, P.nm);
        }
        for (int s0 = 0; s0 < 32; s0 += gsz) {
            const long long n = first_block + (n0b + s0 / gsz) * block_stride;
            if (n >= n_end) break;  // warp-uniform
            const int s = s0 + sub;
            const int lo = __shfl_sync(kFull, mine.lo, s), hi = __shfl_sync(kFull, mine.hi, s);
            const int len = hi >= lo ? hi - lo + 1 : 0;  // rows past the end were clipped empty
            const int kfull = (int)__reduce_min_sync(kFull, (unsigned)(len >> lpr_log2));
            const int kall = (int)__reduce_max_sync(kFull, (unsigned)((len + lpr - 1) >> lpr_log2));
            if (kall == 0) continue;
            const unsigned ub0 = (unsigned)__shfl_sync(kFull, mine.u0, s), ub1 = (unsigned)__shfl_sync(kFull, mine.u1, s),
                           ub2 = (unsigned)__shfl_sync(kFull, mine.u2, s);
            const long long r = (n * nwarps + warp) * gsz + sub;
            // unsigned: lanes past their row's end may step outside the int range; only in-range lanes use them
            unsigned U0 = ub0 + (unsigned)st0 * col, U1 = ub1 + (unsigned)st1 * col, U2 = ub2 + (unsigned)st2 * col;
            const uint8_t *__restrict__ fp = P.fbins + (len > 0 ? (size_t)r * nf0 + lo + col : 0);
            int k = 0;
            int bf_next = kfull > 0 ? (int)__ldg(fp) : 0;
#pragma unroll 2
            for (; k < kfull; ++k) {
                const int bf = bf_next;
                fp += lpr;
                if (k + 1 < kfull) bf_next = (int)__ldg(fp);
                H.add(bf, (sample_value<FM, PairT>(P, zoff, U0, U1, U2) * bins) >> mdepth, true);
                U0 += d0;
                U1 += d1;
                U2 += d2;
            }
            for (; k < kall; ++k) {
                const bool valid = (k << lpr_log2) + col < len;
                int bf = 0, bm = 0;
                if (valid) {
                    bm = (sample_value<FM, PairT>(P, zoff, U0, U1, U2) * bins) >> mdepth;
                    bf = (int)__ldg(fp);
                }
                H.add(bf, bm, valid);
                fp += lpr;
                U0 += d0;
                U1 += d1;
                U2 += d2;
            }
        }
    }
}

// Stream walk (quad and gather fetches, every fixed voxel).  A warp clips its next 32 rows at once
// (lane s takes row s of the batch), then walks their overlap intervals as one stream of voxels: lane
// l takes stream positions l, l + 32, ...  An exclusive scan of the interval lengths gives each row's
// start in the stream; a lane crossing the end of its row moves to the next non-empty one and
// re-reads that row's 16.16 index and fixed-bin offset by shuffles from the row's clipping lane.
// Between row ends the warp runs segments of full steps (the most steps before any lane leaves its
// row, one warp-wide minimum) exactly like the row walk's predicate-free loop; only the batch's last
// step is partial (instead of every row's).  U = u_lo + st (i - lo) inside a row's interval is exact
// in 32 bits.
template <typename PairT, int FM, class Hist>
__device__ void accumulate_stream(const PairDev &P, const int *q, const float2 *zoff, long long first_block,
                                  long long block_stride, long long n_end, Hist &H) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int nf0 = P.nf[0], nf1 = P.nf[1];
    const long long R = (long long)nf1 * P.nf[2];
    const int st0 = q[0], st1 = q[4], st2 = q[8];
    const int bins = P.bins, mdepth = P.mdepth;
    const unsigned d0 = 32u * (unsigned)st0, d1 = 32u * (unsigned)st1, d2 = 32u * (unsigned)st2;
    for (long long n0b = 0;; n0b += 32) {
        if (first_block + n0b * block_stride >= n_end) break;
        RowClip mine;
        mine.lo = 0;
        mine.hi = -1;
        mine.u0 = mine.u1 = mine.u2 = 0;
        long long rl = 0;
        const long long nl = first_block + (n0b + lane) * block_stride;
        if (nl < n_end) {
            rl = nl * nwarps + warp;
            if (rl < R) mine = clip_row(q, (int)rl % nf1, (int)rl / nf1, nf0, P.nm);
        }
        const int len = mine.hi >= mine.lo ? mine.hi - mine.lo + 1 : 0;
        int incl = len;  // inclusive scan: the end of this lane's row in the stream
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += y;
        }
        const int total = __shfl_sync(kFull, incl, 31);
        if (total == 0) continue;
        // offset of the row's first overlap voxel in the fixed bins (rows past the end are empty)
        const long long rowoff = len > 0 ? rl * nf0 + mine.lo : 0;
        int s = -1, e = 0;  // this lane's row and that row's end in the stream
        unsigned U0 = 0, U1 = 0, U2 = 0;
        const uint8_t *__restrict__ fp = P.fbins;
        for (int g0 = 0; g0 < total;) {
            const int g = g0 + lane;
            bool moved = false;  // warp-uniform
            while (__any_sync(kFull, g < total && g >= e)) {
                if (g < total && g >= e) ++s;
                e = __shfl_sync(kFull, incl, s & 31);
                moved = true;
            }
            if (moved) {  // lanes that stayed re-read their own row: no change
                const int sc = s & 31;
                const int start = e - __shfl_sync(kFull, len, sc);
                const unsigned dd = (unsigned)(g - start);
                U0 = (unsigned)__shfl_sync(kFull, mine.u0, sc) + (unsigned)st0 * dd;
                U1 = (unsigned)__shfl_sync(kFull, mine.u1, sc) + (unsigned)st1 * dd;
                U2 = (unsigned)__shfl_sync(kFull, mine.u2, sc) + (unsigned)st2 * dd;
                fp = P.fbins + (__shfl_sync(kFull, rowoff, sc) + (long long)dd);
            }
            if (g0 + 32 <= total) {
                // a segment of full steps in which no lane leaves its row: predicate-free, two steps per
                // trip, the next step's fixed bin loaded one step ahead
                int nfree = (int)__reduce_min_sync(kFull, (unsigned)((e - g + 31) >> 5));
                nfree = min(nfree, (total - g0) >> 5);
                int bf_next = (int)__ldg(fp);
#pragma unroll 2
                for (int k = 0; k < nfree; ++k) {
                    const int bf = bf_next;
                    fp += 32;
                    if (k + 1 < nfree) bf_next = (int)__ldg(fp);
                    H.add(bf, (sample_value<FM, PairT>(P, zoff, U0, U1, U2) * bins) >> mdepth, true);
                    U0 += d0;
                    U1 += d1;
                    U2 += d2;
                }
                g0 += 32 * nfree;
            } else {  // the batch's last, partial step
                const bool valid = g < total;
                int bf = 0, bm = 0;
                if (valid) {
                    bf = (int)__ldg(fp);
                    bm = (sample_value<FM, PairT>(P, zoff, U0, U1, U2) * bins) >> mdepth;
                }
                H.add(bf, bm, valid);
                g0 = total;
            }
        }
    }
}

// The voxel walk of a variant: quad and gather fetches over every fixed voxel take the stream walk
// (lpr_log2 == 0) or the row-group walk, the other fetches the one-row-at-a-time walk; random sampling has its
// own.
template <typename PairT, int FM, class Hist>
__device__ __forceinline__ void walk_rows(const PairDev &P, const int *q, const float2 *zoff, long long first_block,
                                          long long block_stride, long long n_end, int lpr_log2, Hist &H) {
    if (P.srow != nullptr) {
        accumulate_sampled<PairT, FM>(P, q, zoff, first_block, block_stride, n_end, H);
        return;
    }
    if constexpr (FM == FM_QUAD || FM == FM_GATHER) {
        if (lpr_log2 == 0)
            accumulate_stream<PairT, FM>(P, q, zoff, first_block, block_stride, n_end, H);
        else
            accumulate_groups<PairT, FM>(P, q, zoff, first_block, block_stride, n_end, lpr_log2, H);
    } else {
        accumulate_rows<PairT, FM>(P, q, first_block, block_stride, n_end, H);
    }
}

// Copies the per-plane atlas offsets of pair P into shared memory (gather fetches only).
template <int FM>
__device__ __forceinline__ void load_zoff(const PairDev &P, float2 *s_zoff) {
    if constexpr (FM == FM_GATHER) {
        for (int z = threadIdx.x; z < P.nm[2]; z += blockDim.x) s_zoff[z] = P.zoff[z];
    }
}

// ---------------------------------------------------------------------------
// Entropy reduction of one histogram by one CTA (Eq. 1, Eq. 2, Tsallis)
// ---------------------------------------------------------------------------

// Entropy terms of a count v < 2^31: v ln v (q == 1) or v^q, from the count-indexed table of 2^TB entries;
// beyond it, with m the leading TB bits of v, v = 2^e m (1 + x), 0 <= x < 2^(1 - TB), from the table's
// entries of m and 2^e and the series of ln(1 + x) or (1 + x)^q: three terms for a context's 65536 entries
// (TB 16), eight for the 256 an evaluation without a context builds itself (TB 8), whose rest is below
// 2^-54 of the result for q <= 7 (larger q: pow).  FP64 units are few (two lanes a clock an SM, so a
// warp's instruction takes 16 clocks whatever its active lanes), and a log or a pow is some 50 or 250
// instructions; the series takes eight for x, shared by every q, and five (ten) per q.
__device__ __noinline__ double pow_term(double v, double q) { return pow(v, q); }

struct Split {  // v = 2^e m (1 + x); e < 0: v is below the table's end
    int e;
    uint32_t m;
    double x;
};

template <int TB>
__device__ __forceinline__ Split split_count(uint32_t v) {
    Split s;
    s.e = v < (1u << TB) ? -1 : 32 - TB - __clz((int)v);
    if (s.e < 0) {
        s.m = v;
        s.x = 0.0;
        return s;
    }
    s.m = v >> s.e;
    const double dm = (double)s.m;
    double y = (double)__frcp_rn((float)s.m);  // 1 / m to 2^-24, then 2^-47, then (for x < 2^-7) 2^-53
    y = fma(fma(-dm, y, 1.0), y, y);
    if (TB < 16) y = fma(fma(-dm, y, 1.0), y, y);
    s.x = (double)(v - (s.m << s.e)) * y * __hiloint2double((1023 - s.e) << 20, 0);
    return s;
}

template <int TB>
__device__ __forceinline__ double split_term(uint32_t v, const Split &s, int iq, const QSet &Q) {
    constexpr int terms = TB == 16 ? 3 : kSeries;
    static_assert(TB == 16 || TB == 8, "terms are chosen for these tables");
    const double *__restrict__ tab = Q.tab[iq];
    const double tm = __ldg(tab + s.m);
    if (s.e < 0) return tm;
    const float qf = Q.q[iq];
    const double x = s.x;
    if (qf == 1.0f) {
        double l = 1.0 / terms;
#pragma unroll
        for (int k = terms - 1; k >= 1; --k) l = fma(-x, l, 1.0 / k);
        return fma((double)v, fma((double)s.e, 0.69314718055994530942, x * l), fma(x, tm, tm) * (double)(1u << s.e));
    }
    if (qf > 7.0f) return pow_term((double)v, (double)qf);
    double p = Q.binom[iq][terms - 2];
#pragma unroll
    for (int k = terms - 1; k >= 2; --k) p = fma(x, p, Q.binom[iq][k - 2]);
    p = x * fma(x, p, (double)qf);
    const double t = tm * __ldg(tab + (s.e < TB ? 1u << s.e : (1u << TB) + s.e - TB));
    return fma(t, p, t);
}

template <int TB>
__device__ __forceinline__ double term(uint32_t v, int iq, const QSet &Q) {
    return split_term<TB>(v, split_count<TB>(v), iq, Q);
}

// Warp-wide FP64 sums of four values: lane l gets the sum of a[l & 3].  Half of the values change lanes in
// each of the first two steps, so six additions are issued instead of twenty (16 clocks each).
__device__ __forceinline__ double warp_sum4(const double (&a)[4]) {
    const bool odd = threadIdx.x & 1, upper = threadIdx.x & 2;
    const double b0 = (odd ? a[1] : a[0]) + __shfl_xor_sync(kFull, odd ? a[0] : a[1], 1);
    const double b1 = (odd ? a[3] : a[2]) + __shfl_xor_sync(kFull, odd ? a[2] : a[3], 1);
    double c = (upper ? b1 : b0) + __shfl_xor_sync(kFull, upper ? b0 : b1, 2);
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) c += __shfl_xor_sync(kFull, c, o);
    return c;
}

// Entropies and MI of transform t from the overlap count N and, per q, the sums S over the fixed marginal,
// the moving marginal and the joint cells of c ln c (q == 1) or c^q: H = (N ln N - S) / N (Eq. 1),
// S_q = (1 - S / N^q) / (q - 1), MI = H_F + H_M - H_FM (Eq. 2) plus (1 - q) S_q(F) S_q(M) in the
// pseudo-additive form.  N ln N and N^q are the term of a cell that holds every voxel.  One warp: lane
// 3 iq + w brings sum w of q iq (so every division is issued once).
template <int TB>
__device__ void write_mi(uint32_t N, double S, const QSet &Q, long long t, const Outputs &O) {
    const int lane = threadIdx.x & 31, nq = Q.nq;
    if (lane == 0) {
        if (O.count) O.count[t] = (long long)N;
        if (N == 0 && O.flags) atomicOr(&O.flags[0], 1);
    }
    const int iq = min(lane / 3, nq - 1);
    const float qf = Q.q[iq];
    double h;
    if (N == 0) {
        h = __longlong_as_double(0x7ff8000000000000ll);
    } else {
        const double full = term<TB>(N, iq, Q);
        const bool shannon = qf == 1.0f;
        double unit = shannon ? (double)N : full;
        if (shannon && Q.bits) unit *= 0.69314718055994530942;
        const double r = (shannon ? full - S : S) / unit;
        h = shannon ? r : (1.0 - r) * Q.inv_q1[iq];
    }
    const double hm = __shfl_down_sync(kFull, h, 1), hj = __shfl_down_sync(kFull, h, 2);
    if (lane < 3 * nq) {
        if (O.h) O.h[t * nq * 3 + lane] = h;
        if (lane % 3 == 0 && O.mi) {
            double I = h + hm - hj;
            if (qf != 1.0f && Q.form == 1) I += (1.0 - (double)qf) * h * hm;
            O.mi[t * nq + iq] = I;
        }
    }
}

// Entropies of one histogram by one CTA, in one pass over the cells: marginals (row sums by warps,
// column sums by shared atomics) and the joint terms of every q.  FP64 bounds it, so additions are saved
// and FP64 instructions issued with full warps: most cells hold small counts, which are only counted
// (small[c] = number of cells that hold c < kSmallCounts, an integer atomic) and enter the sums as one
// product per count; counts below the table's end are looked up on the way; the few beyond it are listed
// and taken side by side at the end, largest first: warps list them in whatever order they come by, and sums that
// followed it differed from call to call.  One addition per cell and q, in a pass
// per q, with every thread adding every warp's partial sums and log / pow beyond the table, was 4 % of the
// batched kernel at 256 bins and four q (with the split tail, 4096 transforms of 256^3: 168.3 -> 163.6 ms a call).
constexpr int kSmallCounts = 768;
constexpr int kBigCounts = 255;

// The shared words of a reduction (kReduceWords): cells per small count, then the listed counts.
template <int TB>
struct CountTable {
    static constexpr uint32_t kBig = 1u << 16;  // counts listed (with TB 16 those beyond the table)
    uint32_t *small;  // null: no room, every term is taken on the way
    __device__ __forceinline__ uint32_t *nbig() const { return small + kSmallCounts; }
    __device__ __forceinline__ uint32_t *big() const { return small + kSmallCounts + 1; }
    __device__ void zero() {
        if (small)
            for (int c = threadIdx.x; c <= kSmallCounts; c += blockDim.x) small[c] = 0;
    }
    // True if the table took the count; else the caller adds its terms.
    __device__ __forceinline__ bool take(uint32_t v) {
        if (!small) return false;
        if (v < (uint32_t)kSmallCounts) {
            atomicAdd(&small[v], 1u);
            return true;
        }
        if (v < kBig) return false;
        const uint32_t i = atomicAdd(nbig(), 1u);
        if (i < (uint32_t)kBigCounts) big()[i] = v;
        return true;
    }
    // After the pass that took the counts: more large ones than the list holds.  Which of them it holds depends on
    // the warps' order, so it is not used: the caller repeats the pass and adds every large count's terms.
    __device__ __forceinline__ bool overflowed() const { return small && *nbig() > (uint32_t)kBigCounts; }
    // Orders the list by value (the whole CTA; each entry counts those before it).
    __device__ void sort() {
        const int n = small ? (int)*nbig() : 0, tid = threadIdx.x;
        if (n < 2) return;  // (the same for every thread)
        uint32_t v = 0;
        int rank = 0;
        if (tid < n) {
            v = big()[tid];
#pragma unroll 4
            for (int j = 0; j < n; ++j) {
                const uint32_t w = big()[j];
                rank += w > v || (w == v && j < tid);
            }
        }
        __syncthreads();
        if (tid < n) big()[rank] = v;
        __syncthreads();
    }
    // take's answer for a pass after the first.
    __device__ __forceinline__ bool taken_before(uint32_t v) const {
        return small && (v < (uint32_t)kSmallCounts || (v >= kBig && !overflowed()));
    }
    // This thread's share of the table's terms of q0 .. q0 + 3.
    __device__ __forceinline__ void add_terms(double (&a)[4], int q0, const QSet &Q) const {
        if (!small) return;
#pragma unroll 3
        for (int c = threadIdx.x; c < kSmallCounts; c += blockDim.x) {
            const uint32_t m = small[c];
            double tv[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) tv[k] = m && q0 + k < Q.nq ? term<TB>((uint32_t)c, q0 + k, Q) : 0.0;
            if (m) {
                const double dm = (double)m;
#pragma unroll
                for (int k = 0; k < 4; ++k) a[k] = fma(dm, tv[k], a[k]);
            }
        }
        const int n = overflowed() ? 0 : (int)*nbig();
        for (int i = threadIdx.x; i < n; i += blockDim.x) add_count(a, big()[i], q0, Q);
    }
    __device__ __forceinline__ static void add_count(double (&a)[4], uint32_t v, int q0, const QSet &Q) {
        const Split s = split_count<TB>(v);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (q0 + k < Q.nq) a[k] += split_term<TB>(v, s, q0 + k, Q);
    }
};
static_assert(kSmallCounts + 1 + kBigCounts == kReduceWords, "the table fills its shared words");

template <class Hist>
__device__ void reduce_entropies(const Hist &H, int B, const QSet &Q, uint32_t *s_rows, uint32_t *s_cols,
                                 double *s_red, CountTable<16> C, long long t, const Outputs &O) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const int nq = Q.nq;
    double *s_res = s_red + 3 * 32;  // 3 nq results after the per-warp scratch
    for (int c = tid; c < B; c += blockDim.x) s_cols[c] = 0;
    C.zero();
    __syncthreads();
    // four q per pass over the cells: the accumulators of more would spill
    bool first = true;  // the pass that takes the counts
    for (int q0 = 0; q0 < nq; q0 += 4) {
        double aj[4] = {0.0, 0.0, 0.0, 0.0};
        for (int r = warp; r < B; r += nwarps) {
            uint32_t rsum = 0;
            for (int c = lane; c < B; c += 32) {
                const uint32_t v = H.count(r, c);
                if (v == 0) continue;
                bool taken;
                if (first) {
                    rsum += v;
                    atomicAdd(&s_cols[c], v);
                    taken = C.take(v);
                } else {
                    taken = C.taken_before(v);
                }
                if (!taken) CountTable<16>::add_count(aj, v, q0, Q);
            }
            if (first) {
                rsum = __reduce_add_sync(kFull, rsum);
                if (lane == 0) s_rows[r] = rsum;
            }
        }
        __syncthreads();
        if (first) {
            first = false;
            if (C.overflowed()) {  // the first four q again, large counts on the way
                q0 -= 4;
                continue;
            }
            C.sort();
        }
        C.add_terms(aj, q0, Q);
        // joint sums: the upper 16 warps' into the lower 16; marginals: up to 64 entries a warp, warps
        // 0..3 the rows and 4..7 the columns; then warp 0 takes lane = 4 j + k for q0 + k
        double *s_joint = s_red, *s_marg = s_red + 64;
        double j = warp_sum4(aj);
        if (warp >= 16 && lane < 4) s_joint[4 * (warp - 16) + lane] = j;
        __syncthreads();
        if (warp < 16 && lane < 4) s_joint[4 * warp + lane] = j + (warp + 16 < nwarps ? s_joint[4 * warp + lane] : 0.0);
        if (warp < 8) {
            const uint32_t *m = warp < 4 ? s_rows : s_cols;
            double am[4] = {0.0, 0.0, 0.0, 0.0};
            for (int x = (warp & 3) * 32 + lane; x < B; x += 128)
                if (m[x]) CountTable<16>::add_count(am, m[x], q0, Q);
            const double v = warp_sum4(am);
            if (lane < 4) s_marg[4 * warp + lane] = v;
        }
        __syncthreads();
        if (warp == 0) {
            const int k = lane & 3, i = lane >> 2;
            double v = s_joint[4 * i + k] + s_joint[4 * (i + 8) + k], mg = s_marg[4 * i + k];
#pragma unroll
            for (int o = 4; o < 16; o <<= 1) {
                v += __shfl_xor_sync(kFull, v, o);
                mg += __shfl_xor_sync(kFull, mg, o);
            }
            v += __shfl_xor_sync(kFull, v, 16);
            if (q0 + k < nq) {
                if (i == 0) s_res[3 * (q0 + k) + 0] = mg;
                if (i == 4) s_res[3 * (q0 + k) + 1] = mg;
                if (i == 0) s_res[3 * (q0 + k) + 2] = v;
            }
        }
    }
    __syncthreads();
    if (warp == 0) {
        uint32_t N = 0;  // fewer than 2^31 voxels
        for (int r = lane; r < B; r += 32) N += s_rows[r];
        N = __reduce_add_sync(kFull, N);
        write_mi<16>(N, lane < 3 * nq ? s_res[lane] : 0.0, Q, t, O);
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------
// Entropies of the histograms in global memory (transforms whose work was split over CTAs)
// ---------------------------------------------------------------------------

// Grid (parts, slots): CTA (p, i) takes rows p, p + parts, ... of slot i's histogram (their cells' joint
// terms and their sums, the fixed marginal) and a contiguous share of its columns (the moving marginal).
// part[(i parts + p) kPartStride]: per q the sums of the fixed, moving and joint terms and, last, the
// count; the CTA that finishes a slot last (a counter in `done`, zeroed by the caller) adds the parts in a
// fixed order and writes the results.
// What bounds it: for one slot the latency of dependent FP64 instructions (64 clocks and more each on the
// SM's few FP64 lanes), so loads are issued together, sums are trees, marginal entries take a lane each
// beside one another and no step is left to one CTA but the last sum; for many slots the FP64 issue (16
// clocks a warp), so a CTA with many cells counts the small counts first (CountTable).
// Two launches (parts, then one CTA per transform), log / pow beyond the table and sums by one thread took
// 81 us for one transform at 256 bins and four q and 332 us for 81 at 128 bins and six; this takes 23 and 53.
constexpr int kPartStride = 3 * kMaxQ + 1;
constexpr int kEntThreads = 256;

__device__ __forceinline__ double tree8(const double *v, int stride) {
    return ((v[0] + v[stride]) + (v[2 * stride] + v[3 * stride])) +
           ((v[4 * stride] + v[5 * stride]) + (v[6 * stride] + v[7 * stride]));
}

// TB: bits of the tables in Q.  slots null: one histogram, `single`.
template <int TB>
__global__ void __launch_bounds__(kEntThreads, 4)
    k_entropy_slots(const uint32_t *__restrict__ hist, long long hist_stride, const Slot *__restrict__ slots, Slot single,
                    const __grid_constant__ QSet Q, unsigned int *__restrict__ done, double *__restrict__ part,
                    const __grid_constant__ Outputs O) {
    constexpr int nwarps = kEntThreads / 32;
    static_assert(nwarps == 8 && kPartStride <= 32, "trees over eight warps, a lane per sum");
    __shared__ uint32_t s_rows[256], s_cols[256], s_words[kReduceWords];
    __shared__ double s_joint[nwarps][kMaxQ], s_marg[nwarps][kMaxQ], s_part[nwarps][32];
    __shared__ uint32_t s_n[nwarps];
    __shared__ bool s_last;
    const int slot = blockIdx.y, p = blockIdx.x, parts = gridDim.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const Slot S0 = slots ? slots[slot] : single;
    const int t = S0.t, B = S0.bins, nq = Q.nq;
    const uint32_t *h = hist + (size_t)slot * hist_stride;
    const bool few = B * B <= 2048 * parts;  // few cells: looked up on the way
    CountTable<TB> C{few ? nullptr : s_words};
    const int c0 = (int)((long long)B * p / parts), ncols = (int)((long long)B * (p + 1) / parts) - c0;
    const int nrows = (B - p + parts - 1) / parts;
    s_cols[tid] = 0;
    C.zero();
    __syncthreads();
    bool first = true;  // the pass that takes the counts
    for (int q0 = 0; q0 < nq; q0 += 4) {
        double aj[4] = {0.0, 0.0, 0.0, 0.0};
        if (first && parts > 1)  // the column share; with one part the row pass meets every column
            for (int x = tid; x < B * ncols; x += kEntThreads) {
                const uint32_t v = __ldcg(h + (size_t)(x / ncols) * B + c0 + x % ncols);
                if (v) atomicAdd(&s_cols[x % ncols], v);
            }
        for (int i = warp; i < nrows; i += nwarps) {
            const uint32_t *row = h + (size_t)(p + parts * i) * B;
            uint32_t v[8], rsum = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = lane + 32 * k < B ? __ldcg(row + lane + 32 * k) : 0u;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (v[k] == 0) continue;
                bool taken;
                if (first) {
                    rsum += v[k];
                    if (parts == 1) atomicAdd(&s_cols[lane + 32 * k], v[k]);
                    taken = C.take(v[k]);
                } else {
                    taken = C.taken_before(v[k]);
                }
                if (!taken) CountTable<TB>::add_count(aj, v[k], q0, Q);
            }
            if (first) {
                rsum = __reduce_add_sync(kFull, rsum);
                if (lane == 0) s_rows[i] = rsum;
            }
        }
        __syncthreads();
        if (first) {
            first = false;
            if (C.overflowed()) {  // the first four q again, large counts on the way
                q0 -= 4;
                continue;
            }
            C.sort();
        }
        // marginal entries: warps 0..3 the rows, 4..7 the columns
        const uint32_t *line = warp < 4 ? s_rows : s_cols;
        const int nline = warp < 4 ? nrows : ncols;
        double m = 0.0;
        if ((warp & 3) * 32 < nline) {
            double am[4] = {0.0, 0.0, 0.0, 0.0};
            for (int i = tid & 127; i < nline; i += 128)
                if (line[i]) CountTable<TB>::add_count(am, line[i], q0, Q);
            m = warp_sum4(am);
        }
        C.add_terms(aj, q0, Q);
        const double j = warp_sum4(aj);
        if (lane < 4) {
            s_joint[warp][q0 + lane] = j;
            s_marg[warp][q0 + lane] = m;
        }
    }
    uint32_t n = 0;  // fewer than 2^31 voxels
    for (int i = tid; i < nrows; i += kEntThreads) n += s_rows[i];
    n = __reduce_add_sync(kFull, n);
    if (lane == 0) s_n[warp] = n;
    __syncthreads();
    // lane 3 iq + w of warp 0: this CTA's sum w of q iq (fixed, moving, joint); lane 3 nq: its count
    double S = 0.0;
    uint32_t N = 0;
    if (warp == 0) {
        const int iq = lane / 3, w = lane % 3;
        for (int k = 0; k < nwarps; ++k) N += s_n[k];
        if (lane < 3 * nq) {
            const double *g = &s_marg[w == 1 ? 4 : 0][iq];
            S = w == 2 ? tree8(&s_joint[0][iq], kMaxQ) : (g[0] + g[kMaxQ]) + (g[2 * kMaxQ] + g[3 * kMaxQ]);
        }
    }
    if (parts > 1) {
        double *out = part + (size_t)slot * parts * kPartStride;
        if (warp == 0 && lane <= 3 * nq) out[(size_t)p * kPartStride + lane] = lane < 3 * nq ? S : (double)N;
        __threadfence();  // this CTA's part is visible before it counts as finished
        __syncthreads();
        if (tid == 0) s_last = atomicAdd(done + slot, 1u) == (unsigned)parts - 1u;
        __syncthreads();
        if (!s_last) return;
        __threadfence();
        double a = 0.0;
        if (lane <= 3 * nq) {
#pragma unroll 4
            for (int k = warp; k < parts; k += nwarps) a += __ldcg(out + (size_t)k * kPartStride + lane);
        }
        s_part[warp][lane] = a;
        __syncthreads();
        S = tree8(&s_part[0][lane], 32);
        N = (uint32_t)__shfl_sync(kFull, S, 3 * nq);
    }
    if (warp == 0) write_mi<TB>(N, S, Q, t, O);
}

// ---------------------------------------------------------------------------
// Persistent CTAs, one work item (a whole transform, or one part of one) per CTA at a time
// ---------------------------------------------------------------------------

template <int HV, int FM>
__global__ void __launch_bounds__(1024, 1)
    k_batched(const PairDev *__restrict__ pairs, const int32_t *__restrict__ aff, const Item *__restrict__ items,
              int nitems, int *ticket, int max_bins, int rows_words, int zmax, Tile tile,
              const __grid_constant__ QSet Q, const __grid_constant__ Outputs O,
              uint32_t *__restrict__ slot_hist, long long slot_stride) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_item, s_slab;
    __shared__ int q[12];
    static_assert(sizeof s_item + sizeof s_slab + sizeof q <= kStaticSmem, "kMaxCtaSmem leaves room for these");
    const SmemLayout L = smem_layout(HV, FM, max_bins, rows_words, zmax);
    float2 *s_zoff = (float2 *)(smem + L.zoff);
    const int nwarps = blockDim.x >> 5;
    const int slabs = tile.slabs;
    int *phase = ticket + 1;  // the slab most recently started by any CTA
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(ticket, 1);
        __syncthreads();
        const int it = s_item;
        if (it >= nitems) break;
        const Item I = items[it];
        const PairDev P = pairs[I.pair];
        const int B = P.bins;
        if (threadIdx.x < 12) q[threadIdx.x] = aff[(size_t)I.t * 12 + threadIdx.x];
        load_zoff<FM>(P, s_zoff);
        auto H = make_hist<HV>(smem, L, B, O.flags, P.rows_words);
        H.load_info(P.rowinfo);
        H.zero();
        __syncthreads();
        // The sweep is cut into `slabs` slabs of row blocks, done in any order (counts do not depend
        // on it).  Each slab goes to the first remaining one at or after the slab most recently
        // started by any CTA, so CTAs working on different transforms keep to neighbouring slabs
        // of the volumes and their working set stays in L2.  No CTA waits for another.
        const int block_rows = nwarps * walk_rows_per_step(FM, tile.lpr_log2, P.srow != nullptr);
        const long long NB = ((long long)P.nf[1] * P.nf[2] + block_rows - 1) / block_rows;
        if (I.slot >= 0) {
            // one part of a transform: row blocks part, part + parts, ... (interleaved, so every part
            // meets the same share of the overlap), added to the transform's slot
            if (P.mdtype == 1)
                walk_rows<uint32_t, FM>(P, q, s_zoff, I.part, I.parts, NB, tile.lpr_log2, H);
            else
                walk_rows<uint16_t, FM>(P, q, s_zoff, I.part, I.parts, NB, tile.lpr_log2, H);
            __syncthreads();
            uint32_t *gh = slot_hist + (size_t)I.slot * slot_stride;
            for (int r = threadIdx.x >> 5; r < B; r += nwarps)
                for (int c = threadIdx.x & 31; c < B; c += 32) {
                    const uint32_t v = H.count(r, c);
                    if (v) atomicAdd(gh + r * B + c, v);
                }
            __syncthreads();
            continue;
        }
        const long long SB = (NB + slabs - 1) / slabs;
        unsigned left = (1u << slabs) - 1u;
        while (left) {
            if (threadIdx.x == 0) {
                int k = *(volatile int *)phase;
                k = k < 0 || k >= slabs ? 0 : k;
                while (!((left >> k) & 1u)) k = k + 1 == slabs ? 0 : k + 1;
                s_slab = k;
                *(volatile int *)phase = k;
            }
            __syncthreads();
            const int k = s_slab;
            left &= ~(1u << k);
            const long long b0 = (long long)k * SB, b1 = b0 + SB < NB ? b0 + SB : NB;
            if (b0 < b1) {
                if (P.mdtype == 1)
                    walk_rows<uint32_t, FM>(P, q, s_zoff, b0, 1, b1, tile.lpr_log2, H);
                else
                    walk_rows<uint16_t, FM>(P, q, s_zoff, b0, 1, b1, tile.lpr_log2, H);
            }
            __syncthreads();  // s_slab is rewritten for the next slab
        }
        __syncthreads();
        if (O.dump) {
            uint32_t *dh = O.dump + (size_t)I.t * B * B;
            for (int r = threadIdx.x >> 5; r < B; r += nwarps)
                for (int c = threadIdx.x & 31; c < B; c += 32) dh[r * B + c] = H.count(r, c);
        }
        reduce_entropies(H, P.bins, Q, (uint32_t *)(smem + L.rows), (uint32_t *)(smem + L.cols),
                         (double *)(smem + L.red), CountTable<16>{L.has_small ? (uint32_t *)(smem + L.small) : nullptr}, I.t, O);
    }
}

// ---------------------------------------------------------------------------
// Resampling v(T(x)) on the fixed grid
// ---------------------------------------------------------------------------

template <typename MovT>
__global__ void k_resample(const PairDev *__restrict__ pairs, const int32_t *__restrict__ aff, MovT *__restrict__ out) {
    const PairDev P = pairs[0];
    const long long n = (long long)P.nf[0] * P.nf[1] * P.nf[2];
    int q[12];
#pragma unroll
    for (int e = 0; e < 12; ++e) q[e] = aff[e];
    for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < n; x += (long long)gridDim.x * blockDim.x) {
        const long long i = x % P.nf[0], j = (x / P.nf[0]) % P.nf[1], k = x / ((long long)P.nf[0] * P.nf[1]);
        long long U[3];
        bool in = true;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            U[a] = (long long)q[4 * a] * i + (long long)q[4 * a + 1] * j + (long long)q[4 * a + 2] * k + q[4 * a + 3];
            in = in && U[a] >= 0 && U[a] <= ((long long)(P.nm[a] - 1) << 16);
        }
        out[x] = in ? (MovT)sample_hard<MovT>((const MovT *)P.mov, P.nm[0], P.nm[1], P.nm[2], (int)U[0], (int)U[1],
                                               (int)U[2])
                    : (MovT)0;
    }
}

inline int grid_for(long long n, int threads) {
    long long g = (n + threads - 1) / threads;
    return (int)(g < 1 ? 1 : (g > 65535 * 8 ? 65535 * 8 : g));
}

template <class K>
cudaError_t set_smem(K kernel, size_t bytes) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

}  // namespace

size_t hard_smem_bytes(int variant, int bins, int rows_words, int zmax) {
    return smem_layout(hv_kind(variant), hv_fetch(variant), bins, rows_words, zmax).total;
}

// MurmurHash3's 32-bit finalizer: xor-shift 16, multiply 0x85ebca6b, xor-shift 13, multiply 0xc2b2ae35,
// xor-shift 16 (mod 2^32).
__host__ __device__ inline uint32_t fmix32(uint32_t k) {
    k ^= k >> 16;
    k *= 0x85ebca6bu;
    k ^= k >> 13;
    k *= 0xc2b2ae35u;
    k ^= k >> 16;
    return k;
}

// One thread per fixed row: how many of its voxels are sampled (hseed = fmix32(seed)).
__global__ void k_sample_count(int n0, long long R, uint32_t hseed, uint32_t thr, uint32_t *__restrict__ counts) {
    for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < R; r += (long long)gridDim.x * blockDim.x) {
        uint32_t c = 0;
        const uint32_t x0 = (uint32_t)(r * n0);
        for (int i = 0; i < n0; ++i) c += fmix32((x0 + (uint32_t)i) ^ hseed) < thr ? 1u : 0u;
        counts[r] = c;
    }
}

// One thread per fixed row: its sampled voxels' x indices (ascending) and fixed bins.
__global__ void k_sample_fill(int n0, long long R, uint32_t hseed, uint32_t thr, const uint8_t *__restrict__ fbins,
                              const uint32_t *__restrict__ row_ptr, uint16_t *__restrict__ cols,
                              uint8_t *__restrict__ bins) {
    for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < R; r += (long long)gridDim.x * blockDim.x) {
        uint32_t o = row_ptr[r];
        const uint32_t x0 = (uint32_t)(r * n0);
        for (int i = 0; i < n0; ++i)
            if (fmix32((x0 + (uint32_t)i) ^ hseed) < thr) {
                cols[o] = (uint16_t)i;
                bins[o] = fbins[(size_t)r * n0 + i];
                ++o;
            }
    }
}

cudaError_t launch_sample_count(int n0, long long R, uint32_t seed, uint32_t threshold, uint32_t *counts,
                                cudaStream_t s) {
    k_sample_count<<<grid_for(R, 256), 256, 0, s>>>(n0, R, fmix32(seed), threshold, counts);
    return cudaGetLastError();
}

cudaError_t launch_sample_fill(int n0, long long R, uint32_t seed, uint32_t threshold, const uint8_t *fbins,
                               const uint32_t *row_ptr, uint16_t *cols, uint8_t *bins, cudaStream_t s) {
    k_sample_fill<<<grid_for(R, 256), 256, 0, s>>>(n0, R, fmix32(seed), threshold, fbins, row_ptr, cols, bins);
    return cudaGetLastError();
}

cudaError_t launch_f32_to_u16(const float *in, long long n, uint16_t *out, cudaStream_t s) {
    k_f32_to_u16<<<grid_for(n, 256), 256, 0, s>>>(in, n, out);
    return cudaGetLastError();
}

// Blocks of 256 threads for n elements, eight a thread, at most eight blocks an SM.
static int eight_grid(long long n) {
    const long long g = (n + 2047) / 2048;
    return (int)(g < 1 ? 1 : (g > 8 * 152 ? 8 * 152 : g));
}

cudaError_t launch_copy_clamp(const void *in, int dtype, int depth, long long n, void *out, cudaStream_t s) {
    const uint32_t vmax = (uint32_t)((1ull << depth) - 1ull);
    if (dtype == 0)
        k_copy_clamp<uint8_t><<<eight_grid(n), 256, 0, s>>>((const uint8_t *)in, n, vmax, aligned8<uint8_t>(in), (uint8_t *)out);
    else
        k_copy_clamp<uint16_t><<<eight_grid(n), 256, 0, s>>>((const uint16_t *)in, n, vmax, aligned8<uint16_t>(in),
                                                             (uint16_t *)out);
    return cudaGetLastError();
}

cudaError_t launch_make_pairs(const void *mov, int dtype, const int nm[3], void *out, cudaStream_t s) {
    const long long n = (long long)nm[0] * (nm[1] + 1) * (nm[2] + 1);
    if (dtype == 0)
        k_make_pairs<uint8_t, uint16_t><<<grid_for(n, 256), 256, 0, s>>>((const uint8_t *)mov, nm[0], nm[1], nm[2],
                                                                          (uint16_t *)out);
    else
        k_make_pairs<uint16_t, uint32_t><<<grid_for(n, 256), 256, 0, s>>>((const uint16_t *)mov, nm[0], nm[1], nm[2],
                                                                           (uint32_t *)out);
    return cudaGetLastError();
}

cudaError_t launch_make_zpairs(const void *mov, int dtype, const int nm[3], int ph, cudaSurfaceObject_t out,
                               cudaStream_t s) {
    const dim3 grid((nm[0] + 31) / 32, (nm[1] + 7) / 8, nm[2]), block(32, 8);
    if (dtype == 0)
        k_make_zpairs<uint8_t><<<grid, block, 0, s>>>((const uint8_t *)mov, nm[0], nm[1], nm[2], ph, out);
    else
        k_make_zpairs<uint16_t><<<grid, block, 0, s>>>((const uint16_t *)mov, nm[0], nm[1], nm[2], ph, out);
    return cudaGetLastError();
}

cudaError_t launch_make_quads(const void *mov, int dtype, const int nm[3], cudaSurfaceObject_t out, cudaStream_t s) {
    const dim3 grid((nm[0] + 31) / 32, (nm[1] + 7) / 8, nm[2]), block(32, 8);
    if (dtype == 0)
        k_make_quads<uint8_t><<<grid, block, 0, s>>>((const uint8_t *)mov, nm[0], nm[1], nm[2], out);
    else
        k_make_quads<uint16_t><<<grid, block, 0, s>>>((const uint16_t *)mov, nm[0], nm[1], nm[2], out);
    return cudaGetLastError();
}

cudaError_t launch_bin_fixed(const void *data, int dtype, int depth, long long n, int bins, uint8_t *out,
                             unsigned long long *counts, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(counts, 0, (size_t)bins * sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    if (dtype == 0)
        k_bin_fixed<uint8_t><<<eight_grid(n), 256, 0, s>>>((const uint8_t *)data, n, depth, bins, aligned8<uint8_t>(data), out,
                                                           counts);
    else
        k_bin_fixed<uint16_t><<<eight_grid(n), 256, 0, s>>>((const uint16_t *)data, n, depth, bins, aligned8<uint16_t>(data),
                                                            out, counts);
    return cudaGetLastError();
}

cudaError_t launch_table(double *tab, float q, cudaStream_t s) {
    k_table<<<kTab / 256, 256, 0, s>>>(tab, q);
    return cudaGetLastError();
}

// Every variant as (public value, counter kind, fetch mode).
#define MI_VARIANTS(X)                                                                              \
    X(HV_U32, HV_U32, FM_LDG) X(HV_U32_MATCH, HV_U32_MATCH, FM_LDG) X(HV_U16, HV_U16, FM_LDG)        \
    X(HV_U16_MATCH, HV_U16_MATCH, FM_LDG) X(HV_TEX + HV_U32, HV_U32, FM_TEX)                        \
    X(HV_TEX + HV_U32_MATCH, HV_U32_MATCH, FM_TEX) X(HV_TEX + HV_U16, HV_U16, FM_TEX)                \
    X(HV_TEX + HV_U16_MATCH, HV_U16_MATCH, FM_TEX) X(HV_ROWS, HV_ROWS, FM_LDG)                      \
    X(HV_ROWS_TEX, HV_ROWS, FM_TEX)                                                                 \
    X(HV_ROWS_QUAD, HV_ROWS, FM_QUAD) X(HV_U32_QUAD, HV_U32, FM_QUAD) X(HV_U16_QUAD, HV_U16, FM_QUAD) \
    X(HV_ROWS_GATHER, HV_ROWS, FM_GATHER) X(HV_U32_GATHER, HV_U32, FM_GATHER)                       \
    X(HV_U16_GATHER, HV_U16, FM_GATHER)

cudaError_t launch_entropy_slots(const uint32_t *d_hist, long long hist_stride, const Slot *d_slots, int nslots,
                                 int parts, const QSet &Q, unsigned int *d_done, double *d_part, const Outputs &O,
                                 cudaStream_t s) {
    k_entropy_slots<16><<<dim3(parts, nslots), kEntThreads, 0, s>>>(d_hist, hist_stride, d_slots, Slot{}, Q, d_done,
                                                                    d_part, O);
    return cudaGetLastError();
}

// Parts per slot: about two CTAs an SM over all slots (more would only repeat the reductions, whose FP64
// additions bound a launch over many slots), each of at least eight rows (one per warp).
int entropy_parts(int max_bins, int nslots, int sms) {
    const int most = (max_bins + 7) / 8, want = (2 * sms + nslots - 1) / nslots;
    return want < most ? want : most;
}
size_t entropy_part_bytes(int parts, int nslots) { return (size_t)parts * nslots * kPartStride * sizeof(double); }

static const void *batched_fn(int variant) {
    switch (variant) {
#define MI_BATCHED_CASE(V, K, F) \
    case V: return (const void *)k_batched<K, F>;
        MI_VARIANTS(MI_BATCHED_CASE)
#undef MI_BATCHED_CASE
        default: return nullptr;
    }
}

int batched_ctas_per_sm(int variant, int max_bins, int threads, int rows_words, int zmax) {
    const size_t smem = hard_smem_bytes(variant, max_bins, rows_words, zmax);
    const void *fn = batched_fn(variant);
    if (!fn) return 0;
    int nb = 0;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, threads, smem) != cudaSuccess) {
        cudaGetLastError();  // the answer is "none": the next launch's check must not find this error
        return 0;
    }
    return nb;
}

cudaError_t launch_batched(const PairDev *d_pairs, const int32_t *d_aff, const Item *d_items, int nitems,
                           int *d_ticket, int max_bins, int rows_words, int zmax, int variant, int threads, int ctas,
                           Tile tile, const QSet &Q, const Outputs &O, uint32_t *slot_hist, long long slot_stride,
                           cudaStream_t s) {
    const size_t smem = hard_smem_bytes(variant, max_bins, rows_words, zmax);
    const void *fn = batched_fn(variant);
    if (!fn) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    void *args[] = {(void *)&d_pairs, (void *)&d_aff, (void *)&d_items, (void *)&nitems, (void *)&d_ticket,
                    (void *)&max_bins, (void *)&rows_words, (void *)&zmax, (void *)&tile, (void *)&Q, (void *)&O,
                    (void *)&slot_hist, (void *)&slot_stride};
    return cudaLaunchKernel(fn, dim3(ctas < nitems ? ctas : nitems), dim3(threads), args, smem, s);
}

cudaError_t launch_resample(const PairDev *d_pair, const PairDev &h_pair, const int32_t *d_aff, void *out,
                            cudaStream_t s) {
    const long long n = (long long)h_pair.nf[0] * h_pair.nf[1] * h_pair.nf[2];
    if (h_pair.mdtype == 0)
        k_resample<uint8_t><<<grid_for(n, 256), 256, 0, s>>>(d_pair, d_aff, (uint8_t *)out);
    else
        k_resample<uint16_t><<<grid_for(n, 256), 256, 0, s>>>(d_pair, d_aff, (uint16_t *)out);
    return cudaGetLastError();
}

cudaError_t set_drain_cap(int cap) { return cudaMemcpyToSymbol(g_drain_cap, &cap, sizeof cap); }

}  // namespace mi

// ===========================================================================
// Allocation-free variant of the plain path (entry point in mi_noalloc.cu):
// the fixed volume is binned on the fly from its raw values, and the
// histogram, the entropy tables (256 entries a q) and the partial sums live
// in caller-provided scratch (a static device array).
// ===========================================================================

namespace mi {
namespace {

struct RawPair {
    const void *fix;
    const void *mov;
    int nf[3], nm[3];
    int bins, fdepth, mdepth;
};

struct Q12 {
    int q[12];
};

// sample_hard on a volume used as given: each of the 8 neighbours is clamped to vmax = 2^d - 1 as it
// is read, as the context path clamps every voxel when it copies the volume.
template <typename MovT>
__device__ __forceinline__ int sample_hard_raw(const MovT *__restrict__ mov, int n0, int n1, int n2, int ux, int uy,
                                               int uz, int vmax) {
    const int ix = ux >> 16, iy = uy >> 16, iz = uz >> 16;
    const int fx = (ux >> 8) & 255, fy = (uy >> 8) & 255, fz = (uz >> 8) & 255;
    const int sx = ix < n0 - 1 ? 1 : 0;
    const int sy = iy < n1 - 1 ? n0 : 0;
    const int sz = iz < n2 - 1 ? n0 * n1 : 0;
    const MovT *p = mov + (ix + n0 * (iy + n1 * iz));
    const int v000 = min((int)__ldg(p), vmax), v001 = min((int)__ldg(p + sx), vmax);
    const int v010 = min((int)__ldg(p + sy), vmax), v011 = min((int)__ldg(p + sy + sx), vmax);
    const int v100 = min((int)__ldg(p + sz), vmax), v101 = min((int)__ldg(p + sz + sx), vmax);
    const int v110 = min((int)__ldg(p + sz + sy), vmax), v111 = min((int)__ldg(p + sz + sy + sx), vmax);
    const int e00 = lerp8(v000, v001, fx), e01 = lerp8(v010, v011, fx);
    const int e10 = lerp8(v100, v101, fx), e11 = lerp8(v110, v111, fx);
    const int g0 = lerp8(e00, e01, fy), g1 = lerp8(e10, e11, fy);
    return lerp8(g0, g1, fz);
}

// Warp w of all takes rows w, w + warps, ...; 32 of them are clipped at once (lane l: its l-th).
template <typename FixT, typename MovT, class Hist>
__device__ void accumulate_rows_raw(const RawPair &P, const int *q, Hist &H) {
    const int lane = threadIdx.x & 31;
    const int nf0 = P.nf[0], nf1 = P.nf[1];
    const long long R = (long long)nf1 * P.nf[2];
    const long long first = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5,
                    warps = ((long long)gridDim.x * blockDim.x) >> 5;
    const int n0 = P.nm[0], n1 = P.nm[1], n2 = P.nm[2];
    const int st0 = q[0], st1 = q[4], st2 = q[8];
    const int bins = P.bins, mdepth = P.mdepth, fdepth = P.fdepth;
    const uint32_t fvmax = (uint32_t)((1ull << fdepth) - 1ull);
    const int vmax = (int)((1u << mdepth) - 1u);
    const MovT *__restrict__ mov = (const MovT *)P.mov;
    for (long long rb = first; rb < R; rb += 32 * warps) {
        RowClip mine;
        mine.lo = 0;
        mine.hi = -1;
        mine.u0 = mine.u1 = mine.u2 = 0;
        const long long rl = rb + lane * warps;
        if (rl < R) mine = clip_row(q, (int)rl % nf1, (int)rl / nf1, nf0, P.nm);
        for (int s = 0; s < 32; ++s) {
            const long long r = rb + s * warps;
            if (r >= R) break;  // warp-uniform
            const int lo = __shfl_sync(kFull, mine.lo, s), hi = __shfl_sync(kFull, mine.hi, s);
            if (lo > hi) continue;
            const int U0 = __shfl_sync(kFull, mine.u0, s), U1 = __shfl_sync(kFull, mine.u1, s),
                      U2 = __shfl_sync(kFull, mine.u2, s);
            const FixT *__restrict__ frow = (const FixT *)P.fix + (size_t)r * nf0;
#pragma unroll 2
            for (int i = lo + lane; i <= hi; i += 32) {
                const int d = i - lo;
                // volumes are read in place; each value is clamped to its bit depth as it is read
                const int v = sample_hard_raw<MovT>(mov, n0, n1, n2, U0 + st0 * d, U1 + st1 * d, U2 + st2 * d, vmax);
                uint32_t fv = (uint32_t)__ldg(frow + i);
                fv = fv > fvmax ? fvmax : fv;
                H.add((int)((fv * (uint32_t)bins) >> fdepth), (v * bins) >> mdepth, true);
            }
        }
    }
}

// 32-bit counters up to kRawU32Bins bins, drained 16-bit ones above (where the 32-bit ones leave the L1
// too little for the volumes, then do not fit).  What bounds it is the latency of the eight scattered
// loads a voxel, so every warp of every SM takes rows: with batches of 32 rows a warp, a 192 x 192 x 128
// volume's 24576 rows occupied 768 of the 4864 warps and the kernel took 148 us; now 33.
// The first lanes of each CTA build the entropy tables on the way.
constexpr int kRawU32Bins = 160;

template <typename FixT, typename MovT, int HV>
__global__ void __launch_bounds__(1024, 1)
    k_hist_raw(RawPair P, Q12 A, const __grid_constant__ QSet Q, NoallocScratch *__restrict__ D) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int B = P.bins;
    const SmemLayout L = smem_layout(HV, FM_LDG, B, 0, 0);
    __shared__ int q[12];
    if (threadIdx.x < 12) q[threadIdx.x] = A.q[threadIdx.x];
    auto H = make_hist<HV>(smem, L, B, D->flags);
    H.zero();
    // entry c < 256: c ln c or c^q; entry 256 + i: that of 2^(8 + i)
    constexpr int entries = 256 + 16;
    for (int x = threadIdx.x * gridDim.x + blockIdx.x; x < entries * Q.nq; x += blockDim.x * gridDim.x) {
        const int iq = x / entries, c = x % entries;
        const double d = c < 256 ? (double)c : (double)(1u << (c - 248));
        D->tab[iq][c] = c == 0 ? 0.0 : Q.q[iq] == 1.0f ? d * log(d) : pow(d, (double)Q.q[iq]);
    }
    __syncthreads();
    const int nwarps = blockDim.x >> 5;
    accumulate_rows_raw<FixT, MovT>(P, q, H);
    __syncthreads();
    for (int r = threadIdx.x >> 5; r < B; r += nwarps)
        for (int c = threadIdx.x & 31; c < B; c += 32) {
            const uint32_t v = H.count(r, c);
            if (v) atomicAdd(D->hist + r * B + c, v);
        }
}

}  // namespace

cudaError_t launch_noalloc_eval(const void *fix, int fdtype, int fdepth, const void *mov, int mdtype, int mdepth,
                                const int nf[3], const int nm[3], int bins, const int32_t q16[12], QSet Q,
                                NoallocScratch *d, int sms, cudaStream_t s) {
    RawPair P;
    P.fix = fix;
    P.mov = mov;
    for (int a = 0; a < 3; ++a) {
        P.nf[a] = nf[a];
        P.nm[a] = nm[a];
    }
    P.bins = bins;
    P.fdepth = fdepth;
    P.mdepth = mdepth;
    Q12 A;
    for (int e = 0; e < 12; ++e) A.q[e] = q16[e];
    for (int i = 0; i < Q.nq; ++i) Q.tab[i] = d->tab[i];
    const int threads = 1024;
    const long long rows = (long long)nf[1] * nf[2], all = (rows + 31) / 32;  // a row a warp at least
    const int ctas = (int)(all < sms ? all : sms);
    const bool u32 = bins <= kRawU32Bins;
    const size_t smem = smem_layout(u32 ? HV_U32 : HV_U16, FM_LDG, bins, 0, 0).total;
    cudaError_t e = cudaMemsetAsync(d, 0, offsetof(NoallocScratch, hist) + (size_t)bins * bins * sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
#define MI_RAW_H(FT, MT, HV)                                                                \
    do {                                                                                   \
        if ((e = set_smem(k_hist_raw<FT, MT, HV>, smem)) != cudaSuccess) return e;         \
        k_hist_raw<FT, MT, HV><<<ctas, threads, smem, s>>>(P, A, Q, d);                    \
    } while (0)
#define MI_RAW(FT, MT)                  \
    do {                                \
        if (u32) MI_RAW_H(FT, MT, HV_U32); \
        else MI_RAW_H(FT, MT, HV_U16);  \
    } while (0)
    if (fdtype == 0 && mdtype == 0) MI_RAW(uint8_t, uint8_t);
    else if (fdtype == 0) MI_RAW(uint8_t, uint16_t);
    else if (mdtype == 0) MI_RAW(uint16_t, uint8_t);
    else MI_RAW(uint16_t, uint16_t);
#undef MI_RAW
#undef MI_RAW_H
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    Outputs O;
    O.mi = d->mi;
    O.h = nullptr;
    O.count = nullptr;
    O.dump = nullptr;
    O.flags = d->flags;
    k_entropy_slots<8><<<dim3(entropy_parts(bins, 1, sms), 1), kEntThreads, 0, s>>>(d->hist, 0, nullptr, Slot{0, bins}, Q,
                                                                                    &d->done, d->part, O);
    return cudaGetLastError();
}

}  // namespace mi
