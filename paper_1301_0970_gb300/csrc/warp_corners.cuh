// Trilinear warp of the moving image and of the structure terms at one
// point (the first pass of the two-pass force, Algorithm A steps 5-6 of
// Sec. 2.2): the eight corners' values and mask bits are loaded, then I0~,
// the corners' bit AND / OR and, where the corners disagree on bit j, P_j
// are written to the two-pass scratch of ForceArgs.  Shared by the force
// kernels and the fused smoothing + warp kernel, so both give the same bits.
#pragma once

#include "cgdir_internal.cuh"

namespace cgdir {

// One interpolation point: the weights and the linear indices of the low
// corners of its two planes (lo, hi; equal at the last plane), and the index
// steps to the high corners in x and y (0 at the border).
struct Cell {
    float wx, wy, wz;
    int lo, hi, dx, dy;
};

// The four corners of one plane of a cell, loaded.  Values of 16-bit images
// stay raw until corner_finish converts them: a conversion at the load would
// wait for the load there, before the other gathers of the thread are issued.
//   c  values (float images)
//   m  float images: the corners' moving-mask bits; 16-bit images: the raw
//      value in the low half, mask bits in bits 16-23 (the texel word)
template <typename IT>
struct CornerQuad {
    float c[4];
    unsigned m[4];
};

// The float value of a raw 16-bit image value (the low half of w).
template <typename IT>
__device__ __forceinline__ float from_raw16(unsigned w);
template <>
__device__ __forceinline__ float from_raw16<__half>(unsigned w) { return __half2float(__ushort_as_half((unsigned short)w)); }
template <>
__device__ __forceinline__ float from_raw16<__nv_bfloat16>(unsigned w) {
    return __uint_as_float(w << 16);        // a bfloat16 is the high half of a float
}
template <>
__device__ __forceinline__ float from_raw16<float>(unsigned w) { return __uint_as_float(w); }   // not used

// Clamp x + u and find the corners.
__device__ __forceinline__ Cell corner_cell(const ForceArgs &a, float ux, float uy, float uz, int x, int y, int z) {
    const int nx = a.nx, ny = a.ny, nz = a.nz, nxy = nx * ny;
    const float px = fminf(fmaxf((float)x + ux, 0.f), (float)(nx - 1));
    const float py = fminf(fmaxf((float)y + uy, 0.f), (float)(ny - 1));
    const float pz = fminf(fmaxf((float)z + uz, 0.f), (float)(nz - 1));
    const float fx = floorf(px), fy = floorf(py), fz = floorf(pz);
    const int ix = (int)fx, iy = (int)fy, iz = (int)fz;
    Cell w;
    w.wx = px - fx; w.wy = py - fy; w.wz = pz - fz;
    w.dx = ix < nx - 1 ? 1 : 0; w.dy = iy < ny - 1 ? nx : 0;
    w.lo = iz * nxy + iy * nx + ix;
    w.hi = w.lo + (iz < nz - 1 ? nxy : 0);
    return w;
}

// Issue the loads of the four corners b, b + dx, b + dy, b + dy + dx of one
// plane (texels when the structure terms are on, else image values).
template <bool CONTOUR, typename IT>
__device__ __forceinline__ void corner_quad(const ForceArgs &a, int b, int dx, int dy, CornerQuad<IT> &cs) {
    const int o[4] = {0, dx, dy, dy + dx};
    const void *base = CONTOUR ? a.mtex : a.I0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (sizeof(IT) == 2) {
            cs.m[q] = CONTOUR ? (unsigned)__ldg(static_cast<const uint32_t *>(base) + b + o[q])
                              : (unsigned)__ldg(static_cast<const unsigned short *>(base) + b + o[q]);
        } else if (CONTOUR) {
            const float2 t = __ldg(static_cast<const float2 *>(base) + b + o[q]);
            cs.c[q] = t.x;
            cs.m[q] = __float_as_uint(t.y);
        } else {
            cs.c[q] = __ldg(static_cast<const float *>(base) + b + o[q]);
        }
    }
}

template <typename IT>
__device__ __forceinline__ float corner_value(const CornerQuad<IT> &cs, int q) {
    return sizeof(IT) == 4 ? cs.c[q] : from_raw16<IT>(cs.m[q]);
}

// Interpolate I0~ at voxel i from the loaded corners of the cell's low and
// high plane, write it, the corner bits' AND / OR and, where they disagree, P_j.
template <bool CONTOUR, typename IT>
__device__ __forceinline__ void corner_finish(const ForceArgs &a, int i, int N, const Cell &w,
                                              const CornerQuad<IT> &lo, const CornerQuad<IT> &hi) {
    const float wx = w.wx, wy = w.wy, wz = w.wz;
    float c[8];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        c[q] = corner_value<IT>(lo, q);
        c[4 + q] = corner_value<IT>(hi, q);
    }
    const float e00 = fmaf(wx, c[1] - c[0], c[0]), e10 = fmaf(wx, c[3] - c[2], c[2]);
    const float e01 = fmaf(wx, c[5] - c[4], c[4]), e11 = fmaf(wx, c[7] - c[6], c[6]);
    const float f0 = fmaf(wy, e10 - e00, e00), f1 = fmaf(wy, e11 - e01, e01);
    a.wfield[i] = fmaf(wz, f1 - f0, f0);
    if (CONTOUR) {
        unsigned m[8];
#pragma unroll
        for (int q = 0; q < 4; ++q) { m[q] = lo.m[q]; m[4 + q] = hi.m[q]; }
        constexpr int sh = sizeof(IT) == 2 ? 16 : 0;      // where the mask bits lie in m
        // the words hold nothing above the mask bits (texel bits 24-31 are zero)
        const unsigned andb = (m[0] & m[1] & m[2] & m[3] & m[4] & m[5] & m[6] & m[7]) >> sh;
        const unsigned orb = (m[0] | m[1] | m[2] | m[3] | m[4] | m[5] | m[6] | m[7]) >> sh;
        a.wstate[i] = (uint16_t)((andb << 8) | orb);
        unsigned mixed = orb & ~andb;
        if (mixed) {
            const float off = a.offset;
            const float ax = 1.f - wx, ay = 1.f - wy, az = 1.f - wz;
            // products rounded on their own (never contracted into the sums
            // below), so every kernel that inlines this gives the same bits
            auto w3 = [](float p, float q, float r, float v) { return __fmul_rn(__fmul_rn(__fmul_rn(p, q), r), v); };
            float q[8];
            q[0] = w3(ax, ay, az, c[0] + off); q[1] = w3(wx, ay, az, c[1] + off);
            q[2] = w3(ax, wy, az, c[2] + off); q[3] = w3(wx, wy, az, c[3] + off);
            q[4] = w3(ax, ay, wz, c[4] + off); q[5] = w3(wx, ay, wz, c[5] + off);
            q[6] = w3(ax, wy, wz, c[6] + off); q[7] = w3(wx, wy, wz, c[7] + off);
            while (mixed) {
                const int j = __ffs(mixed) - 1;
                mixed &= mixed - 1u;
                float pj = 0.f;
#pragma unroll
                for (int t = 0; t < 8; ++t) pj += ((m[t] >> (sh + j)) & 1u) ? q[t] : 0.f;
                a.pfield[(size_t)j * N + i] = pj;
            }
        }
    }
}

}  // namespace cgdir
