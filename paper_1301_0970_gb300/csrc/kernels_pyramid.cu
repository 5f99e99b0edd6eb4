// Set-up kernels of CG-DIR: mask bit-packing, the factor-2 image pyramid and
// the prolongation of the DVF between levels (multi-scale strategy,
// Sec. 2.2), the UROI map of the stopping criterion (Sec. 2.2), the sums
// behind the automatic sign of the modified images (Sec. 2.1) and image
// type conversion.  None of these run per iteration.
#include "cgdir_internal.cuh"

#include <algorithm>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

namespace cgdir {

namespace {

unsigned flat_grid(size_t n, size_t cap = 152 * 16) {
    size_t g = (n + 255) / 256;
    if (g > cap) g = cap;
    return (unsigned)(g ? g : 1);
}

// Row launches: a CTA covers RB consecutive x of one (y, z) row, so no
// index is recovered by division (the grid-stride loops above divide a
// 64-bit index per voxel).  Volumes with ny or nz above the grid limit keep
// the grid-stride kernels.
constexpr int RB = 128;
bool rows_ok(int ny, int nz) { return ny <= 65535 && nz <= 65535; }
dim3 row_grid(int nx, int ny, int nz) { return dim3((unsigned)((nx + RB - 1) / RB), (unsigned)ny, (unsigned)nz); }

struct MaskPtrs {
    const uint8_t *p[kMaxMasks];
};

// Four voxels per thread: one 32-bit load per mask, a byte-wise nonzero test.
__global__ void k_pack4(MaskPtrs m, int k, size_t n4, uint32_t *__restrict__ bits) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4;
         i += (size_t)gridDim.x * blockDim.x) {
        uint32_t b = 0;
#pragma unroll
        for (int j = 0; j < kMaxMasks; ++j)
            if (j < k) b |= __vcmpne4(__ldg(reinterpret_cast<const uint32_t *>(m.p[j]) + i), 0u) & (0x01010101u << j);
        bits[i] = b;
    }
}

// Sixteen voxels per thread (16-byte loads, all masks' in flight together).
__global__ void k_pack16(MaskPtrs m, int k, size_t n16, uint4 *__restrict__ bits) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n16) return;
    uint4 w[kMaxMasks];
#pragma unroll
    for (int j = 0; j < kMaxMasks; ++j)
        if (j < k) w[j] = __ldg(reinterpret_cast<const uint4 *>(m.p[j]) + i);
    uint4 b = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int j = 0; j < kMaxMasks; ++j)
        if (j < k) {
            const uint32_t one = 0x01010101u << j;
            b.x |= __vcmpne4(w[j].x, 0u) & one; b.y |= __vcmpne4(w[j].y, 0u) & one;
            b.z |= __vcmpne4(w[j].z, 0u) & one; b.w |= __vcmpne4(w[j].w, 0u) & one;
        }
    bits[i] = b;
}

__global__ void k_pack(MaskPtrs m, int k, size_t n, uint8_t *__restrict__ bits) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x) {
        unsigned b = 0;
#pragma unroll
        for (int j = 0; j < kMaxMasks; ++j)
            if (j < k && __ldg(m.p[j] + i)) b |= 1u << j;
        bits[i] = (uint8_t)b;
    }
}

// 2x2x2 box mean, source indices clamped (odd sizes replicate the border),
// accumulated in float32 and stored in the output level's image type.
template <typename IT, typename OT>
__global__ void k_restrict_image(const IT *__restrict__ in, int nx, int ny, int nz,
                                 OT *__restrict__ out) {
    const int cx = (nx + 1) / 2, cy = (ny + 1) / 2, cz = (nz + 1) / 2;
    const size_t Nc = (size_t)cx * cy * cz;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < Nc;
         i += (size_t)gridDim.x * blockDim.x) {
        const int X = (int)(i % cx), Y = (int)((i / cx) % cy), Z = (int)(i / ((size_t)cx * cy));
        float s = 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int x = min(2 * X + (q & 1), nx - 1), y = min(2 * Y + ((q >> 1) & 1), ny - 1),
                      z = min(2 * Z + ((q >> 2) & 1), nz - 1);
            s += ld_img<IT>(in + vox(x, y, z, nx, ny));
        }
        out[i] = from_f<OT>(s * 0.125f);
    }
}

// The same box mean per coarse row (X = thread, Y, Z = grid).
template <typename IT, typename OT>
__global__ void k_restrict_image_rows(const IT *__restrict__ in, int nx, int ny, int nz, OT *__restrict__ out) {
    const int cx = (nx + 1) / 2, cy = (ny + 1) / 2;
    const int X = blockIdx.x * RB + threadIdx.x, Y = blockIdx.y, Z = blockIdx.z;
    if (X >= cx) return;
    float s = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int x = min(2 * X + (q & 1), nx - 1), y = min(2 * Y + ((q >> 1) & 1), ny - 1),
                  z = min(2 * Z + ((q >> 2) & 1), nz - 1);
        s += ld_img<IT>(in + vox(x, y, z, nx, ny));
    }
    out[vox(X, Y, Z, cx, cy)] = from_f<OT>(s * 0.125f);
}

// The same where nx is even and rows are aligned for pairs: the two x
// neighbours come by one load, a coarse value's four pairs are in flight.
template <typename IT>
struct PairOf { using type = unsigned; };
template <>
struct PairOf<float> { using type = float2; };
__device__ __forceinline__ float2 pair_f(float2 v, float) { return v; }
__device__ __forceinline__ float2 pair_f(unsigned v, __half) {
    return make_float2(from_bits16<__half>(v & 0xffffu), from_bits16<__half>(v >> 16));
}
__device__ __forceinline__ float2 pair_f(unsigned v, __nv_bfloat16) {
    return make_float2(from_bits16<__nv_bfloat16>(v & 0xffffu), from_bits16<__nv_bfloat16>(v >> 16));
}
template <typename IT, typename OT>
__global__ void k_restrict_image_pairs(const IT *__restrict__ in, int nx, int ny, int nz, OT *__restrict__ out) {
    using PT = typename PairOf<IT>::type;
    const int cx = nx / 2, cy = (ny + 1) / 2;
    const int X = blockIdx.x * RB + threadIdx.x, Y = blockIdx.y, Z = blockIdx.z;
    if (X >= cx) return;
    const int y1 = min(2 * Y + 1, ny - 1), z1 = min(2 * Z + 1, nz - 1);
    PT p[4];
    p[0] = __ldg(reinterpret_cast<const PT *>(in + vox(2 * X, 2 * Y, 2 * Z, nx, ny)));
    p[1] = __ldg(reinterpret_cast<const PT *>(in + vox(2 * X, y1, 2 * Z, nx, ny)));
    p[2] = __ldg(reinterpret_cast<const PT *>(in + vox(2 * X, 2 * Y, z1, nx, ny)));
    p[3] = __ldg(reinterpret_cast<const PT *>(in + vox(2 * X, y1, z1, nx, ny)));
    float s = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float2 v = pair_f(p[q], IT());
        s += v.x;
        s += v.y;
    }
    out[vox(X, Y, Z, cx, cy)] = from_f<OT>(s * 0.125f);
}

// Per bit: inside if at least 4 of the 8 source voxels are inside.
__global__ void k_restrict_bits(const uint8_t *__restrict__ in, int nx, int ny, int nz,
                                uint8_t *__restrict__ out) {
    const int cx = (nx + 1) / 2, cy = (ny + 1) / 2, cz = (nz + 1) / 2;
    const size_t Nc = (size_t)cx * cy * cz;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < Nc;
         i += (size_t)gridDim.x * blockDim.x) {
        const int X = (int)(i % cx), Y = (int)((i / cx) % cy), Z = (int)(i / ((size_t)cx * cy));
        int cnt[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int x = min(2 * X + (q & 1), nx - 1), y = min(2 * Y + ((q >> 1) & 1), ny - 1),
                      z = min(2 * Z + ((q >> 2) & 1), nz - 1);
            const unsigned b = __ldg(in + vox(x, y, z, nx, ny));
#pragma unroll
            for (int j = 0; j < 8; ++j) cnt[j] += (b >> j) & 1u;
        }
        unsigned o = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) o |= (cnt[j] >= 4 ? 1u : 0u) << j;
        out[i] = (uint8_t)o;
    }
}

// (256x256x96: 11.6 -> 5.2 us against the loop over bits below.)
// Eight fine voxels of a row (one 8-byte load from each of the 2 x 2 rows) to
// four coarse ones, nx % 8 == 0: the eight bytes of a coarse voxel are added
// bit by bit with carry-save adders on 16-bit lanes (two coarse voxels per
// word); the count is at least 4 where two of the four carries (worth 2
// each) are set.
__device__ __forceinline__ uint32_t majority8(const uint32_t *a) {
    auto carry = [](uint32_t x, uint32_t y, uint32_t z) { return (x & y) | (z & (x ^ y)); };
    const uint32_t s1 = a[0] ^ a[1] ^ a[2], c1 = carry(a[0], a[1], a[2]);
    const uint32_t s2 = a[3] ^ a[4] ^ a[5], c2 = carry(a[3], a[4], a[5]);
    const uint32_t s3 = a[6] ^ a[7], c3 = a[6] & a[7];
    const uint32_t c4 = carry(s1, s2, s3);
    return (c1 & c2) | (c3 & c4) | ((c1 | c2) & (c3 | c4));
}
__global__ void k_restrict_bits8(const uint8_t *__restrict__ in, int nx, int ny, int nz, uint8_t *__restrict__ out) {
    const int cx = nx / 2, cy = (ny + 1) / 2;
    const int g = blockIdx.x * RB + threadIdx.x, Y = blockIdx.y, Z = blockIdx.z;
    if (8 * g >= nx) return;
    const int y1 = min(2 * Y + 1, ny - 1), z1 = min(2 * Z + 1, nz - 1);
    uint2 r[4];
    r[0] = __ldg(reinterpret_cast<const uint2 *>(in + vox(8 * g, 2 * Y, 2 * Z, nx, ny)));
    r[1] = __ldg(reinterpret_cast<const uint2 *>(in + vox(8 * g, y1, 2 * Z, nx, ny)));
    r[2] = __ldg(reinterpret_cast<const uint2 *>(in + vox(8 * g, 2 * Y, z1, nx, ny)));
    r[3] = __ldg(reinterpret_cast<const uint2 *>(in + vox(8 * g, y1, z1, nx, ny)));
    uint32_t lo[8], hi[8];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        lo[2 * q] = r[q].x & 0x00ff00ffu; lo[2 * q + 1] = (r[q].x >> 8) & 0x00ff00ffu;
        hi[2 * q] = r[q].y & 0x00ff00ffu; hi[2 * q + 1] = (r[q].y >> 8) & 0x00ff00ffu;
    }
    const uint32_t a = majority8(lo), b = majority8(hi);
    *reinterpret_cast<uint32_t *>(out + vox(4 * g, Y, Z, cx, cy)) =
        (a & 0xffu) | ((a >> 8) & 0xff00u) | ((b & 0xffu) << 16) | ((b & 0xff0000u) << 8);
}

__global__ void k_restrict_bits_rows(const uint8_t *__restrict__ in, int nx, int ny, int nz,
                                     uint8_t *__restrict__ out) {
    const int cx = (nx + 1) / 2, cy = (ny + 1) / 2;
    const int X = blockIdx.x * RB + threadIdx.x, Y = blockIdx.y, Z = blockIdx.z;
    if (X >= cx) return;
    int cnt[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int x = min(2 * X + (q & 1), nx - 1), y = min(2 * Y + ((q >> 1) & 1), ny - 1),
                  z = min(2 * Z + ((q >> 2) & 1), nz - 1);
        const unsigned b = __ldg(in + vox(x, y, z, nx, ny));
#pragma unroll
        for (int j = 0; j < 8; ++j) cnt[j] += (b >> j) & 1u;
    }
    unsigned o = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) o |= (cnt[j] >= 4 ? 1u : 0u) << j;
    out[vox(X, Y, Z, cx, cy)] = (uint8_t)o;
}

// u_f(x) = 2 u_c((x + 0.5)/2 - 0.5), trilinear with clamped coordinates.
// Tiles of 64 x 8 x 8 fine voxels: the coarse values the interpolations read
// (34 x 6 x 6 per component, indices clamped) are staged in shared memory; a
// thread forms 2 x 2 x 2 fine voxels (2X, 2X + 1 and so on) of one component at
// a time from the 3 x 3 x 3 coarse values around (X, Y, Z): 27 shared reads
// for 8 outputs.  Along an axis the even voxel's corners are the first two of
// those three values and the odd one's the last two, with k_prolong's weights
// and terms (same bits); at the low border, where the clamped coordinate is 0 and
// the corners are voxels 0 and 1 with weights 1 and 0, voxel 1 stands in the place
// before voxel 0 and the weights change places.
constexpr int PX = 64, PY = 8, PZ = 8;
constexpr int PCX = PX / 2 + 2, PCY = PY / 2 + 2, PCZ = PZ / 2 + 2;
// Weights (low, high corner) of fine index x on a coarse axis of c voxels.
__device__ __forceinline__ void prolong_axis(int x, int c, float *w) {
    const float p = fminf(fmaxf((x + 0.5f) * 0.5f - 0.5f, 0.f), (float)(c - 1));
    const float f = p - floorf(p);
    w[1] = x > 0 ? f : 1.f;
    w[0] = 1.f - w[1];
}
// The coarse index staged at place i of an axis of c voxels.
__device__ __forceinline__ int prolong_src(int i, int c) { return i < 0 ? min(1, c - 1) : min(i, c - 1); }
__global__ void __launch_bounds__(128) k_prolong_tile(const float *__restrict__ uc, int cx, int cy, int cz, int nx,
                                                      int ny, int nz, float *__restrict__ uf) {
    __shared__ float t[3][PCZ][PCY][PCX];
    const int x0 = blockIdx.x * PX, y0 = blockIdx.y * PY, z0 = blockIdx.z * PZ;
    const int bx = x0 / 2 - 1, by = y0 / 2 - 1, bz = z0 / 2 - 1;      // coarse origin of the tile
    const size_t Nc = (size_t)cx * cy * cz, N = (size_t)nx * ny * nz;
    // a warp per coarse row, nine rows' loads in flight
    static_assert(3 * PCZ * PCY % 36 == 0, "4 warps x 9 rows per turn");
    const int ca = prolong_src(bx + (int)threadIdx.x, cx), cb = prolong_src(bx + 32 + (int)threadIdx.x, cx);
    for (int r0 = threadIdx.y; r0 < 3 * PCZ * PCY; r0 += 36) {
        float v[9], e[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const int row = r0 + 4 * q, j = row % PCY, k = (row / PCY) % PCZ, comp = row / (PCY * PCZ);
            const float *src = uc + comp * Nc + ((size_t)prolong_src(bz + k, cz) * cy + prolong_src(by + j, cy)) * cx;
            v[q] = __ldg(src + ca);
            e[q] = threadIdx.x < PCX - 32 ? __ldg(src + cb) : 0.f;
        }
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const int row = r0 + 4 * q, j = row % PCY, k = (row / PCY) % PCZ, comp = row / (PCY * PCZ);
            t[comp][k][j][threadIdx.x] = v[q];
            if (threadIdx.x < PCX - 32) t[comp][k][j][32 + threadIdx.x] = e[q];
        }
    }
    __syncthreads();
    const int lx = threadIdx.x, ly = threadIdx.y;                     // coarse cell of this thread: (lx, ly) of 32 x 4
    const int xa = x0 + 2 * lx, ya = y0 + 2 * ly;
    if (xa >= nx || ya >= ny) return;
    float wx[2][2], wy[2][2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        prolong_axis(xa + h, cx, wx[h]);
        prolong_axis(ya + h, cy, wy[h]);
    }
    const bool pair = xa + 1 < nx && nx % 2 == 0 && (reinterpret_cast<uintptr_t>(uf) & 7u) == 0;
    for (int lz = 0; lz < PZ / 2; ++lz) {
        const int za = z0 + 2 * lz;
        if (za >= nz) break;
        float wz[2][2];
        prolong_axis(za, cz, wz[0]);
        prolong_axis(za + 1, cz, wz[1]);
#pragma unroll
        for (int comp = 0; comp < 3; ++comp) {
            float c[3][3][3];
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
                for (int j = 0; j < 3; ++j)
#pragma unroll
                    for (int i = 0; i < 3; ++i) c[k][j][i] = t[comp][lz + k][ly + j][lx + i];
#pragma unroll
            for (int hz = 0; hz < 2; ++hz) {
                if (za + hz >= nz) continue;
#pragma unroll
                for (int hy = 0; hy < 2; ++hy) {
                    if (ya + hy >= ny) continue;
                    float o[2];
#pragma unroll
                    for (int hx = 0; hx < 2; ++hx) {
                        float acc = 0.f;
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const int i = q & 1, j = (q >> 1) & 1, k = q >> 2;
                            acc = fmaf(wx[hx][i] * wy[hy][j] * wz[hz][k], c[hz + k][hy + j][hx + i], acc);
                        }
                        o[hx] = 2.f * acc;
                    }
                    float *d = uf + comp * N + vox(xa, ya + hy, za + hz, nx, ny);
                    if (pair) {
                        *reinterpret_cast<float2 *>(d) = make_float2(o[0], o[1]);
                    } else {
                        d[0] = o[0];
                        if (xa + 1 < nx) d[1] = o[1];
                    }
                }
            }
        }
    }
}

__global__ void k_prolong(const float *__restrict__ uc, int cx, int cy, int cz, int nx, int ny,
                          int nz, float *__restrict__ uf) {
    const size_t N = (size_t)nx * ny * nz, Nc = (size_t)cx * cy * cz;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < N;
         i += (size_t)gridDim.x * blockDim.x) {
        const int x = (int)(i % nx), y = (int)((i / nx) % ny), z = (int)(i / ((size_t)nx * ny));
        const Corners c = corners((x + 0.5f) * 0.5f - 0.5f, (y + 0.5f) * 0.5f - 0.5f,
                                  (z + 0.5f) * 0.5f - 0.5f, cx, cy, cz);
#pragma unroll
        for (int comp = 0; comp < 3; ++comp) {
            const float *f = uc + comp * Nc;
            float acc = 0.f;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int qx = (q & 1) ? c.x1 : c.x0, qy = (q & 2) ? c.y1 : c.y0, qz = (q & 4) ? c.z1 : c.z0;
                const float w = ((q & 1) ? c.wx : 1.f - c.wx) * ((q & 2) ? c.wy : 1.f - c.wy) *
                                ((q & 4) ? c.wz : 1.f - c.wz);
                acc = fmaf(w, __ldg(f + vox(qx, qy, qz, cx, cy)), acc);
            }
            uf[comp * N + i] = 2.f * acc;
        }
    }
}

// ---- UROI: exact ellipsoidal dilation on bit rows ---------------------------
// The union of the structures is packed to one bit per voxel, rows of
// ceil(nx / 32) words, so a thread handles 32 voxels with shifts and ORs:
//   k_uroi_bits   bytes -> bits (N bytes read, N / 8 written)
//   k_uroi_rows   per word of row (y, z) and per |dz| = 0 .. rz, the OR over dy
//                 of row y + dy dilated in x by ext(dy, dz), the x extent the
//                 ellipsoid admits there (-1: none); a dilation by r is built
//                 from the one by r - 1 with two shifts over the neighbour words
//   k_uroi_out    OR over dz of the |dz| words at z + dz, expanded to bytes
// The extents are computed on the host with the same double expression as the
// definition, so the decision equals the brute-force test voxel by voxel.
// Two bytes per voxel must move; 256x256x96 with 10 mm takes 19 us, where byte
// maps (row distances and per-voxel z masks, about 31 byte loads per voxel)
// took 146 us.
constexpr int kMaxUroiRadius = 15;
struct UroiTable {
    int rx, ry, rz;
    int8_t ext[kMaxUroiRadius + 1][kMaxUroiRadius + 1];   // [|dz|][|dy|], -1 = none
};

// Word i of the bit rows: its row (y, z) and first voxel x.
struct BitWord {
    long long row;
    int x;
    __device__ BitWord(long long i, int wpr) {
        row = i < (1ll << 31) ? (long long)((unsigned)i / (unsigned)wpr) : i / wpr;
        x = (int)(i - row * wpr) * 32;
    }
    __device__ int z(int ny) const {
        return (int)(row < (1ll << 31) ? (unsigned)row / (unsigned)ny : row / ny);
    }
};

// Bit q set where byte q of w has a bit of the mask.
__device__ __forceinline__ uint32_t bits_of(uint32_t w, uint32_t mask4) {
    const uint32_t b = __vcmpne4(w & mask4, 0u) & 0x08040201u;      // bit q of byte q
    return (b | (b >> 8) | (b >> 16) | (b >> 24)) & 0xfu;
}
__global__ void k_uroi_bits(const uint8_t *__restrict__ sbits, unsigned mask, int nx, long long words, int wpr, int vec,
                            uint32_t *__restrict__ bits) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= words) return;
    const BitWord bw(i, wpr);
    const int x = bw.x;
    const uint8_t *src = sbits + (size_t)bw.row * nx + x;
    uint32_t b = 0;
    if (vec && x + 32 <= nx) {                     // 16-byte aligned rows
        const uint32_t m4 = mask * 0x01010101u;
        const uint4 p = __ldg(reinterpret_cast<const uint4 *>(src)), q = __ldg(reinterpret_cast<const uint4 *>(src) + 1);
        b = bits_of(p.x, m4) | bits_of(p.y, m4) << 4 | bits_of(p.z, m4) << 8 | bits_of(p.w, m4) << 12 |
            bits_of(q.x, m4) << 16 | bits_of(q.y, m4) << 20 | bits_of(q.z, m4) << 24 | bits_of(q.w, m4) << 28;
    } else {
#pragma unroll 8
        for (int e = 0; e < 32; ++e)
            if (x + e < nx && (__ldg(src + e) & mask)) b |= 1u << e;
    }
    bits[i] = b;
}

// NZ: accumulators (|dz| values) per thread, at least rz + 1.
template <int NZ>
__global__ void k_uroi_rows(const uint32_t *__restrict__ bits, const __grid_constant__ UroiTable t, int ny,
                            long long words, int wpr, uint32_t *__restrict__ zrows) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= words) return;
    const BitWord bw(i, wpr);
    const int c = bw.x / 32, y = (int)(bw.row - (long long)bw.z(ny) * ny);
    uint32_t acc[NZ];
#pragma unroll
    for (int z = 0; z < NZ; ++z) acc[z] = 0u;
    for (int dy = -t.ry; dy <= t.ry; ++dy) {
        if (y + dy < 0 || y + dy >= ny) continue;
        const uint32_t *r = bits + i + (long long)dy * wpr;
        const uint32_t w = __ldg(r), pw = c > 0 ? __ldg(r - 1) : 0u, nw = c + 1 < wpr ? __ldg(r + 1) : 0u;
        if ((w | pw | nw) == 0u) continue;
        uint32_t d = w;                             // the row dilated by q
        for (int q = 0; q <= t.rx; ++q) {
            if (q > 0) d |= __funnelshift_l(pw, w, q) | __funnelshift_r(w, nw, q);
#pragma unroll
            for (int z = 0; z < NZ; ++z)
                if (z <= t.rz && t.ext[z][dy < 0 ? -dy : dy] == q) acc[z] |= d;
        }
    }
    for (int z = 0; z < NZ; ++z)
        if (z <= t.rz) zrows[(size_t)z * words + i] = acc[z];
}

// The bytes 0 / 1 of bits 4 e .. 4 e + 3 of w.
__device__ __forceinline__ uint32_t byte4(uint32_t w, int e) {
    const uint32_t n = (w >> (4 * e)) & 0xfu;
    return (n | (n << 7) | (n << 14) | (n << 21)) & 0x01010101u;
}
__global__ void k_uroi_out(const uint32_t *__restrict__ zrows, int rz, int nx, int ny, int nz,
                           long long words, int wpr, int vec, uint8_t *__restrict__ out) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x, plane = (long long)ny * wpr;
    if (i >= words) return;
    const BitWord bw(i, wpr);
    const int x = bw.x, z = bw.z(ny);
    uint32_t b = 0;
    for (int dz = -rz; dz <= rz; ++dz) {
        if (z + dz < 0 || z + dz >= nz) continue;
        b |= __ldg(zrows + (size_t)(dz < 0 ? -dz : dz) * words + i + dz * plane);
    }
    uint8_t *dst = out + (size_t)bw.row * nx + x;
    if (vec && x + 32 <= nx) {
        reinterpret_cast<uint4 *>(dst)[0] = make_uint4(byte4(b, 0), byte4(b, 1), byte4(b, 2), byte4(b, 3));
        reinterpret_cast<uint4 *>(dst)[1] = make_uint4(byte4(b, 4), byte4(b, 5), byte4(b, 6), byte4(b, 7));
    } else {
        for (int e = 0; e < 32 && x + e < nx; ++e) dst[e] = (uint8_t)((b >> e) & 1u);
    }
}

// Rows of one word (nx <= 32) without the |dz| words: the OR over dz and dy of
// rows dilated in place.  For volumes so narrow that the words, one per row
// however short, would outgrow byte maps (nx <= 13 at the most).
__global__ void k_uroi_narrow(const uint32_t *__restrict__ bits, const __grid_constant__ UroiTable t, int nx, int ny,
                              int nz, uint8_t *__restrict__ out) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)ny * nz) return;
    const int z = (int)(i / ny), y = (int)(i - (long long)z * ny);
    uint32_t b = 0;
    for (int dz = -t.rz; dz <= t.rz; ++dz) {
        if (z + dz < 0 || z + dz >= nz) continue;
        for (int dy = -t.ry; dy <= t.ry; ++dy) {
            const int e = t.ext[dz < 0 ? -dz : dz][dy < 0 ? -dy : dy];
            if (e < 0 || y + dy < 0 || y + dy >= ny) continue;
            const uint32_t w = __ldg(bits + i + (long long)dz * ny + dy);
            if (w == 0u) continue;
            for (int q = 0; q <= e; ++q) b |= (w << q) | (w >> q);
        }
    }
    uint8_t *dst = out + (size_t)i * nx;
    for (int e = 0; e < nx; ++e) dst[e] = (uint8_t)((b >> e) & 1u);
}

__global__ void k_fill_u8(uint8_t *p, size_t n, uint8_t v) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        p[i] = v;
}

// ---- automatic sign ---------------------------------------------------
// Per structure {sum T0 inside, count inside, sum T0 in the shell, count of the
// shell}, the shell being the voxels outside the structure within Chebyshev
// distance 2 of it.  k_dilate_xy ORs the mask bytes over 5 x 5 voxels in each
// plane; k_sign_sums marches along z with five planes of that in registers and
// reads T0 only where some structure or shell is.  A thread owns V x-adjacent
// voxels (V = 4, one 32-bit word of mask bytes, where nx % 4 == 0).  A thread
// sums its 64 voxels at most in triples of floats (exact to 2^-64 of the sum, so
// no less than an FP64 sum), because FP64 adds take a warp 14 cycles of the SM
// here; across threads the sums are FP64, and a sum that overflows a float is
// taken again in FP64.  A structure costs the voxels and warps that it does not
// reach one test.
// 256x256x96, 5 structures, all three kernels and the read-back: 56 us, as with
// pairs of floats (48 bits); a third register per sum 69; FP64 sums per thread
// about 100; three dilation launches and, per structure, an FP64 pass over T0 and
// a serial sum of its partials 670.
constexpr int SB = 256, SZ = 16;                  // threads, planes per CTA at most (thin volumes: more)
// A 1-D grid of SB threads of V voxels over the columns of a plane, then z: no
// limit on any extent, and no idle threads in narrow or flat volumes.
struct SignTile {
    size_t col;            // first voxel of the thread's columns in a plane
    bool in;
    int bz;
    __device__ SignTile(int nx, int ny, int v) {
        const size_t cols = (size_t)nx * ny / v;
        const unsigned tiles = (unsigned)((cols + SB - 1) / SB);
        bz = (int)(blockIdx.x / tiles);
        const size_t c = (size_t)(blockIdx.x - bz * tiles) * SB + threadIdx.x;
        in = c < cols;
        col = c * v;
    }
};
// A sum of floats as high part, the rounding errors' sum (both exact by Knuth's
// two-sum) and, in *low, that sum's own rounding errors.  *low lies in shared
// memory: values that vary as CT numbers do hardly ever reach it, and a third
// register per sum would take the kernel from three to two CTAs per SM.
struct TripleSum {
    float s = 0.f, e = 0.f;
    static __device__ __forceinline__ float two_sum(float &s, float v) {      // s += v; the rounding error
        const float t = __fadd_rn(s, v), b = __fsub_rn(t, s), a = __fsub_rn(s, __fsub_rn(t, b));
        s = t;
        return __fadd_rn(a, __fsub_rn(v, b));
    }
    __device__ __forceinline__ void add(float v, float *low) {
        v = two_sum(s, v);
        v = two_sum(e, v);
        if (v != 0.f) *low += v;
    }
    __device__ __forceinline__ double value(const float *low) const { return (double)s + ((double)e + (double)*low); }
};
template <int V>
__global__ void __launch_bounds__(SB) k_dilate_xy(const uint8_t *__restrict__ bits, int nx, int ny,
                                                  uint8_t *__restrict__ out) {
    const SignTile t(nx, ny, V);
    if (!t.in) return;
    const int y = t.col < (1ull << 31) ? (int)((unsigned)t.col / (unsigned)nx) : (int)(t.col / nx);
    const int x = (int)(t.col - (size_t)y * nx);
    // rows outside the volume are read at the border, which lies within
    // distance 2 as well: no branch between the loads
    uint32_t w[5][V == 4 ? 3 : 5];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        const uint8_t *r = bits + ((size_t)t.bz * ny + clampi(y + q - 2, 0, ny - 1)) * nx + x;
        if constexpr (V == 4) {
            const uint32_t *rw = reinterpret_cast<const uint32_t *>(r);
            w[q][0] = __ldg(rw);
            w[q][1] = __ldg(rw - (x > 0 ? 1 : 0));
            w[q][2] = __ldg(rw + (x + 4 < nx ? 1 : 0));
        } else {
#pragma unroll
            for (int e = 0; e < 5; ++e) w[q][e] = __ldg(r + (clampi(x + e - 2, 0, nx - 1) - x));
        }
    }
    uint32_t d = 0;
    const size_t i = ((size_t)t.bz * ny + y) * nx + x;
    if constexpr (V == 4) {
        uint32_t c = 0, p = 0, n = 0;
#pragma unroll
        for (int q = 0; q < 5; ++q) { c |= w[q][0]; p |= w[q][1]; n |= w[q][2]; }
        if (x == 0) p = 0u;
        if (x + 4 >= nx) n = 0u;
        d = c | __funnelshift_l(p, c, 8) | __funnelshift_l(p, c, 16) | __funnelshift_r(c, n, 8) |
            __funnelshift_r(c, n, 16);
        *reinterpret_cast<uint32_t *>(out + i) = d;
    } else {
#pragma unroll
        for (int q = 0; q < 5; ++q)
#pragma unroll
            for (int e = 0; e < 5; ++e) d |= w[q][e];
        out[i] = (uint8_t)d;
    }
}

template <typename IT, int V>
__global__ void __launch_bounds__(SB) k_sign_sums(const IT *__restrict__ T0, const uint8_t *__restrict__ sbits,
                                                  const uint8_t *__restrict__ dxy, int k, int nx, int ny, int nz,
                                                  int zc, double *__restrict__ partial) {
    const SignTile st(nx, ny, V);
    const int zb = st.bz * zc, ze = min(zb + zc, nz);
    const int tid = threadIdx.x, bid = blockIdx.x;
    const unsigned kmask = (1u << k) - 1u;
    TripleSum sin_[kMaxMasks], ssh[kMaxMasks];
    __shared__ float low[2][kMaxMasks][SB];       // each thread's own
#pragma unroll
    for (int j = 0; j < kMaxMasks; ++j) low[0][j][tid] = low[1][j][tid] = 0.f;
    int cnt[kMaxMasks] = {};                      // inside (low 16 bits) and shell: at most V zc each
    unsigned seen = 0;
    const size_t nxy = (size_t)nx * ny, col = st.col;
    auto word = [&](const uint8_t *b, int z) -> uint32_t {           // 0 outside the volume
        if (z < 0 || z >= nz) return 0u;
        const uint8_t *p = b + (size_t)z * nxy + col;
        return V == 4 ? __ldg(reinterpret_cast<const uint32_t *>(p)) : (uint32_t)__ldg(p);
    };
    if (st.in) {
        // planes z - 2 .. z + 2 of the dilated bytes, z + 3 and the next plane's own bytes in flight
        uint32_t d0 = 0, d1 = word(dxy, zb - 2), d2 = word(dxy, zb - 1), d3 = word(dxy, zb), d4 = word(dxy, zb + 1),
                 nd = word(dxy, zb + 2), nc = word(sbits, zb);
        for (int z = zb; z < ze; ++z) {
            d0 = d1; d1 = d2; d2 = d3; d3 = d4; d4 = nd;
            const uint32_t cen = nc, all = (d0 | d1 | d2 | d3 | d4) & (kmask * 0x01010101u);
            nd = word(dxy, z + 3);
            nc = word(sbits, z + 1);
            if (all == 0u) continue;              // no structure within distance 2 of these voxels
            const size_t i = (size_t)z * nxy + col;
            float tv[V];
#pragma unroll
            for (int v = 0; v < V; ++v) tv[v] = ld_img<IT>(T0 + i + v);
#pragma unroll
            for (int j = 0; j < kMaxMasks; ++j) {
                if ((all & (0x01010101u << j)) == 0u) continue;
                seen |= 1u << j;
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    if (!((all >> (8 * v + j)) & 1u)) continue;
                    if ((cen >> (8 * v + j)) & 1u) {
                        sin_[j].add(tv[v], &low[0][j][tid]);
                        cnt[j] += 1;
                    } else {
                        ssh[j].add(tv[v], &low[1][j][tid]);
                        cnt[j] += 1 << 16;
                    }
                }
            }
        }
    }
    // one of this thread's sums in FP64, read again
    auto again = [&](int j, bool shell) {
        double a = 0.0;
        for (int z = zb; z < ze; ++z) {
            uint32_t m = word(sbits, z);
            if (shell) m = (word(dxy, z - 2) | word(dxy, z - 1) | word(dxy, z) | word(dxy, z + 1) | word(dxy, z + 2)) & ~m;
            for (int v = 0; v < V; ++v)
                if ((m >> (8 * v + j)) & 1u) a += (double)ld_img<IT>(T0 + (size_t)z * nxy + col + v);
        }
        return a;
    };
    auto total = [&](const TripleSum &t, int j, bool shell) {
        return isfinite(t.s + t.e) ? t.value(&low[shell][j][tid]) : again(j, shell);
    };
    // block sums in a fixed order: lanes by shuffles, then the 8 warps in turn
    __shared__ double ws[kMaxMasks][2][8];
    __shared__ int wc[kMaxMasks][2][8];
    const unsigned wseen = __reduce_or_sync(0xffffffffu, seen);
#pragma unroll
    for (int j = 0; j < kMaxMasks; ++j) {
        if (j >= k) break;
        double a = 0.0, c = 0.0;
        int ca = 0, cc = 0;
        if ((wseen >> j) & 1u) {                  // the same for the whole warp
            a = total(sin_[j], j, false); c = total(ssh[j], j, true);
            ca = __reduce_add_sync(0xffffffffu, cnt[j] & 0xffff);
            cc = __reduce_add_sync(0xffffffffu, cnt[j] >> 16);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                a += __shfl_xor_sync(0xffffffffu, a, o);
                c += __shfl_xor_sync(0xffffffffu, c, o);
            }
        }
        if ((tid & 31) == 0) {
            ws[j][0][tid >> 5] = a; ws[j][1][tid >> 5] = c;
            wc[j][0][tid >> 5] = ca; wc[j][1][tid >> 5] = cc;
        }
    }
    const bool any = __syncthreads_or(seen != 0u);
    if (tid < 2 * k) {                            // one thread per structure and side
        const int j = tid >> 1, side = tid & 1;
        double A = 0;
        int C = 0;
        if (any)
            for (int w = 0; w < 8; ++w) { A += ws[j][side][w]; C += wc[j][side][w]; }
        double *o = partial + ((size_t)bid * k + j) * 4 + 2 * side;
        o[0] = A; o[1] = (double)C;
    }
}

// Column sums of partial[rows][cols], a CTA per column: each thread takes a
// fixed stride of rows, then lanes and warps are added in a fixed order.
__global__ void __launch_bounds__(256) k_sum_rows(const double *__restrict__ partial, int rows, int cols,
                                                  double *__restrict__ out) {
    __shared__ double ws[8];
    const int c = blockIdx.x, tid = threadIdx.x;
    double s = 0;
    int b = tid;
    for (; b + 7 * 256 < rows; b += 8 * 256) {               // eight rows in flight, added in order
        double v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = __ldg(partial + (size_t)(b + q * 256) * cols + c);
#pragma unroll
        for (int q = 0; q < 8; ++q) s += v[q];
    }
    for (; b < rows; b += 256) s += __ldg(partial + (size_t)b * cols + c);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((tid & 31) == 0) ws[tid >> 5] = s;
    __syncthreads();
    if (tid == 0) {
        double t = 0;
        for (int w = 0; w < 8; ++w) t += ws[w];
        out[c] = t;
    }
}

__global__ void k_make_texels_f32(const float *__restrict__ I0, const uint8_t *__restrict__ bits, size_t n,
                                  float2 *__restrict__ tex) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        tex[i] = make_float2(__ldg(I0 + i), __uint_as_float((unsigned)__ldg(bits + i)));
}

// 16-bit images: low half = the value's bits, bits 16..23 = the mask bits.
__global__ void k_make_texels_16(const unsigned short *__restrict__ I0, const uint8_t *__restrict__ bits,
                                 size_t n, uint32_t *__restrict__ tex) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        tex[i] = (uint32_t)__ldg(I0 + i) | ((uint32_t)__ldg(bits + i) << 16);
}

template <typename IN, typename OUT>
__global__ void k_convert(const IN *__restrict__ in, size_t n, OUT *__restrict__ out) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        out[i] = from_f<OUT>(to_f<IN>(in[i]));
}

}  // namespace

cudaError_t launch_pack_masks(const uint8_t *const *masks, int k, size_t n, uint8_t *bits,
                              cudaStream_t s) {
    MaskPtrs m{};
    uintptr_t low = reinterpret_cast<uintptr_t>(bits) | n;      // low bits of every pointer and the size
    for (int j = 0; j < k && j < kMaxMasks; ++j) {
        m.p[j] = masks[j];
        low |= reinterpret_cast<uintptr_t>(masks[j]);
    }
    if (n == 0) return cudaSuccess;
    if (low % 16 == 0 && n / 16 / 128 < ((size_t)1 << 31) - 1)
        k_pack16<<<(unsigned)((n / 16 + 127) / 128), 128, 0, s>>>(m, k, n / 16, reinterpret_cast<uint4 *>(bits));
    else if (low % 4 == 0)
        k_pack4<<<flat_grid(n / 4), 256, 0, s>>>(m, k, n / 4, reinterpret_cast<uint32_t *>(bits));
    else
        k_pack<<<flat_grid(n), 256, 0, s>>>(m, k, n, bits);
    note_launch();
    return cudaGetLastError();
}

template <typename IT>
static void restrict_image_to(const void *in, int nx, int ny, int nz, void *out, int out_dtype, size_t Nc,
                              cudaStream_t s) {
    const IT *src = static_cast<const IT *>(in);
    const int cx = (nx + 1) / 2, cy = (ny + 1) / 2, cz = (nz + 1) / 2;
    if (rows_ok(cy, cz) && nx % 2 == 0 && (reinterpret_cast<uintptr_t>(in) & (2 * sizeof(IT) - 1)) == 0) {
        const dim3 g = row_grid(cx, cy, cz);
        if (out_dtype == CGDIR_F16)
            k_restrict_image_pairs<IT, __half><<<g, RB, 0, s>>>(src, nx, ny, nz, (__half *)out);
        else if (out_dtype == CGDIR_BF16)
            k_restrict_image_pairs<IT, __nv_bfloat16><<<g, RB, 0, s>>>(src, nx, ny, nz, (__nv_bfloat16 *)out);
        else
            k_restrict_image_pairs<IT, float><<<g, RB, 0, s>>>(src, nx, ny, nz, (float *)out);
        return;
    }
    if (rows_ok(cy, cz)) {
        const dim3 g = row_grid(cx, cy, cz);
        if (out_dtype == CGDIR_F16)
            k_restrict_image_rows<IT, __half><<<g, RB, 0, s>>>(src, nx, ny, nz, (__half *)out);
        else if (out_dtype == CGDIR_BF16)
            k_restrict_image_rows<IT, __nv_bfloat16><<<g, RB, 0, s>>>(src, nx, ny, nz, (__nv_bfloat16 *)out);
        else
            k_restrict_image_rows<IT, float><<<g, RB, 0, s>>>(src, nx, ny, nz, (float *)out);
        return;
    }
    if (out_dtype == CGDIR_F16)
        k_restrict_image<IT, __half><<<flat_grid(Nc), 256, 0, s>>>(src, nx, ny, nz, (__half *)out);
    else if (out_dtype == CGDIR_BF16)
        k_restrict_image<IT, __nv_bfloat16><<<flat_grid(Nc), 256, 0, s>>>(src, nx, ny, nz, (__nv_bfloat16 *)out);
    else
        k_restrict_image<IT, float><<<flat_grid(Nc), 256, 0, s>>>(src, nx, ny, nz, (float *)out);
}

cudaError_t launch_restrict_image(const void *in, int in_dtype, int nx, int ny, int nz, void *out, int out_dtype,
                                  cudaStream_t s) {
    const size_t Nc = (size_t)((nx + 1) / 2) * ((ny + 1) / 2) * ((nz + 1) / 2);
    if (in_dtype == CGDIR_F16)
        restrict_image_to<__half>(in, nx, ny, nz, out, out_dtype, Nc, s);
    else if (in_dtype == CGDIR_BF16)
        restrict_image_to<__nv_bfloat16>(in, nx, ny, nz, out, out_dtype, Nc, s);
    else
        restrict_image_to<float>(in, nx, ny, nz, out, out_dtype, Nc, s);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_restrict_image(const void *in, int dtype, int nx, int ny, int nz, void *out,
                                  cudaStream_t s) {
    return launch_restrict_image(in, dtype, nx, ny, nz, out, dtype, s);
}

cudaError_t launch_restrict_bits(const uint8_t *in, int nx, int ny, int nz, uint8_t *out,
                                 cudaStream_t s) {
    const size_t Nc = (size_t)((nx + 1) / 2) * ((ny + 1) / 2) * ((nz + 1) / 2);
    const int cx = (nx + 1) / 2, cy = (ny + 1) / 2, cz = (nz + 1) / 2;
    if (rows_ok(cy, cz) && nx % 8 == 0 && (reinterpret_cast<uintptr_t>(in) & 7u) == 0 &&
        (reinterpret_cast<uintptr_t>(out) & 3u) == 0)
        k_restrict_bits8<<<row_grid(nx / 8, cy, cz), RB, 0, s>>>(in, nx, ny, nz, out);
    else if (rows_ok(cy, cz))
        k_restrict_bits_rows<<<row_grid(cx, cy, cz), RB, 0, s>>>(in, nx, ny, nz, out);
    else
        k_restrict_bits<<<flat_grid(Nc), 256, 0, s>>>(in, nx, ny, nz, out);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_prolong(const float *uc, int cx, int cy, int cz, int nx, int ny, int nz,
                           float *uf, cudaStream_t s) {
    if (rows_ok(ny, nz) && nx <= 2 * cx && ny <= 2 * cy && nz <= 2 * cz)
        k_prolong_tile<<<dim3((nx + PX - 1) / PX, (ny + PY - 1) / PY, (nz + PZ - 1) / PZ), dim3(32, 4), 0, s>>>(
            uc, cx, cy, cz, nx, ny, nz, uf);
    else
        k_prolong<<<flat_grid((size_t)nx * ny * nz), 256, 0, s>>>(uc, cx, cy, cz, nx, ny, nz, uf);
    note_launch();
    return cudaGetLastError();
}

static int uroi_radius(double margin, double spacing) { return (int)(margin / spacing); }
// Whether the words of rows and |dz| take more than byte maps did (5 per voxel).
static bool uroi_narrow(int nx, int ny, int nz, int rz) {
    const size_t words = (size_t)ny * nz * ((nx + 31) / 32);
    return nx <= 32 && 4 * words * (rz + 2) > 5 * (size_t)nx * ny * nz;
}

// scratch: uroi_scratch_bytes.
cudaError_t launch_uroi(const uint8_t *sbits, int k, int nx, int ny, int nz, const double *spacing,
                        double margin, uint8_t *scratch, uint8_t *out, cudaStream_t s) {
    const size_t N = (size_t)nx * ny * nz;
    if (k <= 0) {
        k_fill_u8<<<flat_grid(N), 256, 0, s>>>(out, N, 1); note_launch();
        return cudaGetLastError();
    }
    if (!(margin >= 0.0) || !(spacing[0] > 0) || !(spacing[1] > 0) || !(spacing[2] > 0))
        return cudaErrorInvalidValue;
    UroiTable t{};
    t.rx = uroi_radius(margin, spacing[0]);
    t.ry = uroi_radius(margin, spacing[1]);
    t.rz = uroi_radius(margin, spacing[2]);
    if (t.rx > kMaxUroiRadius || t.ry > kMaxUroiRadius || t.rz > kMaxUroiRadius)
        return cudaErrorInvalidValue;
    for (int dz = 0; dz <= t.rz; ++dz)
        for (int dy = 0; dy <= t.ry; ++dy) {
            int e = -1;
            for (int dx = 0; dx <= t.rx; ++dx) {
                const double d2 = (dx * spacing[0]) * (dx * spacing[0]) + (dy * spacing[1]) * (dy * spacing[1]) +
                                  (dz * spacing[2]) * (dz * spacing[2]);
                if (d2 <= margin * margin) e = dx;
            }
            t.ext[dz][dy] = (int8_t)e;
        }
    const unsigned mask = (k >= 8) ? 0xffu : ((1u << k) - 1u);
    const int wpr = (nx + 31) / 32;
    const long long words = (long long)ny * nz * wpr;
    uint32_t *bits = reinterpret_cast<uint32_t *>(scratch), *zrows = bits + words;
    const unsigned g = (unsigned)((words + 127) / 128);
    auto aligned = [&](const void *q) { return nx % 16 == 0 && (reinterpret_cast<uintptr_t>(q) & 15u) == 0; };
    k_uroi_bits<<<g, 128, 0, s>>>(sbits, mask, nx, words, wpr, aligned(sbits), bits); note_launch();
    if (uroi_narrow(nx, ny, nz, t.rz)) {
        k_uroi_narrow<<<g, 128, 0, s>>>(bits, t, nx, ny, nz, out); note_launch();
        return cudaGetLastError();
    }
    if (t.rz < 5) k_uroi_rows<5><<<g, 128, 0, s>>>(bits, t, ny, words, wpr, zrows);
    else k_uroi_rows<kMaxUroiRadius + 1><<<g, 128, 0, s>>>(bits, t, ny, words, wpr, zrows);
    note_launch();
    k_uroi_out<<<g, 128, 0, s>>>(zrows, t.rz, nx, ny, nz, words, wpr, aligned(out), out); note_launch();
    return cudaGetLastError();
}

// Bit rows, then rz + 1 words per bit-row word.  (A margin or spacing that
// launch_uroi refuses needs none.)
size_t uroi_scratch_bytes(int nx, int ny, int nz, double spacing_z, double margin) {
    if (!(margin >= 0.0) || !(spacing_z > 0) || margin / spacing_z >= kMaxUroiRadius + 1) return 0;
    const int rz = uroi_radius(margin, spacing_z);
    return (size_t)ny * nz * ((nx + 31) / 32) * 4 * (uroi_narrow(nx, ny, nz, rz) ? 1 : rz + 2);
}

static size_t sign_ctas(int nx, int ny, int nz, int v, int zc) {
    return ((size_t)nx * ny / v + SB - 1) / SB * ((nz + zc - 1) / zc);
}
// Planes per CTA: 16 where that gives 8 CTAs per SM (the march is bound by
// latency), else 8 or 4 (each chunk reads 4 more planes of dilated bytes).  In a
// volume of few columns more, so that the partial sums (a row of 4 per structure
// and CTA) take no more than a byte per voxel; a thread counts its voxels in 16
// bits.
static int sign_zchunk(int nx, int ny, int nz, int v) {
    int zc = SZ;
    while (zc > 4 && sign_ctas(nx, ny, nz, v, zc) < (size_t)8 * sm_count()) zc /= 2;
    while (zc < 4096 && sign_ctas(nx, ny, nz, v, zc) * kMaxMasks * 32 > (size_t)nx * ny * nz + 16384) zc *= 2;
    return zc;
}
size_t sign_partial_rows(int nx, int ny, int nz) {
    const size_t one = sign_ctas(nx, ny, nz, 1, sign_zchunk(nx, ny, nz, 1));
    return nx % 4 == 0 ? std::max(one, sign_ctas(nx, ny, nz, 4, sign_zchunk(nx, ny, nz, 4))) : one;
}

template <typename IT>
static void sign_sums_t(const void *T0, const uint8_t *sbits, int k, int nx, int ny, int nz, uint8_t *dxy,
                        double *partial, double *sums, cudaStream_t s) {
    // four voxels per thread: mask bytes as 32-bit words
    const bool quad = nx % 4 == 0 && (reinterpret_cast<uintptr_t>(sbits) & 3u) == 0;
    const int v = quad ? 4 : 1, zc = sign_zchunk(nx, ny, nz, v);
    const unsigned g = (unsigned)sign_ctas(nx, ny, nz, v, zc);
    const int block = SB;
    const IT *t0 = static_cast<const IT *>(T0);
    if (quad) {
        k_dilate_xy<4><<<(unsigned)sign_ctas(nx, ny, nz, 4, 1), block, 0, s>>>(sbits, nx, ny, dxy);
        k_sign_sums<IT, 4><<<g, block, 0, s>>>(t0, sbits, dxy, k, nx, ny, nz, zc, partial);
    } else {
        k_dilate_xy<1><<<(unsigned)sign_ctas(nx, ny, nz, 1, 1), block, 0, s>>>(sbits, nx, ny, dxy);
        k_sign_sums<IT, 1><<<g, block, 0, s>>>(t0, sbits, dxy, k, nx, ny, nz, zc, partial);
    }
    k_sum_rows<<<4 * k, 256, 0, s>>>(partial, (int)g, 4 * k, sums);
    note_launch(3);
}

// sums: device [k][4]; dxy: N bytes, 4-byte aligned; partial: sign_partial_rows x k x 4 doubles.
cudaError_t launch_sign_sums(const void *T0, int dtype, const uint8_t *sbits, int k, int nx, int ny, int nz,
                             uint8_t *dxy, double *partial, double *sums, cudaStream_t s) {
    if (dtype == CGDIR_F16) sign_sums_t<__half>(T0, sbits, k, nx, ny, nz, dxy, partial, sums, s);
    else if (dtype == CGDIR_BF16) sign_sums_t<__nv_bfloat16>(T0, sbits, k, nx, ny, nz, dxy, partial, sums, s);
    else sign_sums_t<float>(T0, sbits, k, nx, ny, nz, dxy, partial, sums, s);
    return cudaGetLastError();
}

cudaError_t launch_make_texels(const void *I0, int dtype, const uint8_t *bits, size_t n, void *tex,
                               cudaStream_t s) {
    if (dtype == CGDIR_F32)
        k_make_texels_f32<<<flat_grid(n), 256, 0, s>>>((const float *)I0, bits, n, (float2 *)tex);
    else
        k_make_texels_16<<<flat_grid(n), 256, 0, s>>>((const unsigned short *)I0, bits, n, (uint32_t *)tex);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_convert_image(const void *in, int in_dtype, size_t n, void *out, int out_dtype,
                                 cudaStream_t s) {
    if (in_dtype == out_dtype)
        return cudaMemcpyAsync(out, in, n * img_elem_size(in_dtype), cudaMemcpyDeviceToDevice, s);
    const unsigned g = flat_grid(n);
#define CGDIR_CONV(IN, OUT) k_convert<IN, OUT><<<g, 256, 0, s>>>((const IN *)in, n, (OUT *)out)
    if (in_dtype == CGDIR_F32 && out_dtype == CGDIR_F16) CGDIR_CONV(float, __half);
    else if (in_dtype == CGDIR_F32 && out_dtype == CGDIR_BF16) CGDIR_CONV(float, __nv_bfloat16);
    else if (in_dtype == CGDIR_F16 && out_dtype == CGDIR_F32) CGDIR_CONV(__half, float);
    else if (in_dtype == CGDIR_BF16 && out_dtype == CGDIR_F32) CGDIR_CONV(__nv_bfloat16, float);
    else if (in_dtype == CGDIR_F16 && out_dtype == CGDIR_BF16) CGDIR_CONV(__half, __nv_bfloat16);
    else if (in_dtype == CGDIR_BF16 && out_dtype == CGDIR_F16) CGDIR_CONV(__nv_bfloat16, __half);
    else return cudaErrorInvalidValue;
#undef CGDIR_CONV
    note_launch();
    return cudaGetLastError();
}

}  // namespace cgdir
