// Low-pass filter kernel of CG-DIR (kernel 1, Sec. 2.2; Algorithm A steps 2
// and 4) and the composite update (Algorithm A step 3, the vector half of
// kernel 4).
//
// Smoothing: the 3-D Gaussian is applied as x, y and z passes (the
// separability the paper uses) inside ONE kernel, so each component is read
// once and written once.  A CTA owns a column in x-y and marches along z:
// every input plane of the column plus an R-voxel halo goes to shared memory,
// the x pass and the y pass run there, and each thread keeps the last 2R+1
// xy-filtered values of its outputs in registers for the z pass.  The borders
// are clamped (clamp-to-edge).
//
// Where the field satisfies the tensor-map rules (nx a multiple of 4, 16-byte
// aligned base) the planes come by cp.async.bulk.tensor, otherwise by
// cp.async with clamped indices, into a ring of shared-memory stages, so the
// loads of the next planes are in flight while the current one is filtered.
// The plain kernel family (no waits inside kernels) loads the halo with
// ordinary clamped loads.
//
// Every kernel here returns at once when the level's stop flag is set, so a
// level that converged early leaves its fields untouched.
#include "cgdir_internal.cuh"
#include "tma.cuh"

#include <algorithm>
#include <cmath>

namespace cgdir {

int gauss_radius(float sigma) {
    if (!(sigma > 0.f)) return 0;
    return (int)std::ceil(3.0 * (double)sigma - 1e-9);
}

Taps gauss_taps(float sigma) {
    Taps t{};
    t.r = gauss_radius(sigma);
    if (t.r == 0) { t.w[0] = 1.f; return t; }
    double w[2 * kMaxRadius + 1], s = 0.0;
    for (int j = -t.r; j <= t.r; ++j) {
        w[j + t.r] = std::exp(-(double)(j * j) / (2.0 * (double)sigma * (double)sigma));
        s += w[j + t.r];
    }
    for (int j = 0; j <= 2 * t.r; ++j) t.w[j] = (float)(w[j] / s);
    return t;
}

namespace {

constexpr int TX = 32, TY = 8, NT = TX * TY;

template <int R>
__global__ void __launch_bounds__(NT) k_smooth(const float *__restrict__ in,
                                               float *__restrict__ out, int ncomp, Taps taps,
                                               int nx, int ny, int nz, int zchunk,
                                               const int *stop_flag) {
    if (stop_flag && *stop_flag) return;
    constexpr int SX = TX + 2 * R, SY = TY + 2 * R, K = 2 * R + 1;
    __shared__ float S[3][SY][SX];
    __shared__ float X[3][SY][TX];
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX + tx;
    const size_t N = (size_t)nx * ny * nz;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const int zb = blockIdx.z * zchunk, ze = min(zb + zchunk, nz);
    const int x = x0 + tx, y = y0 + ty;
    const bool act = x < nx && y < ny;
    float w[K];
#pragma unroll
    for (int j = 0; j < K; ++j) w[j] = taps.w[j];
    float ring[3][K];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int j = 0; j < K; ++j) ring[c][j] = 0.f;

    for (int zi = zb - R; zi < ze + R; ++zi) {
        const int gz = clampi(zi, 0, nz - 1);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (c >= ncomp) break;
            const float *src = in + c * N;
            for (int p = tid; p < SX * SY; p += NT) {
                const int hx = p % SX, hy = p / SX;
                const int gx = clampi(x0 - R + hx, 0, nx - 1), gy = clampi(y0 - R + hy, 0, ny - 1);
                S[c][hy][hx] = __ldg(src + vox(gx, gy, gz, nx, ny));
            }
        }
        __syncthreads();
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (c >= ncomp) break;
            for (int p = tid; p < SY * TX; p += NT) {
                const int hy = p / TX, xx = p % TX;
                float acc = 0.f;
#pragma unroll
                for (int j = 0; j < K; ++j) acc = fmaf(w[j], S[c][hy][xx + j], acc);
                X[c][hy][xx] = acc;
            }
        }
        __syncthreads();
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (c >= ncomp) break;
            float acc = 0.f;
#pragma unroll
            for (int j = 0; j < K; ++j) acc = fmaf(w[j], X[c][ty + j][tx], acc);
#pragma unroll
            for (int j = 0; j < K - 1; ++j) ring[c][j] = ring[c][j + 1];
            ring[c][K - 1] = acc;
            const int zo = zi - R;
            if (zo >= zb && act) {
                float o = 0.f;
#pragma unroll
                for (int j = 0; j < K; ++j) o = fmaf(w[j], ring[c][j], o);
                out[c * N + vox(x, y, zo, nx, ny)] = o;
            }
        }
    }
}

// ---- one-pass G(du) + composite update (the fused kernel family) ----------
// A CTA (32 x 8 threads) filters the three components of a DVF over a 32 x 16
// column; each thread owns two adjacent output rows.  Per input plane one TMA
// box (x from x0 - ML, ML = R rounded up to 4 so the start is 16-byte
// aligned; y from y0 - R) lands in a 6-stage ring.  x pass: each task
// filters 4 adjacent outputs of one row from 16-byte shared loads; y pass:
// two rows from 2R+2 loads; z pass: a (2R+1)-deep register ring whose slots
// are fixed at compile time by unrolling the plane loop 2R+1 times.  One
// barrier per plane.  The z-pass result is the smoothed du at (x, y, z); the
// epilogue applies Algorithm A step 3 there, u_new = du + u(x + du), so the
// smoothed du never goes back to memory.
constexpr int SY = 16;                 // output rows per CTA (2 per thread)

template <int R>
struct SmoothGeom {
    static constexpr int NC = 3;
    static constexpr int ML = (R + 3) / 4 * 4;
    static constexpr int BXW = TX + 2 * ML;
    static constexpr int BY = SY + 2 * R;
    static constexpr int ST = 6;                                    // pipeline stages
    static constexpr int STAGE = (NC * BY * BXW + 31) / 32 * 32;   // floats per stage
    static constexpr int NV = (4 + R + ML + 3) / 4;                // float4 per x task
    static constexpr int XB = NC * BY * TX;                          // floats per X buffer
    static constexpr int NTASK = NC * BY * (TX / 4);                 // x-pass tasks per plane
    static constexpr int TPT = (NTASK + NT - 1) / NT;                // tasks per thread
    static constexpr size_t bytes() {
        return sizeof(float) * ((size_t)ST * STAGE + 2 * XB) + ST * sizeof(uint64_t) + 128;
    }
};

__device__ __forceinline__ float trilinear_at(const float *__restrict__ f, size_t b0, int ddx, int ddy,
                                              int ddz, float wx, float wy, float wz) {
    const float c000 = __ldg(f + b0), c100 = __ldg(f + b0 + ddx), c010 = __ldg(f + b0 + ddy),
                c110 = __ldg(f + b0 + ddy + ddx), c001 = __ldg(f + b0 + ddz), c101 = __ldg(f + b0 + ddz + ddx),
                c011 = __ldg(f + b0 + ddz + ddy), c111 = __ldg(f + b0 + ddz + ddy + ddx);
    const float e00 = fmaf(wx, c100 - c000, c000), e10 = fmaf(wx, c110 - c010, c010);
    const float e01 = fmaf(wx, c101 - c001, c001), e11 = fmaf(wx, c111 - c011, c011);
    const float f0 = fmaf(wy, e10 - e00, e00), f1 = fmaf(wy, e11 - e01, e01);
    return fmaf(wz, f1 - f0, f0);
}

template <int R>
__global__ void __launch_bounds__(NT) k_smooth_compose_tma(const __grid_constant__ CUtensorMap tin,
                                                           const float *__restrict__ ucomp, int mode,
                                                           float *__restrict__ out, Taps taps, int nx, int ny,
                                                           int nz, int zchunk, const int *stop_flag, int *err) {
    if (stop_flag && *stop_flag) return;
    using G = SmoothGeom<R>;
    constexpr int NC = G::NC;
    constexpr int BY = G::BY, BXW = G::BXW, ML = G::ML, STAGE = G::STAGE, NV = G::NV, K = 2 * R + 1;
    constexpr int ST = G::ST, TPT = G::TPT;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float *stage = reinterpret_cast<float *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    float *Xb = stage + ST * STAGE;                                 // [2][NC][BY][TX]
    uint64_t *bar = reinterpret_cast<uint64_t *>(Xb + 2 * G::XB);

    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX + tx;
    const size_t N = (size_t)nx * ny * nz, nxy = (size_t)nx * ny;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * SY;
    const int zb = (int)blockIdx.z * zchunk, ze = min(zb + zchunk, nz);
    const int P = (ze - zb) + 2 * R;
    const int x = x0 + tx, ya = y0 + 2 * ty;                        // rows ya, ya + 1
    const bool acta = x < nx && ya < ny, actb = x < nx && ya + 1 < ny;
    const bool xin = (x0 - R >= 0) && (x0 + TX + R <= nx);
    const uint32_t tx_bytes = (uint32_t)(NC * BY * BXW * sizeof(float));

    float2 w2[K];
#pragma unroll
    for (int j = 0; j < K; ++j) w2[j] = make_float2(taps.w[j], taps.w[j]);
    float2 ring[NC][K];                                             // {row ya, row ya+1}
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int j = 0; j < K; ++j) ring[c][j] = make_float2(0.f, 0.f);

    // x-pass tasks of this thread (the same in every plane): row offset in a
    // stage, first column of its 4 outputs, destination offset in X
    int t_row[TPT], t_g4[TPT], t_dst[TPT];
#pragma unroll
    for (int q = 0; q < TPT; ++q) {
        const int task = tid + q * NT;
        const int g = task & (TX / 4 - 1), row = task >> 3;         // row = c * BY + hy
        const int c = row / BY, hy = row - c * BY;
        const int ly = clampi(y0 - R + hy, 0, ny - 1) - (y0 - R);
        t_row[q] = task < G::NTASK ? (c * BY + ly) * BXW : -1;
        t_g4[q] = 4 * g;
        t_dst[q] = row * TX + 4 * g;
    }
    const int xlim = nx - x0 + ML;        // first local column beyond the volume's last x
    float *outp[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) outp[c] = out + (size_t)c * N + (size_t)ya * nx + x;

    auto issue = [&](int q) {
        const int sidx = q % ST;
        const int z = clampi(zb - R + q, 0, nz - 1);
        mbar_expect_tx(&bar[sidx], tx_bytes);
        tma_load_4d(stage + sidx * STAGE, &tin, x0 - ML, y0 - R, z, 0, &bar[sidx]);
    };
    if (tid == 0) {
        for (int q = 0; q < ST; ++q) mbar_init(&bar[q], 1);
        fence_mbar_init();
    }
    __syncthreads();
    int issued = 0;
    if (tid == 0)
        for (; issued < ST && issued < P; ++issued) issue(issued);

    bool aborted = false;
    int tw = 0;                         // plane being waited for
    int sidx = 0;                       // its stage
    uint32_t par = 0;                   // and the phase parity of that stage
    for (int t0 = 0; t0 < P && !aborted; t0 += K) {
#pragma unroll
        for (int r = 0; r < K; ++r) {
            const int t = t0 + r;
            if (t >= P) break;
            tw = t;
            const bool ok = mbar_wait_bounded(&bar[sidx], par);
            const float *S = stage + sidx * STAGE;
            float *X = Xb + (t & 1) * G::XB;
            // x pass: 4 adjacent outputs per task, paired FMAs
#pragma unroll
            for (int q = 0; q < TPT; ++q) {
                if (t_row[q] < 0) continue;
                const float *src = S + t_row[q];
                float2 o01 = make_float2(0.f, 0.f), o23 = make_float2(0.f, 0.f);
                float v[4 * NV];
#pragma unroll
                for (int h = 0; h < NV; ++h) {
                    const float4 f = reinterpret_cast<const float4 *>(src + t_g4[q])[h];
                    v[4 * h] = f.x; v[4 * h + 1] = f.y; v[4 * h + 2] = f.z; v[4 * h + 3] = f.w;
                }
                if (!xin) {
                    // the box crosses an x border of the volume (its copy holds
                    // zeros there): the taps outside take the border value
#pragma unroll
                    for (int g = 0; g < ML; g += 4)            // left: x0 = 0, the first ML / 4 tasks of a row
                        if (x0 == 0 && t_g4[q] == g) {
#pragma unroll
                            for (int k = 0; k < ML - g; ++k) v[k] = v[ML - g];
                        }
                    if (t_g4[q] + 4 * NV > xlim) {             // right: columns from xlim on lie beyond nx - 1
                        const float b = src[xlim - 1];
#pragma unroll
                        for (int k = 0; k < 4 * NV; ++k) v[k] = t_g4[q] + k >= xlim ? b : v[k];
                    }
                }
#pragma unroll
                for (int j = 0; j < K; ++j) {
                    if ((j + ML - R) % 2 == 0) {       // operand pairs register-aligned: paired FMAs
                        o01 = __ffma2_rn(w2[j], make_float2(v[j + ML - R], v[j + 1 + ML - R]), o01);
                        o23 = __ffma2_rn(w2[j], make_float2(v[j + 2 + ML - R], v[j + 3 + ML - R]), o23);
                    } else {                           // odd offset: scalar FMAs (same rounding, no moves)
                        o01.x = fmaf(w2[j].x, v[j + ML - R], o01.x);
                        o01.y = fmaf(w2[j].x, v[j + 1 + ML - R], o01.y);
                        o23.x = fmaf(w2[j].x, v[j + 2 + ML - R], o23.x);
                        o23.y = fmaf(w2[j].x, v[j + 3 + ML - R], o23.y);
                    }
                }
                reinterpret_cast<float4 *>(X + t_dst[q])[0] = make_float4(o01.x, o01.y, o23.x, o23.y);
            }
            if (__syncthreads_or(!ok)) { aborted = true; break; }
            if (tid == 0 && issued < P) {
                fence_proxy_async();
                issue(issued);
                ++issued;
            }
            if (++sidx == ST) { sidx = 0; par ^= 1u; }
            // y pass into the ring slot of this plane, z pass for plane t - 2R
            float2 res[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const float *col = X + (c * BY + 2 * ty) * TX + tx;
                float yin[K + 1];
#pragma unroll
                for (int j = 0; j <= K; ++j) yin[j] = col[j * TX];
                float2 a = make_float2(0.f, 0.f);
#pragma unroll
                for (int j = 0; j < K; ++j) {
                    if (j % 2 == 0) {
                        a = __ffma2_rn(w2[j], make_float2(yin[j], yin[j + 1]), a);
                    } else {
                        a.x = fmaf(w2[j].x, yin[j], a.x);
                        a.y = fmaf(w2[j].x, yin[j + 1], a.y);
                    }
                }
                ring[c][r] = a;
                float2 o = make_float2(0.f, 0.f);
#pragma unroll
                for (int j = 0; j < K; ++j) o = __ffma2_rn(w2[j], ring[c][(r + 1 + j) % K], o);
                res[c] = o;
            }
            if (t >= 2 * R) {
                const int zo = zb + t - 2 * R;
                const size_t zoff = (size_t)zo * nxy;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (!(h == 0 ? acta : actb)) continue;
                    const size_t off = zoff + (size_t)h * nx;
                    const int y = ya + h;
                    const size_t i = off + (size_t)ya * nx + x;
                    const float dx = h ? res[0].y : res[0].x, dy = h ? res[1].y : res[1].x,
                                dz = h ? res[2].y : res[2].x;
                    float ax, ay, az;
                    if (mode == CGDIR_ADDITIVE) {
                        ax = __ldg(ucomp + i); ay = __ldg(ucomp + N + i); az = __ldg(ucomp + 2 * N + i);
                    } else {
                        const Corners cc = corners((float)x + dx, (float)y + dy, (float)zo + dz, nx, ny, nz);
                        const int ddx = cc.x1 - cc.x0, ddy = (cc.y1 - cc.y0) * nx, ddz = (cc.z1 - cc.z0) * nx * ny;
                        const size_t b0 = ((size_t)cc.z0 * ny + cc.y0) * nx + cc.x0;
                        ax = trilinear_at(ucomp, b0, ddx, ddy, ddz, cc.wx, cc.wy, cc.wz);
                        ay = trilinear_at(ucomp + N, b0, ddx, ddy, ddz, cc.wx, cc.wy, cc.wz);
                        az = trilinear_at(ucomp + 2 * N, b0, ddx, ddy, ddz, cc.wx, cc.wy, cc.wz);
                    }
                    outp[0][off] = dx + ax;
                    outp[0][N + off] = dy + ay;
                    outp[0][2 * N + off] = dz + az;
                }
            }
        }
    }
    if (aborted) {
        // a wait ran out: record it, drain the loads still in flight (bounded), leave
        if (tid == 0) {
            atomicExch(err, 1);
            for (int q = tw; q < issued; ++q)
                mbar_wait_bounded(&bar[q % ST], (uint32_t)((q / ST) & 1));
        }
        __syncthreads();
    }
}

// ---- z-march (one component per CTA) ---------------------------------------
// A CTA of 128 threads filters a 32-wide, 8 RY-high column of one component
// and marches along z, one barrier per plane:
//  * the input plane of the column plus its halo lands in a ring of ST
//    stages: one TMA box (x from x0 - ML, ML = R rounded up to 4 so that the
//    start is 16-byte aligned; y from y0 - R), or, where no tensor map is
//    possible (nx % 4 != 0, a misaligned field), 4-byte cp.async copies with
//    clamped indices that arrive on the same mbarrier;
//  * x pass: a task is 8 adjacent outputs of one box row (16-byte loads,
//    56 FMAs at R = 3, the register-aligned half of them paired); the clamp
//    at the volume's x borders is a select on the loaded values taken by the
//    CTAs there (the TMA box is zero-filled outside), the clamp in y a
//    remapped row, in z a clamped plane;
//  * y pass: a thread takes a column pair and RY rows: 2R + RY 8-byte loads
//    of the pair, paired FMAs only;
//  * z pass: the last 2R + 1 y-pass results of those 2 RY outputs stay in
//    registers (slots fixed at compile time by unrolling the plane loop
//    2R + 1 times), paired FMAs, one 8-byte store per row.
// The taps are symmetric, so R + 1 pairs of them are held.  Box rows and
// x-pass rows are an odd number of 16-byte units wide and consecutive tasks
// take consecutive rows, so the 16-byte accesses of every quarter-warp fall
// in distinct bank groups.
//
// Bound by shared-memory bandwidth, issue and the per-plane chain together
// (512x512x160, sigma 1: DRAM 69 %, shared memory 65 %, issue 0.61), so the
// tile is chosen to cut all three: four rows per thread need 10 instead of 16
// loads in the y pass per 8 outputs and a 38 / 32 instead of 22 / 16 x-pass
// halo (28 instead of 38 thread instructions per output), and five small CTAs
// per SM (94 registers, 40 KB of shared memory) have five independent
// barriers to wait at.  Per three-component field, against the 64 x 16 tile
// with two rows per thread and 256 threads that it replaces (z chunks each
// side's best): 512x512x160 215 -> 172 us, 256x256x96 43 -> 33, 240x160x70
// 24.6 -> 20.5.  Also measured at 512x512x160: 64 x 32 tiles of 256 threads 183 us
// (2 CTAs per SM), 64 x 32 at 3 CTAs (80 registers, spills) 251, 32 x 24 172 but
// slower at 256x256x96, 32 x 16 194, a fifth warp for the x pass 189, the x pass
// one plane ahead of the y / z passes 189.
// RY = 2 is the 32 x 16 tile: radii 5 and 6, whose z ring would not fit four
// rows' registers, and the MARCH32 variant.  At radius 4 the copy-fed forms
// spill (48 bytes with RY = 4, 32 with RY = 2); no other form does.
constexpr int MT = 128;                // threads
constexpr int MX = 32;                 // tile width
template <int R, int RY>
struct MarchGeom {
    static constexpr int K = 2 * R + 1;
    static constexpr int WY = 8 * RY, BY = WY + 2 * R;          // tile height, box rows
    static constexpr int ML = (R + 3) / 4 * 4;                  // x margin of the box
    static constexpr int W = MX + 2 * ML + 4;                   // box and x-pass row: 11 or 13 units of 16 bytes
    static constexpr int ST = RY == 4 ? 4 : 6;                  // stages
    static constexpr int STAGE = (BY * W + 31) / 32 * 32;       // floats per stage (128-byte multiple)
    static constexpr int XB = BY * W;                           // floats per x-pass buffer
    static constexpr int NTASK = BY * (MX / 8);                 // x-pass tasks per plane
    static constexpr int TPT = (NTASK + MT - 1) / MT;
    static constexpr int CTAS = RY == 4 ? (R <= 3 ? 5 : 4) : (R <= 4 ? 6 : 4);   // resident per SM (registers)
    static constexpr size_t bytes() {
        return sizeof(float) * ((size_t)ST * STAGE + 2 * (size_t)XB) + ST * sizeof(uint64_t) + 128;
    }
    static_assert(W / 4 % 2 == 1, "odd number of 16-byte units per row");
};

// SELF: the self-test's form, in which the loads of plane `hold` are never
// issued and every wait ends after `limit` cycles.
template <int R, int RY, bool ASYNC, bool SELF = false>
__global__ void __launch_bounds__(MT, RY == 4 ? 4 : MarchGeom<R, RY>::CTAS)
    k_smooth_march(const __grid_constant__ CUtensorMap tin, const float *__restrict__ in, float *__restrict__ out,
                   Taps taps, int nx, int ny, int nz, int zchunk, const int *stop_flag, int *err, int hold = -1,
                   long long limit = kWaitLimitCycles) {
    if (stopped(stop_flag)) return;      // (acted on later, the kernel takes 21 registers more and a CTA less)
    using G = MarchGeom<R, RY>;
    constexpr int K = G::K, BY = G::BY, ML = G::ML, W = G::W, ST = G::ST, STAGE = G::STAGE, XB = G::XB, TPT = G::TPT;
    constexpr int NV = 8 + 2 * ML;                               // loaded values of an x task
    extern __shared__ __align__(128) float wsm[];
    // 128-byte aligned base for the TMA stages, still a shared-memory pointer
    const int pad = (int)(((128u - (smem_u32(wsm) & 127u)) & 127u) >> 2);
    float *stage0 = wsm + pad;                                   // [ST][STAGE]
    float *xbuf = stage0 + ST * STAGE;                           // [2][BY][W]
    uint64_t *bar = reinterpret_cast<uint64_t *>(xbuf + 2 * XB);

    const int tid = threadIdx.x;
    const int x0 = blockIdx.x * MX, y0 = blockIdx.y * G::WY;
    const int nchunks = (nz + zchunk - 1) / zchunk;
    const int chunk = (int)blockIdx.z % nchunks, comp = (int)blockIdx.z / nchunks;
    const int zb = chunk * zchunk, ze = min(zb + zchunk, nz);
    const int P = (ze - zb) + 2 * R;
    const size_t nxy = (size_t)nx * ny;

    float2 w2[R + 1];
#pragma unroll
    for (int j = 0; j <= R; ++j) w2[j] = make_float2(taps.w[j], taps.w[j]);
    auto tap = [&](int j) { return w2[j <= R ? j : 2 * R - j]; };

    // x-pass tasks of this thread (fixed for every plane)
    int xsrc[TPT], xdst[TPT];
    bool xt[TPT];
#pragma unroll
    for (int q = 0; q < TPT; ++q) {
        const int task = tid + q * MT, row = task % BY, g = task / BY;
        xt[q] = task < G::NTASK;
        // the clamped source row (the asynchronous copies are clamped themselves)
        const int srow = ASYNC ? row : clampi(y0 - R + row, 0, ny - 1) - (y0 - R);
        xsrc[q] = srow * W + 8 * g;
        xdst[q] = row * W + 8 * g;
    }
    const bool xedge = !ASYNC && (x0 == 0 || x0 + MX + R > nx); // the same for the whole CTA
    // y / z pass: column pair and RY rows of this thread
    const int yc = 2 * (tid % (MX / 2)), yr = RY * (tid / (MX / 2));
    const int gx = x0 + yc, gy = y0 + yr;
    const int nact = gx < nx ? min(max(ny - gy, 0), RY) : 0;     // rows inside the volume
    float *optr = out + (size_t)comp * nxy * nz + (size_t)zb * nxy + (size_t)gy * nx + gx;

    // issue the loads of plane q into the stage at offset so, completing on b
    // (one thread; with ASYNC every thread)
    auto issue = [&](int q, int so, uint64_t *b) {
        const int z = clampi(zb - R + q, 0, nz - 1);
        if (SELF && q == hold) return;
        if (!ASYNC) {
            mbar_expect_tx(b, (uint32_t)(BY * W * sizeof(float)));
            tma_load_4d(stage0 + so, &tin, x0 - ML, y0 - R, z, comp, b);
            return;
        }
        // warp w takes rows w, w + 4, ...: lane l the columns l and, for the
        // 2R further ones, 32 + l
        const int lane = tid & 31, r0 = tid >> 5;
        const float *src = in + (size_t)comp * nxy * nz + (size_t)z * nxy;
        const int ca = clampi(x0 - R + lane, 0, nx - 1), cb = clampi(x0 - R + MX + lane, 0, nx - 1);
        const uint32_t d0 = smem_u32(stage0 + so + r0 * W + ML - R + lane);
        if (y0 >= R && y0 + G::WY + R <= ny) {
            const float *pa = src + (size_t)(y0 - R + r0) * nx;
            const size_t step = (size_t)4 * nx;
#pragma unroll 5
            for (int i = 0; i < (BY + 3) / 4; ++i, pa += step) {
                if (4 * i + r0 >= BY) break;
                cp_async4(d0 + i * 16 * W, pa + ca);
                if (lane < 2 * R) cp_async4(d0 + i * 16 * W + 128, pa + cb);
            }
        } else {
            for (int i = 0; 4 * i + r0 < BY; ++i) {
                const float *pa = src + (size_t)clampi(y0 - R + r0 + 4 * i, 0, ny - 1) * nx;
                cp_async4(d0 + i * 16 * W, pa + ca);
                if (lane < 2 * R) cp_async4(d0 + i * 16 * W + 128, pa + cb);
            }
        }
        cp_async_arrive(b);
    };
    // the issuing thread: the last one that waits for every plane itself
    constexpr int kIssuer = (G::NTASK < MT ? G::NTASK : MT) - 1;
    if (tid == kIssuer) {
        for (int q = 0; q < ST; ++q) mbar_init(&bar[q], ASYNC ? MT : 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (ASYNC || tid == kIssuer)
        for (int q = 0; q < ST && q < P; ++q) issue(q, q * STAGE, bar + q);

    float2 ring[RY][K];
#pragma unroll
    for (int h = 0; h < RY; ++h)
#pragma unroll
        for (int j = 0; j < K; ++j) ring[h][j] = make_float2(0.f, 0.f);

    // x pass of one task; xend: outputs of it inside the volume
    auto xpass = [&](const float *src, float *d, bool left, int xend) {
        float v[NV];
#pragma unroll
        for (int h = 0; h < NV / 4; ++h) {
            const float4 f = *reinterpret_cast<const float4 *>(src + 4 * h);
            v[4 * h] = f.x; v[4 * h + 1] = f.y; v[4 * h + 2] = f.z; v[4 * h + 3] = f.w;
        }
        if (xedge) {                   // CTAs at an x border of the volume only (nx % 4 == 0)
#pragma unroll
            for (int k = ML - R; k < ML; ++k) v[k] = left ? v[ML] : v[k];
#pragma unroll
            for (int k = 4 + ML; k < 8 + ML + R; ++k) v[k] = xend == 4 ? v[3 + ML] : v[k];
#pragma unroll
            for (int k = 8 + ML; k < 8 + ML + R; ++k) v[k] = xend == 8 ? v[7 + ML] : v[k];
            if (ML > 4) {              // radii above 4 reach past the next group's first half
#pragma unroll
                for (int k = 12 + ML; k < 8 + ML + R; ++k) v[k] = xend == 12 ? v[11 + ML] : v[k];
            }
        }
        float2 o[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) o[m] = make_float2(0.f, 0.f);
#pragma unroll
        for (int j = 0; j < K; ++j) {
            constexpr int B = ML - R;
            if ((B + j) % 2 == 0) {            // operand pairs register-aligned
#pragma unroll
                for (int m = 0; m < 4; ++m)
                    o[m] = __ffma2_rn(tap(j), make_float2(v[B + j + 2 * m], v[B + j + 2 * m + 1]), o[m]);
            } else {                           // odd offset: scalar FMAs (same rounding, no moves)
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    o[m].x = fmaf(tap(j).x, v[B + j + 2 * m], o[m].x);
                    o[m].y = fmaf(tap(j).x, v[B + j + 2 * m + 1], o[m].y);
                }
            }
        }
        *reinterpret_cast<float4 *>(d) = make_float4(o[0].x, o[0].y, o[1].x, o[1].y);
        *reinterpret_cast<float4 *>(d + 4) = make_float4(o[2].x, o[2].y, o[3].x, o[3].y);
    };

    auto wait = [&](uint64_t *b, uint32_t parity) {
        return SELF ? mbar_wait_bounded(b, parity, limit) : mbar_wait_bounded(b, parity);
    };
    // tw: the plane whose wait ran out in this thread (-1: none); it skips the
    // later waits, and the CTA leaves at the next turn of the plane loop or
    // after the last plane, where its threads agree on it
    int tw = -1;
    bool leave = false;
    uint32_t par = 0;                   // phase parity of the current stage
    int so = 0, xo = 0;                 // offsets of the current stage and x-pass buffer
    uint64_t *bcur = bar;
    int t0 = 0;
    for (; t0 < P; t0 += K) {
#pragma unroll
        for (int r = 0; r < K; ++r) {
            const int t = t0 + r;
            if (t >= P) break;
            if (xt[0] && tw < 0 && !wait(bcur, par)) tw = t;
#pragma unroll
            for (int q = 0; q < TPT; ++q) {
                const int xg = xdst[q] % W;
                if (xt[q]) xpass(stage0 + so + xsrc[q], xbuf + xo + xdst[q], x0 == 0 && xg == 0, nx - x0 - xg);
            }
            if (r == 0) {
                if (__syncthreads_or(tw >= 0)) { leave = true; break; }
            } else {
                __syncthreads();
            }
            if (t + ST < P) {           // the stage just consumed takes plane t + ST
                if (ASYNC) {
                    issue(t + ST, so, bcur);
                } else if (tid == kIssuer && tw < 0) {
                    fence_proxy_async();
                    issue(t + ST, so, bcur);
                }
            }
            so += STAGE; ++bcur;
            if (so == ST * STAGE) { so = 0; bcur = bar; par ^= 1u; }
            // y pass into the plane's ring slot, z pass for plane t - 2R
            const float *col = xbuf + xo + yr * W + yc;
            float2 yin[2 * R + RY];
#pragma unroll
            for (int j = 0; j < 2 * R + RY; ++j) yin[j] = *reinterpret_cast<const float2 *>(col + j * W);
#pragma unroll
            for (int h = 0; h < RY; ++h) {
                float2 a = make_float2(0.f, 0.f);
#pragma unroll
                for (int j = 0; j < K; ++j) a = __ffma2_rn(tap(j), yin[h + j], a);
                ring[h][r] = a;
            }
            if (t >= 2 * R) {
#pragma unroll
                for (int h = 0; h < RY; ++h) {
                    float2 o = make_float2(0.f, 0.f);
#pragma unroll
                    for (int j = 0; j < K; ++j) o = __ffma2_rn(tap(j), ring[h][(r + 1 + j) % K], o);
                    if (h < nact) {
                        float *d = optr + (size_t)h * nx;
                        if (ASYNC) {              // odd rows are not 8-byte aligned
                            d[0] = o.x;
                            if (gx + 1 < nx) d[1] = o.y;
                        } else {
                            *reinterpret_cast<float2 *>(d) = o;
                        }
                    }
                }
                optr += nxy;
            }
            xo ^= XB;
        }
        if (leave) break;
    }
    if (!leave) leave = __syncthreads_or(tw >= 0);
    if (leave) {
        // record it, let the loads in flight land (bounded waits), leave.  The
        // issuer has issued the planes below qe (with ASYNC every thread has,
        // whatever its waits did), and waited for all of them but the last ST.
        if (ASYNC) cp_async_wait_all();
        if (tid == kIssuer) {
            atomicExch(err, 1);
            const int qe = min((!ASYNC && tw >= 0 ? tw : t0) + ST, P);
            for (int q = max(qe - ST, 0); q < qe; ++q) wait(&bar[q % ST], (uint32_t)((q / ST) & 1));
        }
        __syncthreads();
    }
}

// Composite update u_new = du + u(x + du) (trilinear, clamped) or u + du,
// one voxel per thread along x-y tiles marching a few planes in z.  The
// update is bound by the latency of its 24 gathers per voxel, which resident
// warps hide: 5 CTAs per SM (40 warps) rather than 4.
__global__ void __launch_bounds__(NT, 5) k_compose_tiles(const float *__restrict__ u, const float *__restrict__ du,
                                                         int mode, int nx, int ny, int nz, int zc,
                                                         float *__restrict__ out, const int *stop_flag) {
    if (stop_flag && *stop_flag) return;
    const int x = blockIdx.x * TX + threadIdx.x, y = blockIdx.y * TY + threadIdx.y;
    if (x >= nx || y >= ny) return;
    const int zb = blockIdx.z * zc, ze = min(zb + zc, nz);
    const size_t nxy = (size_t)nx * ny, N = nxy * nz;
    const float fxmax = (float)(nx - 1), fymax = (float)(ny - 1), fzmax = (float)(nz - 1);
    const size_t col = (size_t)y * nx + x;
    // the next plane's du loads while this plane's corners are gathered
    float nx0 = 0.f, ny0 = 0.f, nz0 = 0.f;
    if (zb < ze) {
        const size_t i = (size_t)zb * nxy + col;
        nx0 = __ldg(du + i); ny0 = __ldg(du + N + i); nz0 = __ldg(du + 2 * N + i);
    }
    for (int z = zb; z < ze; ++z) {
        const size_t i = (size_t)z * nxy + col;
        const float dx = nx0, dy = ny0, dz = nz0;
        if (mode == CGDIR_ADDITIVE) {
            if (z + 1 < ze) { nx0 = __ldg(du + i + nxy); ny0 = __ldg(du + N + i + nxy); nz0 = __ldg(du + 2 * N + i + nxy); }
            out[i] = __ldg(u + i) + dx;
            out[N + i] = __ldg(u + N + i) + dy;
            out[2 * N + i] = __ldg(u + 2 * N + i) + dz;
            continue;
        }
        const float px = fminf(fmaxf((float)x + dx, 0.f), fxmax);
        const float py = fminf(fmaxf((float)y + dy, 0.f), fymax);
        const float pz = fminf(fmaxf((float)z + dz, 0.f), fzmax);
        const float fx = floorf(px), fy = floorf(py), fz = floorf(pz);
        const int ix = (int)fx, iy = (int)fy, iz = (int)fz;
        const float wx = px - fx, wy = py - fy, wz = pz - fz;
        const int ddx = ix < nx - 1 ? 1 : 0, ddy = iy < ny - 1 ? nx : 0;
        const size_t ddz = iz < nz - 1 ? nxy : 0;
        const size_t b0 = (size_t)iz * nxy + (size_t)iy * nx + ix;
        float cx[8], cy[8], cz[8];
        const size_t o[8] = {0, (size_t)ddx, (size_t)ddy, (size_t)(ddy + ddx), ddz, ddz + ddx, ddz + ddy,
                             ddz + ddy + ddx};
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            cx[q] = __ldg(u + b0 + o[q]);
            cy[q] = __ldg(u + N + b0 + o[q]);
            cz[q] = __ldg(u + 2 * N + b0 + o[q]);
        }
        if (z + 1 < ze) { nx0 = __ldg(du + i + nxy); ny0 = __ldg(du + N + i + nxy); nz0 = __ldg(du + 2 * N + i + nxy); }
        auto tri = [&](const float *c) {
            const float e00 = fmaf(wx, c[1] - c[0], c[0]), e10 = fmaf(wx, c[3] - c[2], c[2]);
            const float e01 = fmaf(wx, c[5] - c[4], c[4]), e11 = fmaf(wx, c[7] - c[6], c[6]);
            const float f0 = fmaf(wy, e10 - e00, e00), f1 = fmaf(wy, e11 - e01, e01);
            return fmaf(wz, f1 - f0, f0);
        };
        out[i] = dx + tri(cx);
        out[N + i] = dy + tri(cy);
        out[2 * N + i] = dz + tri(cz);
    }
}

// The composite update for volumes below 2^31 voxels: the same arithmetic
// with 32-bit indices from per-component base pointers (one multiply-add
// per gather address, 48 registers at 5 CTAs per SM without spills).
// 512x512x160: 313 us per launch against 345 us for the 64-bit kernel at 4
// CTAs per SM; 6 CTAs per SM (40 registers) measured slower.
__global__ void __launch_bounds__(NT, 5) k_compose_tiles32(const float *__restrict__ u,
                                                                       const float *__restrict__ du, int nx, int ny,
                                                                       int nz, int zc, float *__restrict__ out,
                                                                       const int *stop_flag) {
    const bool stop = stopped(stop_flag);
    const int x = blockIdx.x * TX + threadIdx.x, y = blockIdx.y * TY + threadIdx.y;
    if (x >= nx || y >= ny) return;
    const int zb = blockIdx.z * zc, ze = min(zb + zc, nz);
    const int nxy = nx * ny, N = nxy * nz;
    const float *__restrict__ ux = u, *__restrict__ uy = u + N, *__restrict__ uz = uy + N;
    const float *__restrict__ dx_ = du, *__restrict__ dy_ = du + N, *__restrict__ dz_ = dy_ + N;
    float *__restrict__ ox = out, *__restrict__ oy = out + N, *__restrict__ oz = oy + N;
    const float fxmax = (float)(nx - 1), fymax = (float)(ny - 1), fzmax = (float)(nz - 1);
    int i = zb * nxy + y * nx + x;
    float nx0 = 0.f, ny0 = 0.f, nz0 = 0.f;
    if (zb < ze) { nx0 = __ldg(dx_ + i); ny0 = __ldg(dy_ + i); nz0 = __ldg(dz_ + i); }
    if (stop) return;
    for (int z = zb; z < ze; ++z, i += nxy) {
        const float dx = nx0, dy = ny0, dz = nz0;
        const float px = fminf(fmaxf((float)x + dx, 0.f), fxmax);
        const float py = fminf(fmaxf((float)y + dy, 0.f), fymax);
        const float pz = fminf(fmaxf((float)z + dz, 0.f), fzmax);
        const float fx = floorf(px), fy = floorf(py), fz = floorf(pz);
        const int ix = (int)fx, iy = (int)fy, iz = (int)fz;
        const float wx = px - fx, wy = py - fy, wz = pz - fz;
        const int ddx = ix < nx - 1 ? 1 : 0, ddy = iy < ny - 1 ? nx : 0, ddz = iz < nz - 1 ? nxy : 0;
        const int b0 = iz * nxy + iy * nx + ix;
        const int o[8] = {b0, b0 + ddx, b0 + ddy, b0 + ddy + ddx, b0 + ddz, b0 + ddz + ddx, b0 + ddz + ddy,
                          b0 + ddz + ddy + ddx};
        float cx[8], cy[8], cz[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            cx[q] = __ldg(ux + o[q]);
            cy[q] = __ldg(uy + o[q]);
            cz[q] = __ldg(uz + o[q]);
        }
        if (z + 1 < ze) { nx0 = __ldg(dx_ + i + nxy); ny0 = __ldg(dy_ + i + nxy); nz0 = __ldg(dz_ + i + nxy); }
        auto tri = [&](const float *c) {
            const float e00 = fmaf(wx, c[1] - c[0], c[0]), e10 = fmaf(wx, c[3] - c[2], c[2]);
            const float e01 = fmaf(wx, c[5] - c[4], c[4]), e11 = fmaf(wx, c[7] - c[6], c[6]);
            const float f0 = fmaf(wy, e10 - e00, e00), f1 = fmaf(wy, e11 - e01, e01);
            return fmaf(wz, f1 - f0, f0);
        };
        ox[i] = dx + tri(cx);
        oy[i] = dy + tri(cy);
        oz[i] = dz + tri(cz);
    }
}

// ---- 3-D tile version (small volumes) ------------------------------------
// A CTA loads a 16 x 16 x 8 output tile of one component with its R-voxel
// halo into shared memory (clamped indices) and runs the x, y and z passes
// there; no z march, so a small level's whole volume is filtered in one
// short wave instead of a long chain of plane steps.
constexpr int QX = 16, QY = 16, QZ = 8;

template <int R>
struct TileGeom {
    static constexpr int AX = QX + 2 * R, AY = QY + 2 * R, AZ = QZ + 2 * R;
    static constexpr int IN = AX * AY * AZ;            // input with halo
    static constexpr int XO = QX * AY * AZ;            // after the x pass
    static constexpr int YO = QX * QY * AZ;            // after the y pass (reuses the input buffer)
    static constexpr size_t bytes() { return sizeof(float) * ((size_t)IN + XO); }
};

template <int R>
__global__ void __launch_bounds__(NT) k_smooth_tile(const float *__restrict__ in, float *__restrict__ out,
                                                    Taps taps, int nx, int ny, int nz, int tiles_z,
                                                    const int *stop_flag) {
    if (stop_flag && *stop_flag) return;
    using G = TileGeom<R>;
    constexpr int K = 2 * R + 1, AX = G::AX, AY = G::AY;
    extern __shared__ float sm[];
    float *A = sm, *B = sm + G::IN;
    const int tid = threadIdx.x + threadIdx.y * blockDim.x;
    const int comp = blockIdx.z / tiles_z, tz = blockIdx.z % tiles_z;
    const int x0 = blockIdx.x * QX, y0 = blockIdx.y * QY, z0 = tz * QZ;
    const size_t nxy = (size_t)nx * ny;
    const float *src = in + (size_t)comp * nxy * nz;
    // batches of loads in flight before their stores (a load-then-store loop
    // would wait out one memory latency per element)
    constexpr int kBatch = 16;
    for (int p0 = 0; p0 < G::IN; p0 += kBatch * NT) {
        float v[kBatch];
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            const int p = p0 + b * NT + tid;
            if (p < G::IN) {
                const int hx = p % AX, hy = (p / AX) % AY, hz = p / (AX * AY);
                const int gx = clampi(x0 - R + hx, 0, nx - 1), gy = clampi(y0 - R + hy, 0, ny - 1),
                          gz = clampi(z0 - R + hz, 0, nz - 1);
                v[b] = __ldg(src + (size_t)gz * nxy + (size_t)gy * nx + gx);
            }
        }
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            const int p = p0 + b * NT + tid;
            if (p < G::IN) A[p] = v[b];
        }
    }
    __syncthreads();
    for (int p = tid; p < G::XO; p += NT) {            // x pass: [AZ][AY][QX]
        const int ox = p % QX, r = p / QX;
        const float *row = A + r * AX + ox;
        float acc = 0.f;
#pragma unroll
        for (int j = 0; j < K; ++j) acc = fmaf(taps.w[j], row[j], acc);
        B[p] = acc;
    }
    __syncthreads();
    for (int p = tid; p < G::YO; p += NT) {            // y pass: [AZ][QY][QX] into A
        const int ox = p % QX, oy = (p / QX) % QY, hz = p / (QX * QY);
        const float *colp = B + (hz * AY + oy) * QX + ox;
        float acc = 0.f;
#pragma unroll
        for (int j = 0; j < K; ++j) acc = fmaf(taps.w[j], colp[j * QX], acc);
        A[p] = acc;
    }
    __syncthreads();
    float *dst = out + (size_t)comp * nxy * nz;
    for (int p = tid; p < QX * QY * QZ; p += NT) {      // z pass to memory
        const int ox = p % QX, oy = (p / QX) % QY, oz = p / (QX * QY);
        const int gx = x0 + ox, gy = y0 + oy, gz = z0 + oz;
        if (gx >= nx || gy >= ny || gz >= nz) continue;
        const float *colp = A + (oz * QY + oy) * QX + ox;
        float acc = 0.f;
#pragma unroll
        for (int j = 0; j < K; ++j) acc = fmaf(taps.w[j], colp[j * QX * QY], acc);
        dst[(size_t)gz * nxy + (size_t)gy * nx + gx] = acc;
    }
}

// ---- split version: xy pass and z pass as two kernels ------------------------
// k_smooth_xy filters planes in x and y: a CTA takes a 32 x 32 output tile
// of one component over a few consecutive planes; each plane's tile plus its
// R-voxel halo is loaded (clamped indices, positions precomputed once; the
// next plane's loads are issued before the current plane is filtered) into
// shared memory, filtered along x in 4-output register blocks and along y in
// 4-row register blocks.  k_smooth_z marches each (x, y) column through z
// with the three components' last 2R+1 values in registers and, for the
// du field, applies the composite update (Algorithm A step 3) on the spot:
// the z pass is where all three smoothed components of a voxel first meet,
// so the update costs no extra pass over memory.
constexpr int XYT = 32;                // xy output tile (32 x 32)
constexpr int XYZ = 4;                 // planes per CTA in the xy pass

template <int R>
__global__ void __launch_bounds__(NT) k_smooth_xy(const float *__restrict__ in, float *__restrict__ out, Taps taps,
                                                  int nx, int ny, int nz, int zgroups, const int *stop_flag) {
    if (stop_flag && *stop_flag) return;
    constexpr int K = 2 * R + 1, AX = XYT + 2 * R, AY = XYT + 2 * R, NA = AX * AY;
    constexpr int LPT = (NA + NT - 1) / NT;          // loads per thread per plane
    constexpr int XT = AY * (XYT / 4);               // x-pass tasks (4 outputs each)
    __shared__ float A[NA];
    __shared__ __align__(16) float B[AY * XYT];
    const int tid = threadIdx.y * TX + threadIdx.x;
    const int x0 = blockIdx.x * XYT, y0 = blockIdx.y * XYT;
    const int comp = blockIdx.z / zgroups, zb = (blockIdx.z % zgroups) * XYZ, ze = min(zb + XYZ, nz);
    const size_t nxy = (size_t)nx * ny, N = nxy * nz;
    const float *src = in + (size_t)comp * N;
    float *dst = out + (size_t)comp * N;
    int loff[LPT];
#pragma unroll
    for (int q = 0; q < LPT; ++q) {
        const int pidx = tid + q * NT;
        const int hy = pidx / AX, hx = pidx - hy * AX;
        const int gx = clampi(x0 - R + hx, 0, nx - 1), gy = clampi(y0 - R + hy, 0, ny - 1);
        loff[q] = pidx < NA ? gy * nx + gx : -1;
    }
    float pre[LPT];
#pragma unroll
    for (int q = 0; q < LPT; ++q) pre[q] = loff[q] >= 0 ? __ldg(src + (size_t)zb * nxy + loff[q]) : 0.f;
    const int tx = threadIdx.x, ty = threadIdx.y;
    for (int z = zb; z < ze; ++z) {
#pragma unroll
        for (int q = 0; q < LPT; ++q)
            if (loff[q] >= 0) A[tid + q * NT] = pre[q];
        __syncthreads();
        if (z + 1 < ze) {                            // next plane's loads fly during the passes
#pragma unroll
            for (int q = 0; q < LPT; ++q) pre[q] = loff[q] >= 0 ? __ldg(src + (size_t)(z + 1) * nxy + loff[q]) : 0.f;
        }
        for (int task = tid; task < XT; task += NT) {   // x pass: row, 4 outputs
            const int row = task >> 3, xs = (task & 7) * 4;
            const float *a = A + row * AX + xs;
            float v[4 + 2 * R];
#pragma unroll
            for (int i = 0; i < 4 + 2 * R; ++i) v[i] = a[i];
            float o0 = 0.f, o1 = 0.f, o2 = 0.f, o3 = 0.f;
#pragma unroll
            for (int j = 0; j < K; ++j) {
                o0 = fmaf(taps.w[j], v[j], o0);
                o1 = fmaf(taps.w[j], v[j + 1], o1);
                o2 = fmaf(taps.w[j], v[j + 2], o2);
                o3 = fmaf(taps.w[j], v[j + 3], o3);
            }
            *reinterpret_cast<float4 *>(B + row * XYT + xs) = make_float4(o0, o1, o2, o3);
        }
        __syncthreads();
        {                                              // y pass: column tx, rows 4ty .. 4ty+3
            float c[4 + 2 * R];
#pragma unroll
            for (int i = 0; i < 4 + 2 * R; ++i) c[i] = B[(4 * ty + i) * XYT + tx];
            float o[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int j = 0; j < K; ++j)
#pragma unroll
                for (int m = 0; m < 4; ++m) o[m] = fmaf(taps.w[j], c[j + m], o[m]);
            const int x = x0 + tx;
            if (x < nx) {
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const int y = y0 + 4 * ty + m;
                    if (y < ny) dst[(size_t)z * nxy + (size_t)y * nx + x] = o[m];
                }
            }
        }
        // the next plane overwrites A only after every thread has left the x pass
    }
}

template <int R, int NC, bool COMPOSE>
__global__ void __launch_bounds__(NT) k_smooth_z(const float *__restrict__ in, const float *__restrict__ u, int mode,
                                                 float *__restrict__ out, Taps taps, int nx, int ny, int nz,
                                                 int zchunk, const int *stop_flag) {
    if (stop_flag && *stop_flag) return;
    constexpr int K = 2 * R + 1;
    const int x = blockIdx.x * TX + threadIdx.x, y = blockIdx.y * TY + threadIdx.y;
    if (x >= nx || y >= ny) return;
    const int nchunks = (nz + zchunk - 1) / zchunk;
    const int comp = NC == 1 ? (int)blockIdx.z / nchunks : 0;
    const int zb = ((int)blockIdx.z % nchunks) * zchunk, ze = min(zb + zchunk, nz);
    const int P = (ze - zb) + 2 * R;
    const size_t nxy = (size_t)nx * ny, N = nxy * nz, col = (size_t)y * nx + x;
    const float *src = in + (size_t)comp * N + col;
    float *dst = out + (size_t)comp * N + col;
    // planes loaded ahead: two (u smoothed, per launch pair: 213x248x48 42 -> 37 us,
    // 237x213x107 87 -> 73; three 38 and 77); one where the update's gathers
    // need the registers (76 against 126: 133 -> 153 us)
    constexpr int ZAHEAD = COMPOSE ? 1 : 2;
    constexpr int M = K + ZAHEAD;         // planes t - 2r .. t and the loads in flight behind them
    float ring[NC][M];
    auto load = [&](int t, float (&v)[NC][M], int slot) {
        const size_t zo = (size_t)clampi(zb - R + t, 0, nz - 1) * nxy;
#pragma unroll
        for (int c = 0; c < NC; ++c) v[c][slot] = __ldg(src + c * N + zo);
    };
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int j = 0; j < M; ++j) ring[c][j] = 0.f;
#pragma unroll
    for (int t = 0; t < ZAHEAD; ++t)
        if (t < P) load(t, ring, t);
    const float fxmax = (float)(nx - 1), fymax = (float)(ny - 1), fzmax = (float)(nz - 1);
    for (int t0 = 0; t0 < P; t0 += M) {
#pragma unroll
        for (int r = 0; r < M; ++r) {
            const int t = t0 + r;
            if (t >= P) break;
            if (t + ZAHEAD < P) load(t + ZAHEAD, ring, (r + ZAHEAD) % M);
            if (t < 2 * R) continue;
            const int z = zb + t - 2 * R;
            float sv[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                float acc = 0.f;
#pragma unroll
                for (int j = 0; j < K; ++j) acc = fmaf(taps.w[j], ring[c][(r + ZAHEAD + 1 + j) % M], acc);
                sv[c] = acc;
            }
            const size_t i = (size_t)z * nxy;
            if (COMPOSE) {
                float a0, a1, a2;
                if (mode == CGDIR_ADDITIVE) {
                    a0 = __ldg(u + i + col); a1 = __ldg(u + N + i + col); a2 = __ldg(u + 2 * N + i + col);
                } else {
                    const float px = fminf(fmaxf((float)x + sv[0], 0.f), fxmax);
                    const float py = fminf(fmaxf((float)y + sv[NC > 1 ? 1 : 0], 0.f), fymax);
                    const float pz = fminf(fmaxf((float)z + sv[NC > 2 ? 2 : 0], 0.f), fzmax);
                    const float fx = floorf(px), fy = floorf(py), fz = floorf(pz);
                    const int ix = (int)fx, iy = (int)fy, iz = (int)fz;
                    const float wx = px - fx, wy = py - fy, wz = pz - fz;
                    const int ddx = ix < nx - 1 ? 1 : 0, ddy = iy < ny - 1 ? nx : 0;
                    const size_t ddz = iz < nz - 1 ? nxy : 0;
                    const size_t b0 = (size_t)iz * nxy + (size_t)iy * nx + ix;
                    a0 = trilinear_at(u, b0, ddx, ddy, (int)ddz, wx, wy, wz);
                    a1 = trilinear_at(u + N, b0, ddx, ddy, (int)ddz, wx, wy, wz);
                    a2 = trilinear_at(u + 2 * N, b0, ddx, ddy, (int)ddz, wx, wy, wz);
                }
                dst[i] = sv[0] + a0;
                dst[N + i] = sv[NC > 1 ? 1 : 0] + a1;
                dst[2 * N + i] = sv[NC > 2 ? 2 : 0] + a2;
            } else {
#pragma unroll
                for (int c = 0; c < NC; ++c) dst[c * N + i] = sv[c];
            }
        }
    }
}

__global__ void k_copy(const float *__restrict__ in, float *__restrict__ out, size_t n,
                       const int *stop_flag) {
    if (stop_flag && *stop_flag) return;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        out[i] = in[i];
}

unsigned flat_grid(size_t n) {
    size_t g = (n + 255) / 256;
    if (g > 152 * 16) g = 152 * 16;
    return (unsigned)(g ? g : 1);
}

}  // namespace

template <int R>
static cudaError_t smooth_compose_tma_r(const float *in, const float *ucomp, int mode, float *out, const Taps &t, int nx,
                                        int ny, int nz, const int *stop_flag, int *err, cudaStream_t s,
                                        bool *launched) {
    using G = SmoothGeom<R>;
    CUtensorMap m;
    const uint64_t dims[4] = {(uint64_t)nx, (uint64_t)ny, (uint64_t)nz, 3};
    const uint32_t box[4] = {(uint32_t)G::BXW, (uint32_t)G::BY, 1u, 3u};
    *launched = false;
    if (!encode_tensor_map(&m, in, 4, dims, box, 4)) return cudaSuccess;
    const int zc = pick_zchunk(nz, (long)((nx + TX - 1) / TX) * ((ny + SY - 1) / SY), 2, 2);
    dim3 grid((nx + TX - 1) / TX, (ny + SY - 1) / SY, (nz + zc - 1) / zc), block(TX, TY);
    const size_t smem = G::bytes();
    cudaError_t e = ensure_smem((const void *)k_smooth_compose_tma<R>, smem);
    if (e != cudaSuccess) return e;
    k_smooth_compose_tma<R><<<grid, block, smem, s>>>(m, ucomp, mode, out, t, nx, ny, nz, zc, stop_flag, err);
    *launched = true;
    note_launch();
    return cudaGetLastError();
}

static cudaError_t smooth_compose_tma(const float *in, const float *ucomp, int mode, float *out, const Taps &t, int nx,
                                      int ny, int nz, const int *stop_flag, int *err, cudaStream_t s,
                                      bool *launched) {
    switch (t.r) {
        case 1: return smooth_compose_tma_r<1>(in, ucomp, mode, out, t, nx, ny, nz, stop_flag, err, s, launched);
        case 2: return smooth_compose_tma_r<2>(in, ucomp, mode, out, t, nx, ny, nz, stop_flag, err, s, launched);
        case 3: return smooth_compose_tma_r<3>(in, ucomp, mode, out, t, nx, ny, nz, stop_flag, err, s, launched);
        case 4: return smooth_compose_tma_r<4>(in, ucomp, mode, out, t, nx, ny, nz, stop_flag, err, s, launched);
        case 5: return smooth_compose_tma_r<5>(in, ucomp, mode, out, t, nx, ny, nz, stop_flag, err, s, launched);
        case 6: return smooth_compose_tma_r<6>(in, ucomp, mode, out, t, nx, ny, nz, stop_flag, err, s, launched);
        default: *launched = false; return cudaErrorInvalidValue;
    }
}

// z chunk of the z-march for `tiles` columns (all components) with `res`
// CTAs resident per SM: the chunk count with the least estimated time.  A
// CTA marches zc + 2r planes; a plane takes it 0.3 + 0.14 m (in units of a
// full SM's plane) with m CTAs on its SM, fitted to 256x256x96 (192 columns,
// 5 resident: 1, 2, 3, 4, 6, 8, 12 chunks estimated 59, 39, 33, 43, 38, 44, 47
// us, measured 60, 39, 33, 41, 37, 41, 44); whole waves add up and the last one
// counts with the CTAs it has.  At 512x512x160 it takes the measured best too
// (4 chunks, 172 us; 1 chunk 230, 12 chunks 197).
static int march_zchunk_r(int nz, long tiles, int res, int r) {
    const long sms = sm_count(), wave = (long)res * sms;
    auto plane = [](long m) { return 0.3 + 0.14 * (double)m; };
    int best = nz;
    double bt = 0.0;
    for (int k = 1; k <= nz && k <= 128; ++k) {
        const int zc = (nz + k - 1) / k;
        const long n = tiles * ((nz + zc - 1) / zc), rem = n % wave;
        const double t = (zc + 2 * r) * ((double)(n / wave) * plane(res) + (rem ? plane((rem + sms - 1) / sms) : 0.0));
        if (k == 1 || t < bt) { bt = t; best = zc; }
    }
    return best;
}

template <int R, int RY>
static cudaError_t smooth_march_r(const float *in, float *out, int ncomp, const Taps &t, int nx, int ny, int nz,
                                  const int *stop_flag, int *err, cudaStream_t s, int zc_override, int cap) {
    using G = MarchGeom<R, RY>;
    const int tx = (nx + MX - 1) / MX, ty = (ny + G::WY - 1) / G::WY;
    CUtensorMap m{};
    const uint64_t dims[4] = {(uint64_t)nx, (uint64_t)ny, (uint64_t)nz, (uint64_t)ncomp};
    const uint32_t box[4] = {(uint32_t)G::W, (uint32_t)G::BY, 1u, 1u};
    const bool tma = nx % 4 == 0 && ((uintptr_t)out & 7) == 0 && encode_tensor_map(&m, in, 4, dims, box, 4);
    const int full = tma ? G::CTAS : 4;      // the asynchronous-copy form holds more registers
    const int res = cap > 0 ? std::min(cap, full) : full;
    const int zc = zc_override > 0 ? std::min(zc_override, nz) : march_zchunk_r(nz, (long)tx * ty * ncomp, res, R);
    const dim3 grid(tx, ty, (nz + zc - 1) / zc * ncomp);
    // a cap on CTAs per SM is a shared-memory request above 1/(cap+1) of the SM's 228 KB
    const size_t smem = std::max(G::bytes(), cap > 0 ? (size_t)(228 << 10) / (cap + 1) + 1024 : (size_t)0);
    const void *f = tma ? (const void *)k_smooth_march<R, RY, false> : (const void *)k_smooth_march<R, RY, true>;
    cudaError_t e = ensure_smem(f, smem);
    if (e != cudaSuccess) return e;
    if (tma)
        k_smooth_march<R, RY, false><<<grid, MT, smem, s>>>(m, in, out, t, nx, ny, nz, zc, stop_flag, err);
    else
        k_smooth_march<R, RY, true><<<grid, MT, smem, s>>>(m, in, out, t, nx, ny, nz, zc, stop_flag, err);
    note_launch();
    return cudaGetLastError();
}

// The z-march of a 32 x 32 x nz field (radius 3) whose plane `hold` (counted
// from the chunk's first halo plane) never arrives.
cudaError_t launch_smooth_wait_selftest(const float *in, float *out, int nz, int zchunk, int hold, bool tma,
                                        long long limit, int *err, cudaStream_t s) {
    using G = MarchGeom<3, 4>;
    CUtensorMap m{};
    const uint64_t dims[4] = {32, 32, (uint64_t)nz, 1};
    const uint32_t box[4] = {(uint32_t)G::W, (uint32_t)G::BY, 1u, 1u};
    if (tma && !encode_tensor_map(&m, in, 4, dims, box, 4)) return cudaErrorInvalidValue;
    const dim3 grid(1, 1, (nz + zchunk - 1) / zchunk);
    const Taps t = gauss_taps(1.f);
    const void *f = tma ? (const void *)k_smooth_march<3, 4, false, true> : (const void *)k_smooth_march<3, 4, true, true>;
    cudaError_t e = ensure_smem(f, G::bytes());
    if (e != cudaSuccess) return e;
    if (tma)
        k_smooth_march<3, 4, false, true><<<grid, MT, G::bytes(), s>>>(m, in, out, t, 32, 32, nz, zchunk, nullptr, err,
                                                                       hold, limit);
    else
        k_smooth_march<3, 4, true, true><<<grid, MT, G::bytes(), s>>>(m, in, out, t, 32, 32, nz, zchunk, nullptr, err,
                                                                      hold, limit);
    note_launch();
    return cudaGetLastError();
}

// The z-march: 32 x 32 tiles for radii up to 4, else (and when `narrow`) 32 x 16.
static cudaError_t smooth_march(const float *in, float *out, int ncomp, const Taps &t, int nx, int ny, int nz,
                                bool narrow, const int *stop_flag, int *err, cudaStream_t s, int zc, int cap) {
#define CGDIR_MARCH(R, RY) return smooth_march_r<R, RY>(in, out, ncomp, t, nx, ny, nz, stop_flag, err, s, zc, cap)
    switch (t.r) {
        case 1: if (narrow) CGDIR_MARCH(1, 2); else CGDIR_MARCH(1, 4);
        case 2: if (narrow) CGDIR_MARCH(2, 2); else CGDIR_MARCH(2, 4);
        case 3: if (narrow) CGDIR_MARCH(3, 2); else CGDIR_MARCH(3, 4);
        case 4: if (narrow) CGDIR_MARCH(4, 2); else CGDIR_MARCH(4, 4);
        case 5: CGDIR_MARCH(5, 2);
        case 6: CGDIR_MARCH(6, 2);
        default: return cudaErrorInvalidValue;
    }
#undef CGDIR_MARCH
}

// Without TMA the z-march's planes wait for one asynchronous copy after
// another.  With a scratch field (an iteration has one) the split kernels are
// ahead while the field between them stays in L2 (du smoothed with the update
// plus u, per iteration: 107x91x40 24 + 17 against 33 + 25 us, 181x217x91 92 + 48
// against 102 + 60, 301x213x113 167 + 95 against 202 + 121; 313x301x97, 9.1 M
// voxels, is past the line, 208 + 114 against 197 + 100).
// Without one, small volumes take the one-pass tile (53x59x24 12.3 against
// 14.3 us, 95x71x34 17.5 against 17.7; 83x157x24 is past the line, 20.0 against
// 19.8).  With TMA the z-march is never behind (64x64x24 14.3 + 11.4 against
// the tile's 15.9 + 12.4 us, 256x256x96 96 + 36 against the split's 139 + 94).
constexpr size_t kSplitVoxels = 8000000;

// Whether the grid of the split kernels or of the tile kernel, z slabs times
// components, holds a volume this deep (the z-march's always does).
static bool grid_holds(int variant, int nz, int ncomp) {
    const int slab = variant == SMOOTH_SPLIT ? XYZ : variant == SMOOTH_TILE ? QZ : 0;
    return slab == 0 || ((long)nz + slab - 1) / slab * ncomp <= 65535;
}

int smooth_auto_variant(const float *in, int nx, int ny, int nz, bool scratch) {
    const size_t N = (size_t)nx * ny * nz;
    if (nx % 4 == 0 && ((uintptr_t)in & 15) == 0) return SMOOTH_MARCH;
    if (scratch && N <= kSplitVoxels && grid_holds(SMOOTH_SPLIT, nz, 3)) return SMOOTH_SPLIT;
    return N <= 250000 && grid_holds(SMOOTH_TILE, nz, 3) ? SMOOTH_TILE : SMOOTH_MARCH;
}

int smooth_default_zchunk(int nx, int ny, int nz, int ncomp, float sigma) {
    const int r = std::max(gauss_radius(sigma), 1), wy = r <= 4 ? 32 : 16;
    const int res = nx % 4 == 0 && r <= 3 ? 5 : 4;          // as smooth_march_r has it
    return march_zchunk_r(nz, (long)((nx + MX - 1) / MX) * ((ny + wy - 1) / wy) * ncomp, res, r);
}

template <int R>
static cudaError_t smooth_tile_r(const float *in, int ncomp, const Taps &t, int nx, int ny, int nz, float *out,
                                 const int *stop_flag, cudaStream_t s) {
    const int tz = (nz + QZ - 1) / QZ;
    dim3 grid((nx + QX - 1) / QX, (ny + QY - 1) / QY, tz * ncomp), block(TX, TY);
    const size_t smem = TileGeom<R>::bytes();
    cudaError_t e = ensure_smem((const void *)k_smooth_tile<R>, smem);
    if (e != cudaSuccess) return e;
    k_smooth_tile<R><<<grid, block, smem, s>>>(in, out, t, nx, ny, nz, tz, stop_flag);
    note_launch();
    return cudaGetLastError();
}

static cudaError_t smooth_tile(const float *in, int ncomp, const Taps &t, int nx, int ny, int nz, float *out,
                               const int *stop_flag, cudaStream_t s) {
    switch (t.r) {
        case 1: return smooth_tile_r<1>(in, ncomp, t, nx, ny, nz, out, stop_flag, s);
        case 2: return smooth_tile_r<2>(in, ncomp, t, nx, ny, nz, out, stop_flag, s);
        case 3: return smooth_tile_r<3>(in, ncomp, t, nx, ny, nz, out, stop_flag, s);
        case 4: return smooth_tile_r<4>(in, ncomp, t, nx, ny, nz, out, stop_flag, s);
        case 5: return smooth_tile_r<5>(in, ncomp, t, nx, ny, nz, out, stop_flag, s);
        case 6: return smooth_tile_r<6>(in, ncomp, t, nx, ny, nz, out, stop_flag, s);
        default: return cudaErrorInvalidValue;
    }
}

static cudaError_t smooth_plain(const float *in, int ncomp, const Taps &t, int nx, int ny, int nz,
                                float *out, const int *stop_flag, cudaStream_t s) {
    const int zc = pick_zchunk(nz, (long)((nx + TX - 1) / TX) * ((ny + TY - 1) / TY), 4, 2);
    dim3 grid((nx + TX - 1) / TX, (ny + TY - 1) / TY, (nz + zc - 1) / zc), block(TX, TY);
    switch (t.r) {
        case 1: k_smooth<1><<<grid, block, 0, s>>>(in, out, ncomp, t, nx, ny, nz, zc, stop_flag); break;
        case 2: k_smooth<2><<<grid, block, 0, s>>>(in, out, ncomp, t, nx, ny, nz, zc, stop_flag); break;
        case 3: k_smooth<3><<<grid, block, 0, s>>>(in, out, ncomp, t, nx, ny, nz, zc, stop_flag); break;
        case 4: k_smooth<4><<<grid, block, 0, s>>>(in, out, ncomp, t, nx, ny, nz, zc, stop_flag); break;
        case 5: k_smooth<5><<<grid, block, 0, s>>>(in, out, ncomp, t, nx, ny, nz, zc, stop_flag); break;
        case 6: k_smooth<6><<<grid, block, 0, s>>>(in, out, ncomp, t, nx, ny, nz, zc, stop_flag); break;
        default: return cudaErrorInvalidValue;
    }
    note_launch();
    return cudaGetLastError();
}

template <int R>
static cudaError_t smooth_split_r(const float *in, const float *u, int mode, bool compose, int ncomp, const Taps &t,
                                  int nx, int ny, int nz, float *out, float *scratch, int zc_override,
                                  const int *stop_flag, cudaStream_t s) {
    const int zgroups = (nz + XYZ - 1) / XYZ;
    dim3 g1((nx + XYT - 1) / XYT, (ny + XYT - 1) / XYT, zgroups * ncomp), block(TX, TY);
    k_smooth_xy<R><<<g1, block, 0, s>>>(in, scratch, t, nx, ny, nz, zgroups, stop_flag);
    const long tiles = (long)((nx + TX - 1) / TX) * ((ny + TY - 1) / TY);
    const int zc = zc_override > 0 ? std::min(zc_override, nz) : pick_zchunk(nz, tiles, 8, 1);
    const int nch = (nz + zc - 1) / zc;
    if (compose) {
        dim3 g2((nx + TX - 1) / TX, (ny + TY - 1) / TY, nch);
        k_smooth_z<R, 3, true><<<g2, block, 0, s>>>(scratch, u, mode, out, t, nx, ny, nz, zc, stop_flag);
    } else if (ncomp == 3) {
        dim3 g2((nx + TX - 1) / TX, (ny + TY - 1) / TY, nch);
        k_smooth_z<R, 3, false><<<g2, block, 0, s>>>(scratch, nullptr, 0, out, t, nx, ny, nz, zc, stop_flag);
    } else {
        dim3 g2((nx + TX - 1) / TX, (ny + TY - 1) / TY, nch * ncomp);
        k_smooth_z<R, 1, false><<<g2, block, 0, s>>>(scratch, nullptr, 0, out, t, nx, ny, nz, zc, stop_flag);
    }
    note_launch(2);
    return cudaGetLastError();
}

static cudaError_t smooth_split(const float *in, const float *u, int mode, bool compose, int ncomp, const Taps &t,
                                int nx, int ny, int nz, float *out, float *scratch, int zc, const int *stop_flag,
                                cudaStream_t s) {
    switch (t.r) {
        case 1: return smooth_split_r<1>(in, u, mode, compose, ncomp, t, nx, ny, nz, out, scratch, zc, stop_flag, s);
        case 2: return smooth_split_r<2>(in, u, mode, compose, ncomp, t, nx, ny, nz, out, scratch, zc, stop_flag, s);
        case 3: return smooth_split_r<3>(in, u, mode, compose, ncomp, t, nx, ny, nz, out, scratch, zc, stop_flag, s);
        case 4: return smooth_split_r<4>(in, u, mode, compose, ncomp, t, nx, ny, nz, out, scratch, zc, stop_flag, s);
        case 5: return smooth_split_r<5>(in, u, mode, compose, ncomp, t, nx, ny, nz, out, scratch, zc, stop_flag, s);
        case 6: return smooth_split_r<6>(in, u, mode, compose, ncomp, t, nx, ny, nz, out, scratch, zc, stop_flag, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_smooth(const float *in, int ncomp, float sigma, int nx, int ny, int nz,
                          float *out, const int *stop_flag, cudaStream_t s, int *err, SmoothChoice ch, float *scratch) {
    int variant = ch.variant;
    const Taps t = gauss_taps(sigma);
    const size_t N = (size_t)nx * ny * nz;
    if (t.r == 0) {
        k_copy<<<flat_grid(N * ncomp), 256, 0, s>>>(in, out, N * ncomp, stop_flag);
        note_launch();
        return cudaGetLastError();
    }
    if (err != nullptr) {
        if (variant == SMOOTH_AUTO && ch.zchunk == 0)
            variant = smooth_auto_variant(in, nx, ny, nz, scratch != nullptr && scratch != in && scratch != out);
        if (variant == SMOOTH_FUSED) variant = SMOOTH_TILE;     // nothing to fuse with here
        if (!grid_holds(variant, nz, ncomp)) variant = SMOOTH_MARCH;
        if (variant == SMOOTH_TILE) return smooth_tile(in, ncomp, t, nx, ny, nz, out, stop_flag, s);
        if (variant == SMOOTH_SPLIT && scratch != nullptr && scratch != in && scratch != out)
            return smooth_split(in, nullptr, 0, false, ncomp, t, nx, ny, nz, out, scratch, ch.zchunk, stop_flag, s);
        return smooth_march(in, out, ncomp, t, nx, ny, nz, variant == SMOOTH_MARCH_NARROW, stop_flag, err, s, ch.zchunk,
                            ch.ctas_per_sm);
    }
    return smooth_plain(in, ncomp, t, nx, ny, nz, out, stop_flag, s);
}

cudaError_t launch_smooth_compose(const float *du, const float *u, int mode, float sigma, int nx, int ny,
                                  int nz, float *out, float *tmp, const int *stop_flag, cudaStream_t s,
                                  int *err, bool one_pass, SmoothChoice ch) {
    const Taps t = gauss_taps(sigma);
    if (!one_pass && t.r > 0 && err != nullptr) {
        if (ch.variant == SMOOTH_AUTO && ch.zchunk == 0) ch.variant = smooth_auto_variant(du, nx, ny, nz, tmp != nullptr);
        if (ch.variant == SMOOTH_SPLIT && grid_holds(SMOOTH_SPLIT, nz, 3))   // x/y pass, then the z pass with the
                                                                              // composite update fused
            return smooth_split(du, u, mode, true, 3, t, nx, ny, nz, out, tmp, ch.zchunk, stop_flag, s);
        if (ch.variant == SMOOTH_FUSED && (size_t)nx * ny * nz < (size_t)1 << 31)   // one 3-D tile kernel
            return launch_fused_smooth_compose(du, u, mode, sigma, nx, ny, nz, out, stop_flag, err, s);
    }
    if (one_pass && t.r > 0 && err != nullptr) {
        bool launched = false;
        cudaError_t e = smooth_compose_tma(du, u, mode, out, t, nx, ny, nz, stop_flag, err, s, &launched);
        if (e != cudaSuccess || launched) return e;
    }
    // smooth du into tmp, then compose
    if (ch.variant == SMOOTH_SPLIT) ch.variant = SMOOTH_MARCH;
    cudaError_t e = launch_smooth(du, 3, sigma, nx, ny, nz, tmp, stop_flag, s, err, ch);
    if (e != cudaSuccess) return e;
    return launch_compose(u, tmp, mode, nx, ny, nz, out, stop_flag, s);
}

cudaError_t launch_compose(const float *u, const float *du, int mode, int nx, int ny, int nz,
                           float *out, const int *stop_flag, cudaStream_t s) {
    const long tiles = (long)((nx + TX - 1) / TX) * ((ny + TY - 1) / TY);
    const int zc = pick_zchunk(nz, tiles, 8, 4);
    dim3 grid((nx + TX - 1) / TX, (ny + TY - 1) / TY, (nz + zc - 1) / zc), block(TX, TY);
    if (mode != CGDIR_ADDITIVE && (size_t)nx * ny * nz < ((size_t)1 << 31)) {
        k_compose_tiles32<<<grid, block, 0, s>>>(u, du, nx, ny, nz, zc, out, stop_flag);
        note_launch();
        return cudaGetLastError();
    }
    k_compose_tiles<<<grid, block, 0, s>>>(u, du, mode, nx, ny, nz, zc, out, stop_flag);
    note_launch();
    return cudaGetLastError();
}

}  // namespace cgdir
