// Self-test of the bounded-wait error path (an execution aid, not part of
// the paper's method).  One CTA waits on an mbarrier that nothing completes,
// with a short limit in clock cycles; when the limit runs out it records the
// timeout in the context's error word and returns -- what the TMA kernels do
// when a copy never lands.  Then the z-march smoothing runs on fields one plane
// of which is never copied: it has to report that plane wherever its wait runs
// out; and the fused tile kernel on tiles that are never copied, of a running
// and of a stopped level.  Nothing faults or hangs: every wait is bounded.
#include "runtime_internal.hpp"
#include "tma.cuh"

#include <algorithm>

using namespace cgdir;
using namespace cgdir::rt;

namespace {

__global__ void k_wait_timeout(long long limit_cycles, int *err) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const long long t0 = clock64();
        bool ok = mbar_try_wait(&bar, 0);
        while (!ok && clock64() - t0 <= limit_cycles) ok = mbar_try_wait(&bar, 0);
        if (!ok) atomicExch(err, 1);
    }
}

constexpr int nz = 20;
constexpr size_t n = nz * 32 * 32;             // >= 3 x 16 x 16 x 16

// The kernels that wait for copies, on fields some of which never arrive.
// f: 2 n floats and an int.
int lost_copies(cgdir_ctx *ctx, float *f, long long limit) {
    float *in = f, *out = in + n;
    int *stop = (int *)(out + n);
    CK(cudaMemsetAsync(in, 0, n * sizeof(float), ctx->stream));
    // first, middle and last plane of one turn of the plane loop (chunks of
    // one plane march 7 planes) and of a chunk whose last turn is cut short
    const int at[6][2] = {{1, 0}, {1, 3}, {1, 6}, {nz, 0}, {nz, 21}, {nz, 25}};
    for (const auto &q : at)
        for (int tma = 0; tma < 2; ++tma) {
            CK(launch_smooth_wait_selftest(in, out, nz, q[0], q[1], tma != 0, limit, ctx->err_word, ctx->stream));
            CK(cudaStreamSynchronize(ctx->stream));
            const int rs = check_err_word(ctx);
            if (rs == CGDIR_OK) return fail(ctx, CGDIR_ECUDA, "selftest: the z-march lost a wait that ran out");
            if (rs != CGDIR_ETIMEDOUT) return rs;
        }
    for (int stopped = 0; stopped < 2; ++stopped) {
        CK(cudaMemsetAsync(stop, stopped, sizeof(int), ctx->stream));
        CK(launch_fused_wait_selftest(in, out, stop, limit, ctx->err_word, ctx->stream));
        CK(cudaStreamSynchronize(ctx->stream));
        const int rs = check_err_word(ctx);
        if (rs == CGDIR_OK) return fail(ctx, CGDIR_ECUDA, "selftest: the fused tiles lost a wait that ran out");
        if (rs != CGDIR_ETIMEDOUT) return rs;
    }
    return CGDIR_ETIMEDOUT;
}

}  // namespace

extern "C" int cgdir_selftest_wait_timeout(cgdir_ctx *ctx, int limit_us) {
    if (!ctx) return CGDIR_EINVAL;
    ctx->err.clear();
    if (limit_us < 1 || limit_us > 2000000) return fail(ctx, CGDIR_EINVAL, "selftest: limit_us must be 1..2000000");
    DeviceGuard g(ctx->device);
    // at most 2.1 GHz: the wait lasts at least limit_us
    const long long cycles = (long long)limit_us * 2100;
    k_wait_timeout<<<1, 32, 0, ctx->stream>>>(cycles, ctx->err_word);
    note_launch();
    CK(cudaGetLastError());
    CK(cudaStreamSynchronize(ctx->stream));
    const int rc = check_err_word(ctx);
    if (rc != CGDIR_ETIMEDOUT) return rc;
    float *f = nullptr;                        // not the context's: its budget stays
    CK(cudaMalloc(&f, (2 * n + 1) * sizeof(float)));
    const int rs = lost_copies(ctx, f, std::min<long long>(cycles, 2100000));
    cudaStreamSynchronize(ctx->stream);
    cudaFree(f);
    return rs;
}
