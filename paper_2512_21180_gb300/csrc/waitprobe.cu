// Probe of the bounded-wait path every pipelined kernel of the library relies on:
// a kernel whose warps wait on a shared-memory barrier that nothing completes, with
// the caller's time limit. It exercises exactly the library's mbar_wait (timeout,
// status word, early return), so the path a real kernel takes when its pipeline
// stalls can be tested without a stalled pipeline.
#include "common.cuh"
#include "geom_impl.h"
#include "tma.cuh"

namespace cbct {
namespace {

// One CTA: thread 0 initialises a barrier expecting one arrival that never comes;
// every warp's lane 0 then waits on phase 0 with the limit. The abort flag mirrors
// what the pipelined kernels do: the first warp to give up tells the others.
__global__ void k_wait_probe(int *status, uint64_t limit_ns, int *waited_ok) {
    __shared__ __align__(8) uint64_t bar;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        abort_flag = 0;
        fence_mbar_init();
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0) {
        bool ok = false;
        if (!abort_flag) ok = mbar_wait(&bar, 0u, status, limit_ns);
        if (!ok) abort_flag = 1;
        if (ok) atomicAdd(waited_ok, 1);
    }
    __syncthreads();
}

// Three waiting warps, and a fourth that completes the barriers, run the staged kernels' tile loop:
// every thread of the three waits for the tile, the CTA votes, and a wait that gave up ends
// the loop for all of it before anything is written. late: threads from `late` on take ten times the limit, so that the others
// give up first; arrive: 0 the barrier never completes, 1 it completes at once, 2 it
// completes after three times the limit (the patient threads succeed, the others gave up). odd: the
// thread that reports odd data in the second tile (negative: none). out[thread] counts tiles taken
// normally, out[96 + thread] tiles taken as odd. Before that each warp runs three steps of the
// convolutions' loops on another barrier, a warp-wide sum in each step, and three of the forward
// projector's on a third one, which a lane leaves: out[192 + thread] is 1000 (steps of the latter) +
// 100 (steps that the thread saw alive) + lanes counted by the sums of all steps.
__global__ void k_vote_probe(int *status, uint64_t limit_ns, int late, int arrive, int odd, int *out) {
    __shared__ __align__(8) uint64_t bar, wbar, lbar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_init(&wbar, 1);
        mbar_init(&lbar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    const uint64_t limit = (int)threadIdx.x >= late ? 10 * limit_ns : limit_ns;
    const bool waits = threadIdx.x < 96;
    auto complete = [&](uint64_t *b) {  // thread 96
        if (threadIdx.x != 96 || arrive == 0) return;
        const uint64_t t0 = global_ns();
        while (arrive == 2 && global_ns() - t0 < 3 * limit_ns) {}
        mbar_arrive(b);
    };
    int steps = 0, lanes = 0;
    bool alive = true;
    for (int step = 0; step < 3; ++step) {
        if (waits) {
            mbar_wait_alive(alive, &wbar, (uint32_t)(step & 1), status, limit);
            if (alive) ++steps;
            int one = 1;
            for (int o = 16; o > 0; o >>= 1) one += __shfl_xor_sync(0xffffffffu, one, o);
            lanes += one;
        } else {
            complete(&wbar);
        }
        __syncthreads();
    }
    int passed = 0;
    if (waits) {
        for (int step = 0; step < 3; ++step) {  // (one phase: once completed, every step sees it)
            if (!mbar_wait(&lbar, 0u, status, limit)) {
                leave_warp_loop(3 - step);
                break;
            }
            ++passed;
            __syncwarp();
        }
        out[192 + threadIdx.x] = 1000 * passed + 100 * steps + lanes;
    } else {
        complete(&lbar);
    }
    __syncthreads();
    int normal = 0, odds = 0;
    bool ok = true;
    for (int tile = 0; tile < 3; ++tile) {
        if (waits) ok = mbar_wait(&bar, (uint32_t)(tile & 1), status, limit);
        else complete(&bar);
        const CtaVote v = cta_vote(!ok, ok && (int)threadIdx.x == odd && tile == 1);
        if (v.gave_up) {
            ok = false;
            break;
        }
        if (v.odd) ++odds;
        else ++normal;
        __syncthreads();
    }
    if (!ok || !waits) return;
    out[threadIdx.x] = normal;
    out[96 + threadIdx.x] = odds;
}

}  // namespace
}  // namespace cbct

using namespace cbct;

extern "C" int cbct_wait_probe(const cbct_geom *g, long long limit_ns, int *waited_ok, void *stream) {
    if (!g || !waited_ok || limit_ns < 1 || limit_ns > 100000000LL)
        return fail(CBCT_EINVAL, "cbct_wait_probe: need a geometry, a device counter and 1 <= limit_ns <= 1e8");
    k_wait_probe<<<1, 64, 0, (cudaStream_t)stream>>>(g->status, (uint64_t)limit_ns, waited_ok);
    CBCT_LAUNCH_CHECK("cbct_wait_probe");
    return 0;
}

extern "C" int cbct_vote_probe(const cbct_geom *g, long long limit_ns, int late, int arrive, int odd, int *out, void *stream) {
    if (!g || !out || limit_ns < 1 || limit_ns > 10000000LL)
        return fail(CBCT_EINVAL, "cbct_vote_probe: need a geometry, a device array and 1 <= limit_ns <= 1e7");
    k_vote_probe<<<1, 128, 0, (cudaStream_t)stream>>>(g->status, (uint64_t)limit_ns, late, arrive, odd, out);
    CBCT_LAUNCH_CHECK("cbct_vote_probe");
    return 0;
}
