// Self-test of the bounded waits: the decode kernels' two wait primitives (an mbarrier wait and the grid's
// meeting) are made to run out in a harmless form -- a barrier nobody arrives at, a meeting to which one CTA
// that is counted as begun never comes -- with a small poll limit, so that the give-up branch, the
// status bit and the recovery by clada_workspace_init can be exercised without any kernel ever hanging.
#include "common.cuh"
#include "ffn_common.cuh"

namespace clada {

__global__ void __launch_bounds__(64, 1)
bounded_wait_selftest_kernel(WsCtrl *ctrl, unsigned poll_limit, int32_t *report, int32_t *status) {
    __shared__ uint64_t bar;
    __shared__ int gave_up;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bar), 1);  // one arrival expected; none will come
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        gave_up = 0;
    }
    __syncthreads();
    // every thread waits for phase 0 of the barrier, as the consumers of a ring stage do
    if (!mbar_wait(smem_u32(&bar), 0, poll_limit)) atomicOr(&gave_up, 1);
    __syncthreads();
    const bool mbar_gave_up = gave_up != 0;
    // the meeting of one CTA more than the grid has, all of them counted as begun
    const unsigned n = gridDim.x + 1u;
    if (threadIdx.x == 0) {
        grid_enter(ctrl);
        if (blockIdx.x == 0) grid_enter(ctrl);
        unsigned begun = 0;
        for (unsigned i = 0; i < kBarrierSpinLimit && begun < n; ++i)
            asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(begun) : "l"(&ctrl->started) : "memory");
    }
    const bool meeting_ok = grid_meet(ctrl, n, (int)blockIdx.x, 32, poll_limit).parts >= 0;
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        report[0] = mbar_gave_up ? 1 : 0;
        report[1] = meeting_ok ? 0 : 1;
    }
    if (threadIdx.x == 0 && (mbar_gave_up || !meeting_ok) && status) atomicOr(status, CLADA_STATUS_TIMEOUT);
}

// The meeting with CTAs that begin late, as where other work holds SMs: of n CTAs the last n_late begin only after the others
// have come to the meeting and left it, and come themselves once all have begun.
__global__ void __launch_bounds__(64, 1)
meeting_selftest_kernel(WsCtrl *ctrl, int n_late, int32_t *report, int32_t *status) {
    const unsigned n = gridDim.x, cta = blockIdx.x;
    const unsigned early = n_late > 0 ? n - (unsigned)n_late : 0u;  // n_late 0: all begin, then all come
    if (threadIdx.x == 0) {
        unsigned seen = 0, begun = 0;
        if (cta >= early)
            for (unsigned i = 0; i < kBarrierSpinLimit && seen / kMeetLeft < early; ++i)
                asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(seen) : "l"(&ctrl->arrive) : "memory");
        grid_enter(ctrl);
        if (cta >= early)
            for (unsigned i = 0; i < kBarrierSpinLimit && begun < n; ++i)
                asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(begun) : "l"(&ctrl->started) : "memory");
    }
    const GridPart mine = grid_meet(ctrl, n, (int)cta, 32);
    if (threadIdx.x == 0) {
        report[2 * cta] = mine.part;
        report[2 * cta + 1] = mine.parts;
        if (mine.parts < 0 && status) atomicOr(status, CLADA_STATUS_TIMEOUT);
    }
}

// A group of four CTAs one of which begins delay_ns after the others, longer than poll_limit polls take.
__global__ void __launch_bounds__(64, 1)
late_member_selftest_kernel(WsCtrl *ctrl, unsigned poll_limit, unsigned long long delay_ns, int32_t *report, int32_t *status) {
    unsigned *word = reinterpret_cast<unsigned *>(ctrl) + 8;
    const unsigned n = gridDim.x, cta = blockIdx.x;
    if (threadIdx.x == 0) {
        unsigned long long t0, t;
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
        t = t0;
        for (unsigned i = 0; cta == n - 1 && i < kBarrierSpinLimit && t - t0 < delay_ns; ++i) {
            __nanosleep(1000);
            asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
        }
        grid_enter(ctrl);
        __threadfence();
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(word) : "memory");
        const bool ok = group_wait(ctrl, word, 0, n, n, poll_limit);
        report[cta] = ok ? 1 : 0;
        if (!ok && status) atomicOr(status, CLADA_STATUS_TIMEOUT);
    }
    const GridPart mine = grid_meet(ctrl, n, (int)cta, 32);
    if (threadIdx.x == 0 && mine.parts > 0 && mine.part == 0) *word = 0u;
}

}  // namespace clada

using namespace clada;

extern "C" int clada_selftest_late_member(void *ws, size_t ws_bytes, uint32_t poll_limit, int32_t *report, int32_t *status,
                                          void *stream) {
    if (!ws || !report) return CLADA_ERR_NULL;
    if (ws_bytes < kWsCtrlBytes || (reinterpret_cast<uintptr_t>(ws) & 255u)) return CLADA_ERR_WORKSPACE;
    if (poll_limit < 100 || poll_limit > 1000) return CLADA_ERR_SHAPE;
    late_member_selftest_kernel<<<4, 64, 0, static_cast<cudaStream_t>(stream)>>>(static_cast<WsCtrl *>(ws), poll_limit, 5000ull * poll_limit,
                                                                              report, status);
    CLADA_CUDA_TRY(cudaGetLastError());
    return CLADA_OK;
}

extern "C" int clada_selftest_meeting(void *ws, size_t ws_bytes, int32_t n_ctas, int32_t n_late, int32_t *report,
                                      int32_t *status, void *stream) {
    if (!ws || !report) return CLADA_ERR_NULL;
    if (ws_bytes < kWsCtrlBytes || (reinterpret_cast<uintptr_t>(ws) & 255u)) return CLADA_ERR_WORKSPACE;
    if (n_ctas < 1 || n_ctas > 64 || n_late < 0 || n_late > n_ctas) return CLADA_ERR_SHAPE;  // 64: resident together
    meeting_selftest_kernel<<<n_ctas, 64, 0, static_cast<cudaStream_t>(stream)>>>(static_cast<WsCtrl *>(ws), n_late, report, status);
    CLADA_CUDA_TRY(cudaGetLastError());
    return CLADA_OK;
}

extern "C" int clada_selftest_bounded_waits(void *ws, size_t ws_bytes, uint32_t poll_limit, int32_t *report,
                                            int32_t *status, void *stream) {
    if (!ws || !report) return CLADA_ERR_NULL;
    if (ws_bytes < kWsCtrlBytes || (reinterpret_cast<uintptr_t>(ws) & 255u)) return CLADA_ERR_WORKSPACE;
    if (poll_limit == 0 || poll_limit > (1u << 20)) return CLADA_ERR_SHAPE;  // at most about a second per wait
    bounded_wait_selftest_kernel<<<2, 64, 0, static_cast<cudaStream_t>(stream)>>>(static_cast<WsCtrl *>(ws), poll_limit,
                                                                               report, status);
    CLADA_CUDA_TRY(cudaGetLastError());
    return CLADA_OK;
}
