// What the kernels that hold a whole step share: the control block of a launch, counters between CTAs, bounded waits.
//
// Control block (workspace, ints): [0,1] epoch of the running launch, [2] CTAs that have left, [3] abort flag (the low half of the
// epoch of the launch that gives up), then the kernel's own counters from CTRL_LINE on.  CTA 0 clears the counters and then
// publishes the launch's epoch; a CTA touches a counter only once it has seen the epoch; the last CTA to leave takes it
// back, so that a captured launch can be replayed.  Nothing is expected of what the block holds before: between two launches
// other calls, of other sizes, use the same workspace.
//
// Every wait is bounded and returns true when the waiter has to give up: the wait ran out (status RM_ERR_TIMEOUT with the
// wait's source line and the CTA), or this CTA or the grid is aborting.  The bounds are 10 s and more: a CTA that is resident
// waits for those that are not yet, which is as long as another stream's kernel holds their SMs.  (A look at a counter takes 0.16
// us when nobody else looks, one at a word in shared memory 20 ns; mbarrier.try_wait takes 0.1 to 4 us, so those waits go by the
// clock as well.)
#pragma once
#include "rm_common.cuh"
#include "rm_sm100.cuh"

namespace grid {

constexpr int CTRL_LINE = 32;
constexpr uint32_t COUNTER_POLLS = 1u << 26, SHARED_POLLS = 1u << 29, BARRIER_POLLS = 1u << 27;
// Time limit of a wait, looked at now and then (first look: the wait begins)
struct Limit {
    unsigned long long begin = 0;
    __device__ __forceinline__ bool over() {
        unsigned long long t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (!begin) begin = t;
        return t - begin > 12000000000ull;
    }
};

__device__ __forceinline__ int ld_acquire_gpu(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release_gpu(int* p, int v) {
    asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void st_release_gpu(int* p, int v) {
    asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// (A: the kernel's arguments, with `status`, `ctrl` and `epoch`)
template <class A>
__device__ __forceinline__ bool aborting(const A& a) { return ld_acquire_gpu(a.ctrl + 3) == (int)(unsigned)a.epoch; }
template <class A>
__device__ __forceinline__ void report_timeout(const A& a, volatile int* abort_cta, int line) {
    rm_set_status_at(a.status, RM_ERR_TIMEOUT, (line << 12) | (int)(blockIdx.x & 0xfffu));
    *abort_cta = 1;
    atomicExch(a.ctrl + 3, (int)(unsigned)a.epoch);
}
template <class A>
__device__ __forceinline__ bool wait_slow(uint32_t bar, uint32_t parity, int line, const A& a, volatile int* abort_cta) {
    Limit limit;
    for (uint32_t i = 0; i < BARRIER_POLLS; ++i) {
        if (sm100::mbar_try_wait(bar, parity)) return false;
        if (i > 64) __nanosleep(32);
        if ((i & 1023u) == 1023u) {
            if (*abort_cta || ((i & 16383u) == 16383u && aborting(a))) {
                *abort_cta = 1;
                return true;
            }
            if (limit.over()) break;
        }
    }
    report_timeout(a, abort_cta, line);
    return true;
}
template <class A>
__device__ __forceinline__ bool counter_wait(const int* counter, int target, int line, const A& a, volatile int* abort_cta) {
    for (uint32_t i = 0; i < COUNTER_POLLS; ++i) {
        if (ld_acquire_gpu(counter) >= target) return false;
        if ((i & 255u) == 255u && (*abort_cta || aborting(a))) { *abort_cta = 1; return true; }
    }
    report_timeout(a, abort_cta, line);
    return true;
}
template <class A>
__device__ __forceinline__ bool epoch_wait(const int* ctrl, unsigned long long epoch, int line, const A& a, volatile int* abort_cta) {
    for (uint32_t i = 0; i < COUNTER_POLLS; ++i) {
        unsigned long long v;
        asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(ctrl) : "memory");
        if (v == epoch) return false;
        if ((i & 255u) == 255u && *abort_cta) return true;
    }
    rm_set_status_at(a.status, RM_ERR_TIMEOUT, (line << 12) | (int)(blockIdx.x & 0xfffu));
    *abort_cta = 1;
    return true;
}
__device__ __forceinline__ void epoch_publish(int* ctrl, unsigned long long epoch) {
    __threadfence();
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(ctrl), "l"(epoch) : "memory");
}
// by one thread of every CTA on its way out (it has seen the epoch)
__device__ __forceinline__ void epoch_leave(int* ctrl) {
    if (atomicAdd(ctrl + 2, 1) == (int)gridDim.x - 1) {
        ctrl[3] = 0;
        asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(ctrl), "l"(0ull) : "memory");
    }
}
// OR of a predicate over the threads of a named barrier
__device__ __forceinline__ bool barrier_or(int id, int count, bool pred) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "barrier.cta.red.or.pred q, %2, %3, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r) : "r"((uint32_t)pred), "r"(id), "r"(count) : "memory");
    return r != 0;
}

}  // namespace grid

unsigned long long rm_next_epoch();        // odd, never the same twice in a process
