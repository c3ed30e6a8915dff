// A barrier over the CTAs of one cooperative launch (all of them resident at once).
//
// Each CTA's first thread adds one to a counter (release) and waits for it to reach the next multiple of
// the grid size (acquire); with the CTA barriers around it every thread's earlier writes come before
// any thread's later reads, so plain loads after the barrier see the other CTAs' stores (data that the
// kernel itself writes must not be read through const __restrict__ pointers). The wait is bounded by the global
// timer (two seconds): a run-out sets the context's status word, which the host reads at its next wait for
// the stream (sfg_wait), and the CTA returns; the others' next waits then run out too.
// Costs 1-2 us on 16-608 CTAs, against 2-3 us from the end of one launch to the work of the next (with full
// fences around the count instead of release and acquire 0.4 us more).
#pragma once
#include <cstdint>

// What a launch's barriers need from the host (sfg_grid_wait).
struct GridWait {
    int* status;        // host memory: set when a wait ran out
    uint64_t limit_ns;
    unsigned endless;   // barrier (counted from 1) whose waits only the limit ends; 0 unless a test asks
};

struct GridBar {
    unsigned* count;  // zero at launch; one word per launch
    GridWait wait;
};

__device__ __forceinline__ uint64_t gridbar_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Returns false (in every thread of the CTA) when the wait ran out. `round` counts
// the barriers this CTA has passed and starts at 0.
__device__ __forceinline__ bool grid_barrier(const GridBar& b, unsigned& round) {
    __shared__ int s_bar_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned want = (round + 1) * gridDim.x;
        // release: the CTA's writes (ordered before by the barrier above) before the count
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(b.count) : "memory");
        int ok = 1;
        uint64_t t0 = 0;
        for (unsigned spin = 0;; ++spin) {
            unsigned now;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(now) : "l"(b.count) : "memory");
            if (now >= want && b.wait.endless != round + 1) break;
            if ((spin & 255u) == 255u) {
                const uint64_t t = gridbar_ns();
                if (t0 == 0) t0 = t;
                if (t - t0 > b.wait.limit_ns) {
                    ok = 0;
                    break;
                }
            }
        }
        // The host reads the word after it has waited for the kernel: no fence. (A system-wide fence here, never
        // executed, made the forest of a 64 x 64 grid 4 us slower.)
        if (!ok) *(volatile int*)b.wait.status = 1;
        s_bar_ok = ok;
    }
    __syncthreads();
    ++round;
    return s_bar_ok != 0;
}
