// One warp in the bounded wait of the one-launch scans (wait_device.h, the
// kernel's own source), while a second thread raises the flag at a moment of its
// own: the lanes leave together, with the same answer, whatever that moment is.
// Test infrastructure only.
//   args: trials
#include "cuda_host.h"
#define FULLMASK 0xffffffffu
thread_local dim3e threadIdx;
dim3e blockIdx;
unsigned char *g_smem;
thread_local WarpCtx *g_warp;
SpinBarrier *g_block;
inline void __nanosleep(unsigned) { sched_yield(); }
inline void __threadfence_block() { std::atomic_thread_fence(std::memory_order_seq_cst); }
inline bool __any_sync(unsigned m, bool p) { return __ballot_sync(m, p) != 0u; }
inline void __syncwarp() { g_warp->bar.arrive_and_wait(); }
#include "wait_device.h"

int main(int argc, char **argv)
{
    const int trials = argc > 1 ? atoi(argv[1]) : 100;
    WarpCtx warp;
    SpinBarrier start(33);
    volatile int ready = 0;
    int got[32], seen[2] = {0, 0}, parted = 0, wrong = 0;
    auto trial = [&](int t, int lane) {
        threadIdx.x = lane;
        g_warp = &warp;
        const int limit = 1 + t % 40;
        start.arrive_and_wait();
        got[lane] = wait_slot(&ready, 3, limit);
        start.arrive_and_wait();
    };
    std::vector<std::thread> th;
    for (int l = 0; l < 32; ++l)
        th.emplace_back([&, l] { for (int t = 0; t < trials; ++t) trial(t, l); });
    for (int t = 0; t < trials; ++t) {
        const int kind = t % 4;                      // written before, never, or in between
        ready = kind == 0 ? 4 : 3;
        start.arrive_and_wait();
        if (kind >= 2) {
            for (int q = 0; q < (t * 7) % 50; ++q) sched_yield();
            ready = 4;
        }
        start.arrive_and_wait();
        for (int l = 1; l < 32; ++l) parted += got[l] != got[0];
        wrong += (kind == 0 && !got[0]) || (kind == 1 && got[0]);
        ++seen[got[0] != 0];
    }
    for (auto &x : th) x.join();
    printf("parted %d wrong %d reached %d gave up %d\n", parted, wrong, seen[1], seen[0]);
    return parted || wrong || !seen[0] || !seen[1];
}
