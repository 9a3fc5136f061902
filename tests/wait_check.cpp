// The wait of a column pass (csrc/progress.cuh) as host threads, for the thread sanitizer: 32
// lanes wait for the row groups that another warp's lane writes and publishes, then each reads its
// own row.  The acquiring load, the releasing store and the barrier are the host's; a shuffle hands
// values on without ordering anything, as on the GPU.
#include <pthread.h>
#include <sched.h>

#include <atomic>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <thread>
#include <vector>

#include "cm_internal.h"

namespace {

thread_local struct { unsigned x; } threadIdx;
pthread_barrier_t g_warp;
std::atomic<int> g_shuffled;
int32_t v, groups;                                 // what the inline assembly below does not name

void __syncwarp() { pthread_barrier_wait(&g_warp); }

int __shfl_sync(uint32_t, int x, int lane)
{
    if ((int)threadIdx.x == lane) g_shuffled.store(x + 1, std::memory_order_relaxed);
    int y;
    while ((y = g_shuffled.load(std::memory_order_relaxed)) == 0) sched_yield();
    return y - 1;
}

void __nanosleep(unsigned) { sched_yield(); }

void host_asm(const char* text, const int32_t* at, int32_t& loaded, int32_t stored)
{
    if (std::strstr(text, "ld.acquire")) loaded = __atomic_load_n(at, __ATOMIC_ACQUIRE);
    else if (std::strstr(text, "st.release")) __atomic_store_n(const_cast<int32_t*>(at), stored, __ATOMIC_RELEASE);
}

}  // namespace

#define asm
#define volatile(...) host_asm(#__VA_ARGS__, done, v, groups)
#include "progress.cuh"
#undef volatile
#undef asm

int main()
{
    pthread_barrier_init(&g_warp, nullptr, 32);
    for (int round = 0; round < 20; ++round) {
        std::vector<int32_t> rows(32, 0);
        int32_t done = 0, err = 0;
        std::atomic<int> wrong{0};
        g_shuffled = 0;
        std::vector<std::thread> threads;
        for (int lane = 0; lane < 32; ++lane)
            threads.emplace_back([&, lane] {
                threadIdx.x = lane;
                const bool ok = cm::wait_groups(&done, 32, &err);
                if (!ok || rows[lane] != lane + 1) wrong = 1;
            });
        threads.emplace_back([&] {
            for (int r = 0; r < 32; ++r) rows[r] = r + 1;
            cm::publish_groups(&done, 32);
        });
        for (auto& t : threads) t.join();
        if (wrong) return 1;
    }
    return 0;
}
