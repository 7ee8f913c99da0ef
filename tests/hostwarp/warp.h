// One warp on the host: 32 threads, each a lane, run a kernel's own source text. A vote is a barrier of relaxed
// atomics: it orders execution and gives no memory ordering, as CUDA's vote intrinsics; __syncwarp is one with
// acquire and release. Under -fsanitize=thread a shared word that one lane writes and another reads or
// writes with only votes between is reported as a data race.
#pragma once
#include <sched.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <thread>
#include <type_traits>
#include <vector>

#define __device__
#define __global__
#define __shared__
#define __forceinline__ inline
#define __align__(n)
#define __launch_bounds__(...)

using std::max;
using std::min;

struct Dim { unsigned x; };
static thread_local Dim threadIdx;
static const Dim blockDim{32}, gridDim{1}, blockIdx{0};
alignas(16) static unsigned char smem_raw[1 << 17];

struct float3 { float x, y, z; };
inline float3 make_float3(float x, float y, float z) { return {x, y, z}; }

struct Barrier {
    std::atomic<unsigned> votes{0}, arrived{0}, turn{0}, result{0};
    template <bool ORDER> unsigned meet(unsigned bit)
    {
        const unsigned t = turn.load(std::memory_order_relaxed);
        votes.fetch_or(bit, std::memory_order_relaxed);
        if (arrived.fetch_add(1, ORDER ? std::memory_order_acq_rel : std::memory_order_relaxed) == 31) {
            result.store(votes.load(std::memory_order_relaxed), std::memory_order_relaxed);
            votes.store(0, std::memory_order_relaxed);
            arrived.store(0, std::memory_order_relaxed);
            turn.store(t + 1, ORDER ? std::memory_order_release : std::memory_order_relaxed);
        } else {
            while (turn.load(ORDER ? std::memory_order_acquire : std::memory_order_relaxed) == t) sched_yield();
        }
        return result.load(std::memory_order_relaxed);
    }
};
static Barrier g_barrier;

inline unsigned __ballot_sync(unsigned, bool p) { return g_barrier.meet<false>(p ? 1u << threadIdx.x : 0u); }
inline bool __any_sync(unsigned m, bool p) { return __ballot_sync(m, p) != 0u; }
inline void __syncwarp() { g_barrier.meet<true>(0u); }
inline void __syncthreads() { __syncwarp(); }
template <class T> inline T __shfl_xor_sync(unsigned, T v, int) { return v; }   // not reached by these runs
inline int __popc(unsigned v) { return __builtin_popcount(v); }
inline float __ldg(const float *p) { return *p; }
inline int __float_as_int(float f) { int i; memcpy(&i, &f, 4); return i; }
inline float __int_as_float(int i) { float f; memcpy(&f, &i, 4); return f; }
inline uint32_t __float_as_uint(float f) { return (uint32_t)__float_as_int(f); }
inline float __uint_as_float(uint32_t i) { return __int_as_float((int)i); }
inline float __logf(float x) { return std::log(x); }
inline float __expf(float x) { return std::exp(x); }
template <class T> inline T atomicAdd(T *p, T v) { return __atomic_fetch_add(p, v, __ATOMIC_RELAXED); }
inline float atomicAdd(float *, float) { abort(); }

static std::atomic<int> g_failed{0};
#define CHECK(ok) do { if (!(ok) && !g_failed.exchange(1)) fprintf(stderr, "failed: %s (line %d)\n", #ok, __LINE__); } while (0)
inline bool checked(bool ok) { CHECK(ok); return ok; }
#define FLR_CHK(ok, site, idx) checked(ok)   // the kernels' own bounds of queue and stack

// A path of the model: how many steps it makes, which of them ask for a connection and how long its march is.
inline uint32_t mix(uint64_t pid, uint32_t step, uint32_t salt)
{
    uint64_t h = (pid + 1) * 0x9E3779B97F4A7C15ull ^ ((uint64_t)step << 20 | salt) * 0xC2B2AE3D27D4EB4Full;
    h ^= h >> 29; h *= 0xBF58476D1CE4E5B9ull; h ^= h >> 32;
    return (uint32_t)h;
}
inline uint32_t path_steps(uint64_t pid) { const uint32_t r = mix(pid, 0, 1); return r % 16 == 0 ? 60 : 1 + r % 9; }
inline bool asks(uint64_t pid, uint32_t step) { return mix(pid, step, 2) % 8 < 6; }
inline int march_steps(uint64_t pid, uint32_t step) { const uint32_t r = mix(pid, step, 3); return r % 9 == 0 ? 25 : (int)(r % 5); }

constexpr uint32_t MAX_STEPS = 64;
static std::vector<int> g_made;   // connections made, [path][step]
static void made(uint64_t pid, uint32_t step)
{
    if (!checked(pid < g_made.size() / MAX_STEPS && step < MAX_STEPS)) return;
    __atomic_fetch_add(&g_made[pid * MAX_STEPS + step], 1, __ATOMIC_RELAXED);
}

template <class Kernel> int run_warp(uint64_t n_paths, Kernel kernel)
{
    g_made.assign(n_paths * MAX_STEPS, 0);
    std::vector<std::thread> lanes;
    for (unsigned l = 0; l < 32; ++l) lanes.emplace_back([=] { threadIdx.x = l; kernel(); });
    for (auto &t : lanes) t.join();
    for (uint64_t p = 0; p < n_paths; ++p)
        for (uint32_t s = 0; s < MAX_STEPS; ++s)
            CHECK(g_made[p * MAX_STEPS + s] == (s < path_steps(p) && asks(p, s) ? 1 : 0));
    return g_failed;
}
