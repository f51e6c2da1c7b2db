// Device side of the halo exchange between the co-resident blocks of a resident
// launch (resident.cu, resident_euler.cu).
#pragma once

#include <cstdint>

#include "geometry.cuh"
#include "resident.h"

namespace swp {

// Hard cap on polls of one wait, in case the global timer does not advance.
constexpr uint32_t kMaxWordPolls = 1u << 26;

__device__ __forceinline__ uint64_t clock_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// Published words: data and sequence number in one 8-byte access (FP64: two
// of them, each half of the value).
template <typename R> struct Word;
template <> struct Word<float> {
    static constexpr int N64 = 1;
    static __device__ __forceinline__ void put(uint64_t* p, float v, uint32_t seq)
    {
        const uint64_t w = (uint64_t)seq << 32 | __float_as_uint(v);
        asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
    }
    static __device__ __forceinline__ bool get(const uint64_t* p, float& v, uint32_t seq)
    {
        uint64_t w;
        asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
        v = __uint_as_float((uint32_t)w);
        return (uint32_t)(w >> 32) == seq;
    }
};
template <> struct Word<double> {
    static constexpr int N64 = 2;
    static __device__ __forceinline__ void put(uint64_t* p, double v, uint32_t seq)
    {
        const uint64_t b = (uint64_t)__double_as_longlong(v), s = (uint64_t)seq << 32;
        asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(s | (b & 0xffffffffu)),
                     "l"(s | (b >> 32))
                     : "memory");
    }
    static __device__ __forceinline__ bool get(const uint64_t* p, double& v, uint32_t seq)
    {
        uint64_t a, b;
        asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
        v = __longlong_as_double((long long)((b << 32) | (a & 0xffffffffu)));
        return (uint32_t)(a >> 32) == seq && (uint32_t)(b >> 32) == seq;
    }
};

// Point of [0, N) that stands for point g of the extended line.
__device__ __forceinline__ int64_t fold(int64_t g, int64_t N, int bc)
{
    const int64_t per = bc == PERIODIC ? N : 2 * (N - 1);
    if (g < 0 || g >= per) {
        g %= per;
        if (g < 0) g += per;
    }
    return g < N ? g : per - g;
}

// The published word, within a parity's set, of point p of [0, n): block o owns
// [o n / K, (o + 1) n / K) and publishes all its points, or pub at each end, as words
// o cap, o cap + 1, ... .  n K < 2^31.
__device__ __forceinline__ int word_of(int p, int n, int K, int pub, int cap)
{
    const int o = ((p + 1) * K - 1) / n;   // the block that owns point p
    const int b = o * n / K, own = (o + 1) * n / K - b, at = p - b;
    return o * cap + (own <= 2 * pub || at < pub ? at : at - (own - 2 * pub));
}

// Poll a word until it carries sequence number seq.  Bounded: false when the
// limit passes or another wait of the launch has given up (the status word).
template <typename R>
__device__ __forceinline__ bool wait_word(const uint64_t* w, uint32_t seq, const ResidentSync& y, R& v)
{
    uint32_t polls = 0;
    uint64_t t0 = 0;
    while (!Word<R>::get(w, v, seq)) {
        if ((++polls & 255u) == 0) {
            const uint64_t now = clock_ns();
            if (y.claimed && *reinterpret_cast<const volatile int*>(y.claimed) <= y.last_tile) {
                t0 = now;
                polls = 0;
            }
            if (t0 == 0) t0 = now;
            if (*reinterpret_cast<volatile int*>(y.status) != 0 || now - t0 > y.wait_limit_ns ||
                polls > kMaxWordPolls) {
                atomicExch(y.status, 1);
                return false;
            }
        }
    }
    return true;
}

}  // namespace swp
