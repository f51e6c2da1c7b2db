// One tile of a resident heat / KS advance: registers, warp rounds through shared
// memory, halo exchange between blocks (resident.cu has the idea; used by it and
// by the batched form, resident_batch.cu).
#pragma once

#include <type_traits>

#include "resident.cuh"

namespace swp {

// Two FP32 values advanced by one instruction (add / sub / fma .f32x2, each half
// rounded as the scalar operation).  The FP32 pipe does the same operations per
// clock either way (2.2 clocks per f32x2, 1.1 per scalar FMA), but a KS level's scalar FMAs, each reading three registers, took
// 1.34 to 1.5 issue slots per operation where paired ones take 1.23 to 1.28: KS with
// 2000003 points 1190 to 1087 clocks per level, 2^20 points 3 % faster, small grids
// the same.  Heat's three operations do not pay for building the mixed pairs at a
// run's ends (475 to 520 clocks), nor do KS tiles of the batched form (11.1 to 12.2
// ms), so those stay scalar.
struct Pair {
    uint64_t b;
};
__device__ __forceinline__ Pair make_pair2(float x, float y)
{
    Pair p;
    asm("mov.b64 %0, {%1, %2};" : "=l"(p.b) : "f"(x), "f"(y));
    return p;
}
__device__ __forceinline__ float2 split(Pair p)
{
    float2 v;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(p.b));
    return v;
}
template <> struct Units<Pair> {
    Pair m2;   // -2, -2
};
template <> struct Fp<Pair> {
    using K = const Units<Pair>&;
    static __device__ __forceinline__ Pair add(Pair a, Pair b, K)
    {
        Pair r;
        asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.b) : "l"(a.b), "l"(b.b));
        return r;
    }
    static __device__ __forceinline__ Pair sub(Pair a, Pair b, K)
    {
        Pair r;
        asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.b) : "l"(a.b), "l"(b.b));
        return r;
    }
    static __device__ __forceinline__ Pair fma(Pair a, Pair b, Pair c)
    {
        Pair r;
        asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.b) : "l"(a.b), "l"(b.b), "l"(c.b));
        return r;
    }
    static __device__ __forceinline__ Pair m2(K k) { return k.m2; }
};

// A lane's run of P points in registers.  FP32 runs of a multiple of 4 points move
// to and from shared memory as 16-byte vectors.  Where PAIRS, they are Q = P / 2
// pairs, pair j the run's points j and j + Q, so that the neighbours of a pair's two
// points are the neighbouring pair's; shared memory keeps them interleaved too.
// Else they are single values.
template <typename R, int P>
constexpr bool kVector = sizeof(R) == 4 && P % 4 == 0;
template <typename R, int P, bool PAIRS> struct Run {
    using V = R;
    static constexpr int Q = P;
};
template <typename R, int P> struct Run<R, P, true> {
    static_assert(kVector<R, P>, "pairs move as vectors");
    using V = Pair;
    static constexpr int Q = P / 2;
};

// Shared-memory index of tile slot s.  Lanes read runs of P slots, all lanes
// at once, so the stride of the runs is padded to spread over the banks: vector
// runs to an odd number of 16-byte vectors, even FP64 strides by a value after
// every 16.
template <typename R, int P, bool PAIRS>
__device__ __forceinline__ int slot_at(int s)
{
    if (kVector<R, P>) {
        const int r = s / P, i = s - r * P, h = i >= P / 2;
        return r * (P + ((P / 4) % 2 ? 0 : 4)) + (PAIRS ? 2 * (i - h * (P / 2)) + h : i);
    }
    if (sizeof(R) == 8 && P % 2 == 0) return s + (s >> 4);
    return s;
}

template <typename R, int P, bool PAIRS>
__device__ __forceinline__ void load_run(const R* buf, int s, typename Run<R, P, PAIRS>::V (&u)[Run<R, P, PAIRS>::Q])
{
    if constexpr (PAIRS) {
        const ulonglong2* v = reinterpret_cast<const ulonglong2*>(buf + slot_at<R, P, PAIRS>(s));   // s a multiple of P
#pragma unroll
        for (int i = 0; i < P / 4; ++i) {
            const ulonglong2 w = v[i];
            u[2 * i].b = w.x;
            u[2 * i + 1].b = w.y;
        }
    } else if constexpr (kVector<R, P>) {
        const float4* v = reinterpret_cast<const float4*>(buf + slot_at<R, P, PAIRS>(s));
#pragma unroll
        for (int i = 0; i < P / 4; ++i) {
            const float4 w = v[i];
            u[4 * i] = w.x;
            u[4 * i + 1] = w.y;
            u[4 * i + 2] = w.z;
            u[4 * i + 3] = w.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < P; ++i) u[i] = buf[slot_at<R, P, PAIRS>(s + i)];
    }
}

// Store the points of a lane's run that are still valid: warp points
// [edge, 32 P - edge).  Vector runs: edge is a multiple of P, so whole lanes.
template <typename R, int P, bool PAIRS>
__device__ __forceinline__ void store_run(R* buf, int s, const typename Run<R, P, PAIRS>::V (&u)[Run<R, P, PAIRS>::Q],
                                          int lane, int edge)
{
    if constexpr (kVector<R, P>) {
        if (lane * P >= edge && lane * P < 32 * P - edge) {
            R* at = buf + slot_at<R, P, PAIRS>(s);
#pragma unroll
            for (int i = 0; i < P / 4; ++i) {
                if constexpr (PAIRS)
                    reinterpret_cast<ulonglong2*>(at)[i] = make_ulonglong2(u[2 * i].b, u[2 * i + 1].b);
                else
                    reinterpret_cast<float4*>(at)[i] = make_float4(u[4 * i], u[4 * i + 1], u[4 * i + 2], u[4 * i + 3]);
            }
        }
    } else {
        const unsigned span = (unsigned)(32 * P - 2 * edge);
        const int at = lane * P - edge;
#pragma unroll
        for (int i = 0; i < P; ++i)
            if ((unsigned)(at + i) < span) buf[slot_at<R, P, PAIRS>(s + i)] = u[i];
    }
}

// Values of the rad elements before (lo) and after (hi) this lane's run.
template <int RAD, int Q, typename V>
__device__ __forceinline__ void run_edges(const V (&u)[Q], V (&lo)[RAD], V (&hi)[RAD])
{
    if constexpr (std::is_same<V, Pair>::value) {
#pragma unroll
        for (int k = 0; k < RAD; ++k) {
            const float2 last = split(u[Q - RAD + k]), first = split(u[k]);
            lo[k] = make_pair2(__shfl_up_sync(0xffffffffu, last.y, 1), last.x);
            hi[k] = make_pair2(first.y, __shfl_down_sync(0xffffffffu, first.x, 1));
        }
    } else if constexpr (Q >= RAD) {
#pragma unroll
        for (int k = 0; k < RAD; ++k) {
            lo[k] = __shfl_up_sync(0xffffffffu, u[Q - RAD + k], 1);
            hi[k] = __shfl_down_sync(0xffffffffu, u[k], 1);
        }
    } else {   // one point per lane, rad 2
        lo[0] = __shfl_up_sync(0xffffffffu, u[0], 2);
        lo[1] = __shfl_up_sync(0xffffffffu, u[0], 1);
        hi[0] = __shfl_down_sync(0xffffffffu, u[0], 1);
        hi[1] = __shfl_down_sync(0xffffffffu, u[0], 2);
    }
}

// One level of a lane's run: out = level after src (KS stage 1 with base
// values from out).
template <int EQ, int STAGE, int Q, typename V>
__device__ __forceinline__ void run_level(const V (&src)[Q], V (&out)[Q], const Coefs<V>& c, const Units<V>& ku)
{
    constexpr int RAD = Shape<EQ>::RAD;
    V lo[RAD], hi[RAD];
    run_edges<RAD, Q>(src, lo, hi);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        auto at = [&](int d) -> V {
            const int q = i + d;
            return q < 0 ? lo[RAD + q] : (q >= Q ? hi[q - Q] : src[q]);
        };
        if constexpr (EQ == HEAT)
            out[i] = heat_point(at(-1), at(0), at(1), c.fo, ku);
        else
            out[i] = ks_point(at(-2), at(-1), at(0), at(1), at(2), STAGE == 0 ? src[i] : out[i], c.a1[STAGE],
                              c.a4[STAGE], c.beta[STAGE], c.gam[STAGE], ku);
    }
}

// `levels` levels of a lane's run (KS: an even number, whole timesteps).
template <int EQ, int Q, typename V>
__device__ __forceinline__ void run_levels(V (&u)[Q], int levels, const Coefs<V>& c, const Units<V>& ku)
{
    V v[Q];
#pragma unroll 1
    for (int j = levels; j >= 2; j -= 2) {
        run_level<EQ, 0, Q>(u, v, c, ku);
        run_level<EQ, 1, Q>(v, u, c, ku);
    }
    if (EQ == HEAT && (levels & 1)) {
        run_level<EQ, 0, Q>(u, v, c, ku);
#pragma unroll
        for (int i = 0; i < Q; ++i) u[i] = v[i];
    }
}

// The constants of a kernel's runs of V from a launch's.
template <typename V, int EQ, typename R>
__device__ __forceinline__ Coefs<V> run_coefs(const Coefs<R>& c)
{
    if constexpr (std::is_same<V, Pair>::value) {
        Coefs<Pair> o{};
        if constexpr (EQ == HEAT) o.fo = make_pair2(c.fo, c.fo);
#pragma unroll
        for (int s = 0; s < 2 && EQ == KS; ++s) {
            o.a1[s] = make_pair2(c.a1[s], c.a1[s]);
            o.a4[s] = make_pair2(c.a4[s], c.a4[s]);
            o.beta[s] = make_pair2(c.beta[s], c.beta[s]);
            o.gam[s] = make_pair2(c.gam[s], c.gam[s]);
        }
        return o;
    } else {
        return lane_coefs<R, EQ>(c);
    }
}
template <typename V, int EQ>
__device__ __forceinline__ Units<V> run_units()
{
    if constexpr (std::is_same<V, Pair>::value) return {make_pair2(-2.0f, -2.0f)};
    else return make_units<V, EQ>();
}

// The whole advance of tile k of g.K: points [k N / K, (k + 1) N / K) from row A to
// row B.  False when a wait gave up (all threads together).
// BATCH: g.K may be 1, whose halos are its own points.
template <typename R, int EQ, int P, bool PAIRS, bool BATCH>
__device__ __forceinline__ bool resident_tile(const R* A, R* B, const ResidentGeom& g, int k, unsigned char* smem_raw,
                                              const Coefs<R>& launch_coefs)
{
    constexpr int RAD = Shape<EQ>::RAD, Q = Run<R, P, PAIRS>::Q;
    using V = typename Run<R, P, PAIRS>::V;
    const Coefs<V> c = run_coefs<V, EQ>(launch_coefs);
    const Units<V> ku = run_units<V, EQ>();
    R* cur = reinterpret_cast<R*>(smem_raw);
    R* nxt = cur + g.buf_elems;
    int* hoff = reinterpret_cast<int*>(nxt + g.buf_elems);   // published word of each halo point
    const int T = blockDim.x, tid = threadIdx.x, lane = tid & 31;
    const int K = g.K, h = g.h;
    const int64_t N = g.N;
    const int64_t b0 = k * N / K;
    const int own = (int)((k + 1) * N / K - b0);
    const int edge = RAD * g.L;
    // the lane's run starts at this tile slot; slot s is point b0 - h + s
    const int w0 = (tid >> 5) * (32 * P - 2 * edge), s0 = w0 + lane * P;
    // a batch's tiles vary in length: warps whose valid points lie past the tile's rest
    const bool active = !BATCH || w0 + edge < own + 2 * h;
    const int cap = g.cap, pub = g.pub;   // published points per block: all, or pub at each end
    const bool self = BATCH && K == 1;
    for (int s = tid; s < g.slots; s += T)
        cur[slot_at<R, P, PAIRS>(s)] = s < own + 2 * h ? A[fold(b0 - h + s, N, g.bc)] : R(0);
    if (g.exchanges > 0) {
        for (int e = tid; e < 2 * h; e += T) {
            const int p = (int)fold(b0 - h + (e < h ? e : own + e), N, g.bc);
            hoff[e] = self ? slot_at<R, P, PAIRS>(h + p) : word_of(p, (int)N, K, pub, cap);
        }
    }
    __syncthreads();
    V u[Q];
    for (int64_t x = 0;; ++x) {
        int left = x < g.exchanges ? g.E : g.last;   // levels until the next exchange, or the end
        while (left > 0) {
            const int n = min(left, g.L);
            if (active) {
                load_run<R, P, PAIRS>(cur, s0, u);
                run_levels<EQ, Q>(u, n, c, ku);
                store_run<R, P, PAIRS>(nxt, s0, u, lane, edge);
            }
            __syncthreads();
            R* t = cur;
            cur = nxt;
            nxt = t;
            left -= n;
        }
        if (x >= g.exchanges) break;
        if (self) {
            for (int e = tid; e < 2 * h; e += T) cur[slot_at<R, P, PAIRS>(e < h ? e : own + e)] = cur[hoff[e]];
            __syncthreads();
            continue;
        }
        const uint32_t seq = g.sync.seq + (uint32_t)x;
        uint64_t* words = g.sync.words + (x & 1) * g.parity_words;
        const int words_here = min(own, 2 * pub);
        for (int i = tid; i < words_here; i += T) {
            const int o = i < pub || own <= 2 * pub ? i : own - 2 * pub + i;
            Word<R>::put(words + (int64_t)(k * cap + i) * Word<R>::N64, cur[slot_at<R, P, PAIRS>(h + o)], seq);
        }
        int fail = 0;
        for (int e = tid; e < 2 * h; e += T) {
            R v;
            if (!wait_word<R>(words + (int64_t)hoff[e] * Word<R>::N64, seq + g.sync.wait_offset, g.sync, v)) {
                fail = 1;
                break;
            }
            cur[slot_at<R, P, PAIRS>(e < h ? e : own + e)] = v;
        }
        if (__syncthreads_or(fail)) return false;
    }
    for (int o = tid; o < own; o += T) B[b0 + o] = cur[slot_at<R, P, PAIRS>(h + o)];
    return true;
}

// Tile slots of a block.
inline int slot_count(int P, int warps, int rad, int L) { return warps * (32 * P - 2 * rad * L) + 2 * rad * L; }

// Elements of one shared-memory buffer (slot_at of the last slot, rounded up
// to whole 16-byte vectors).
inline int buffer_elems(int esize, int P, int slots)
{
    int e = slots;
    if (esize == 4 && P % 4 == 0) {   // whole runs, padded
        const int runs = (slots + P - 1) / P;
        e = runs * (P + ((P / 4) % 2 ? 0 : 4));
    }
    if (esize == 8 && P % 2 == 0) e += (slots - 1) >> 4;
    return (e + 3) / 4 * 4;
}

inline size_t resident_smem(int esize, int P, int slots, int h)
{
    return 2 * (size_t)buffer_elems(esize, P, slots) * esize + sizeof(int) * 2 * (size_t)h;
}

}  // namespace swp
