// One tile of a resident heat / KS advance: registers, warp rounds through shared
// memory, halo exchange between blocks (resident.cu has the idea; used by it and
// by the batched form, resident_batch.cu).
#pragma once

#include "resident.cuh"

namespace swp {

// FP32 runs of a multiple of 4 points move as 16-byte vectors.
template <typename R, int P>
constexpr bool kVector = sizeof(R) == 4 && P % 4 == 0;

// Shared-memory index of tile slot s.  Lanes read runs of P slots, all lanes
// at once, so the stride of the runs is padded to spread over the banks: vector
// runs (FP32, P a multiple of 4) to an odd number of 16-byte vectors, even FP64
// strides by a value after every 16.
template <typename R, int P>
__host__ __device__ __forceinline__ constexpr int slot_at(int s)
{
    if (kVector<R, P>) return (P / 4) % 2 ? s : s + s / P * 4;
    if (sizeof(R) == 8 && P % 2 == 0) return s + (s >> 4);
    return s;
}

template <typename R, int P>
__device__ __forceinline__ void load_run(const R* buf, int s, R (&u)[P])
{
    if constexpr (kVector<R, P>) {
#pragma unroll
        for (int i = 0; i < P; i += 4) {
            const float4 v = *reinterpret_cast<const float4*>(buf + slot_at<R, P>(s) + i);   // s a multiple of P
            u[i] = v.x;
            u[i + 1] = v.y;
            u[i + 2] = v.z;
            u[i + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < P; ++i) u[i] = buf[slot_at<R, P>(s + i)];
    }
}

// Store the points of a lane's run that are still valid: warp points
// [edge, 32 P - edge).  Vector runs: edge is a multiple of P, so whole lanes.
template <typename R, int P>
__device__ __forceinline__ void store_run(R* buf, int s, const R (&u)[P], int lane, int edge)
{
    if constexpr (kVector<R, P>) {
        if (lane * P >= edge && lane * P < 32 * P - edge) {
#pragma unroll
            for (int i = 0; i < P; i += 4)
                *reinterpret_cast<float4*>(buf + slot_at<R, P>(s) + i) = make_float4(u[i], u[i + 1], u[i + 2], u[i + 3]);
        }
    } else {
        const unsigned span = (unsigned)(32 * P - 2 * edge);
        const int at = lane * P - edge;
#pragma unroll
        for (int i = 0; i < P; ++i)
            if ((unsigned)(at + i) < span) buf[slot_at<R, P>(s + i)] = u[i];
    }
}

// Values of the rad slots before (lo) and after (hi) this lane's run.
template <typename R, int RAD, int P>
__device__ __forceinline__ void run_edges(const R (&u)[P], R (&lo)[RAD], R (&hi)[RAD])
{
    if constexpr (P >= RAD) {
#pragma unroll
        for (int k = 0; k < RAD; ++k) {
            lo[k] = __shfl_up_sync(0xffffffffu, u[P - RAD + k], 1);
            hi[k] = __shfl_down_sync(0xffffffffu, u[k], 1);
        }
    } else {   // P == 1, RAD == 2
        lo[0] = __shfl_up_sync(0xffffffffu, u[0], 2);
        lo[1] = __shfl_up_sync(0xffffffffu, u[0], 1);
        hi[0] = __shfl_down_sync(0xffffffffu, u[0], 1);
        hi[1] = __shfl_down_sync(0xffffffffu, u[0], 2);
    }
}

// One level of a lane's run: out = level after src (KS stage 1 with base
// values from out).
template <typename R, int EQ, int STAGE, int P>
__device__ __forceinline__ void run_level(const R (&src)[P], R (&out)[P], const Coefs<R>& c,
                                          const Units<R>& ku)
{
    constexpr int RAD = Shape<EQ>::RAD;
    R lo[RAD], hi[RAD];
    run_edges<R, RAD, P>(src, lo, hi);
#pragma unroll
    for (int i = 0; i < P; ++i) {
        auto at = [&](int d) -> R {
            const int q = i + d;
            return q < 0 ? lo[RAD + q] : (q >= P ? hi[q - P] : src[q]);
        };
        if constexpr (EQ == HEAT)
            out[i] = heat_point(at(-1), at(0), at(1), c.fo, ku);
        else
            out[i] = ks_point(at(-2), at(-1), at(0), at(1), at(2), STAGE == 0 ? src[i] : out[i], c.a1[STAGE],
                              c.a4[STAGE], c.beta[STAGE], c.gam[STAGE], ku);
    }
}

// `levels` levels of a lane's run (KS: an even number, whole timesteps).
template <typename R, int EQ, int P>
__device__ __forceinline__ void run_levels(R (&u)[P], int levels, const Coefs<R>& c, const Units<R>& ku)
{
    R v[P];
#pragma unroll 1
    for (int j = levels; j >= 2; j -= 2) {
        run_level<R, EQ, 0, P>(u, v, c, ku);
        run_level<R, EQ, 1, P>(v, u, c, ku);
    }
    if (EQ == HEAT && (levels & 1)) {
        run_level<R, EQ, 0, P>(u, v, c, ku);
#pragma unroll
        for (int i = 0; i < P; ++i) u[i] = v[i];
    }
}

// The whole advance of tile k of g.K: points [k N / K, (k + 1) N / K) from row A to
// row B.  False when a wait gave up (all threads together).
// SELF: g.K may be 1, whose halos are its own points.
template <typename R, int EQ, int P, bool SELF>
__device__ __forceinline__ bool resident_tile(const R* A, R* B, const ResidentGeom& g, int k, unsigned char* smem_raw,
                                              const Coefs<R>& c, const Units<R>& ku)
{
    constexpr int RAD = Shape<EQ>::RAD;
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
    const bool active = w0 + edge < own + 2 * h;   // the warp's valid points reach the tile's
    const int cap = g.cap, pub = g.pub;            // published points per block: all, or pub at each end
    const bool self = SELF && K == 1;
    for (int s = tid; s < g.slots; s += T)
        cur[slot_at<R, P>(s)] = s < own + 2 * h ? A[fold(b0 - h + s, N, g.bc)] : R(0);
    if (g.exchanges > 0) {
        for (int e = tid; e < 2 * h; e += T) {
            const int p = (int)fold(b0 - h + (e < h ? e : own + e), N, g.bc);
            hoff[e] = self ? slot_at<R, P>(h + p) : word_of(p, (int)N, K, pub, cap);
        }
    }
    __syncthreads();
    R u[P];
    for (int64_t x = 0;; ++x) {
        int left = x < g.exchanges ? g.E : g.last;   // levels until the next exchange, or the end
        while (left > 0) {
            const int n = min(left, g.L);
            if (active) {
                load_run<R, P>(cur, s0, u);
                run_levels<R, EQ, P>(u, n, c, ku);
                store_run<R, P>(nxt, s0, u, lane, edge);
            }
            __syncthreads();
            R* t = cur;
            cur = nxt;
            nxt = t;
            left -= n;
        }
        if (x >= g.exchanges) break;
        if (self) {
            for (int e = tid; e < 2 * h; e += T) cur[slot_at<R, P>(e < h ? e : own + e)] = cur[hoff[e]];
            __syncthreads();
            continue;
        }
        const uint32_t seq = g.sync.seq + (uint32_t)x;
        uint64_t* words = g.sync.words + (x & 1) * g.parity_words;
        const int words_here = min(own, 2 * pub);
        for (int i = tid; i < words_here; i += T) {
            const int o = i < pub || own <= 2 * pub ? i : own - 2 * pub + i;
            Word<R>::put(words + (int64_t)(k * cap + i) * Word<R>::N64, cur[slot_at<R, P>(h + o)], seq);
        }
        int fail = 0;
        for (int e = tid; e < 2 * h; e += T) {
            R v;
            if (!wait_word<R>(words + (int64_t)hoff[e] * Word<R>::N64, seq + g.sync.wait_offset, g.sync, v)) {
                fail = 1;
                break;
            }
            cur[slot_at<R, P>(e < h ? e : own + e)] = v;
        }
        if (__syncthreads_or(fail)) return false;
    }
    for (int o = tid; o < own; o += T) B[b0 + o] = cur[slot_at<R, P>(h + o)];
    return true;
}

// Tile slots of a block.
inline int slot_count(int P, int warps, int rad, int L) { return warps * (32 * P - 2 * rad * L) + 2 * rad * L; }

// Elements of one shared-memory buffer (slot_at of the last slot, rounded up
// to whole 16-byte vectors).
inline int buffer_elems(int esize, int P, int slots)
{
    int e = slots;
    if (esize == 4 && P % 8 == 0) e += (slots - 1) / P * 4;
    if (esize == 8 && P % 2 == 0) e += (slots - 1) >> 4;
    return (e + 3) / 4 * 4;
}

inline size_t resident_smem(int esize, int P, int slots, int h)
{
    return 2 * (size_t)buffer_elems(esize, P, slots) * esize + sizeof(int) * 2 * (size_t)h;
}

}  // namespace swp
