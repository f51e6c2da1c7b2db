// Resident form of a single heat / KS advance: one launch, the state in
// registers and shared memory from the first step to the last.
//
// The paper's nodes alternate an inverted and an upright triangle, so a
// half-cycle of H levels takes 2H - 1 dependent levels; that is the shape that
// needs no point twice, and it costs a grid that does not fill the GPU almost
// two level latencies per level.  Here each block owns a contiguous part of
// the grid and advances a tile of it with halos: a level leaves the outermost
// rad points of the tile stale, and after h / rad levels the halos are
// fetched again.  Every level of a tile is one level of progress; the price is
// the halo points' work, which the geometry keeps to a few per cent where the
// arithmetic counts and which is free where the chip would idle.
//
// Three scales:
//  - a thread holds P consecutive points in registers; a level reads its rad
//    neighbours on each side from the adjacent lanes by shuffle, and nothing
//    is predicated (stale edge values are computed and ignored);
//  - a warp advances L levels alone on 32 P points, of which 32 P - 2 rad L
//    are then valid; they go through shared memory (double buffered, one
//    barrier) and each warp reloads its points with fresh neighbours;
//  - after M such rounds the block publishes its owned points that lie within
//    h + 1 (h = rad L M) of its ends and fetches its halos from the neighbouring
//    blocks.  Each published word carries the exchange's sequence number next
//    to its data (8 bytes, stored and loaded as one access), so a reader polls
//    the data itself: no flag, no fence, one trip through L2 each way.
// The blocks wait on one another, so the launch is cooperative (all blocks
// resident); every wait is bounded.  An FP32 grid that the chip does not hold
// runs the same tiles without waits: a launch per L M levels, from one row to the
// other.
//
// Both ends of the domain are index folds: periodic points wrap, and an
// insulated end (u_{-k} = u_k, Appendix A) is the even extension, whose mirrored
// points evolve with the same bits because the stencil's only sum of the two
// neighbours commutes.
//
// Each point update is scheme.cuh's on the same operands as in the classic
// scheme, so the bits are the same.
//
// What bounds it.  FP64: its pipe, a warp-wide FMA every 64 clocks; with one warp
// per SM sub-partition the chain of a level (KS N = 1024: 569 of 667 clocks per level)
// and the exchange between blocks (1340 to 1530 clocks each, clock counters of all
// blocks).  FP32 KS: the FMA pipe, 80 % of it in pairs (an f32x2 takes it two clocks;
// "math pipe throttle" is the top stall).  FP32 heat at 2^17: one warp per
// sub-partition, 59 clocks a level of which 41 % issue, and exchanges of 2940 clocks
// (192 halo points a side) every 192 levels.  86 % of the FP32 instructions are the
// point updates' own.  Measured per advance (write, advance, read) against the forms
// that were the default before (cluster, Register and Shared graphs, per-phase FP32):
//   heat FP64 N = 1024, 4096 steps      1193 -> 615 us
//   heat FP64 reflective 50001, 2000    1556 -> 806 us
//   KS FP64 10007, 2000 steps           3217 -> 1537 us
//   heat FP32 2^17, 4000 steps          1078 -> 178 us
//   KS FP32 2000003, 1000 steps         3699 -> 1024 us
// and beyond the chip, a launch per exchange, in G point-updates/s: heat FP32 2^22
// 1585 -> 6950, 2^24 1640 -> 6490, 2^26 1430 -> 3650; KS FP32 2^22 583 -> 1619, 2^24
// 589 -> 1456, 2^26 575 -> 1257.
#include <algorithm>

#include "resident.h"
#include "resident_tile.cuh"

namespace swp {

namespace {

template <typename R, int EQ, int P>
__global__ void __launch_bounds__(512, sizeof(R) == 4 ? 1 : 0)
    swept_resident_kernel(const R* A, R* B, ResidentGeom g, Coefs<R> c)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    resident_tile<R, EQ, P, EQ == KS && kVector<R, P>, false>(A, B, g, (int)blockIdx.x, smem_raw, c);
}

// Kernel of (precision, equation, points per thread), or NULL.
template <typename R, int EQ>
const void* kernel_of(int P)
{
#define SWP_RESIDENT_P(p) \
    case p: return (const void*)swept_resident_kernel<R, EQ, p>;
    if constexpr (sizeof(R) == 8) {
        switch (P) {
            SWP_RESIDENT_P(1)
            SWP_RESIDENT_P(2)
            SWP_RESIDENT_P(3)
            SWP_RESIDENT_P(4)
            SWP_RESIDENT_P(5)
            SWP_RESIDENT_P(6)
            SWP_RESIDENT_P(7)
            SWP_RESIDENT_P(8)
            SWP_RESIDENT_P(9)
            SWP_RESIDENT_P(10)
            SWP_RESIDENT_P(11)
            SWP_RESIDENT_P(12)
            SWP_RESIDENT_P(13)
            SWP_RESIDENT_P(14)
            SWP_RESIDENT_P(15)
            SWP_RESIDENT_P(16)
        default: return nullptr;
        }
    } else {
        switch (P) {
            SWP_RESIDENT_P(1)
            SWP_RESIDENT_P(2)
            SWP_RESIDENT_P(4)
            SWP_RESIDENT_P(8)
            SWP_RESIDENT_P(12)
            SWP_RESIDENT_P(16)
            SWP_RESIDENT_P(20)
            SWP_RESIDENT_P(24)
            SWP_RESIDENT_P(28)
            SWP_RESIDENT_P(32)
        default: return nullptr;
        }
    }
#undef SWP_RESIDENT_P
}

template <typename R>
const void* kernel_of(int eq, int P)
{
    return eq == HEAT ? kernel_of<R, HEAT>(P) : kernel_of<R, KS>(P);
}

constexpr int kPoints64[] = {1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16};
constexpr int kPoints32[] = {1, 2, 4, 8, 12, 16, 20, 24, 28, 32};

}  // namespace

namespace {

// Estimated clocks per level of a block of `warps` warps with P points per thread
// that owns its tile's points, from a fit to 2294 measured shapes (N from 2^10 to
// 2^21; a clock is 1/2.07 us of event time, the SMs ran at 2.02 to 2.05 GHz): the
// arithmetic of a level, the round through shared memory every L levels (170 to
// 1000) and the exchange between blocks every L M levels (1450 and the polls of its
// halo).  FP64 is its pipe's time (66 such clocks, 64 of the SM's, per warp-wide
// FMA) and a latency that a second warp per SM sub-partition hides; the factors by
// warps are the fit's too: one warp per sub-partition leaves 6 % of the pipe's slots
// empty, three or four fill 2 % that two leave.  FP32 is issue, at 1.1 (heat) slots per
// operation and for KS 1.36, or 1.5 where one warp per sub-partition has no other to
// issue beside it, above the latency of a level's shuffles and chain.
double level_clocks(int eq, int esize, int warps, int P, int L, int M, int h)
{
    const double ops = eq == HEAT ? 3.0 : 7.0, w = warps / 4;
    double level;
    if (esize == 8)
        level = w * P * ops * 66.0 * (warps == 4 ? 1.06 : (warps == 8 ? 1.0 : 0.98)) + (warps == 4 ? 50.0 : 15.0);
    else if (eq == HEAT)
        level = std::max(57.0, 1.1 * w * P * ops + 35.0);
    else
        level = std::max(50.0 + 10.0 * std::min(P, 4), (warps == 4 ? 1.5 : 1.36) * w * P * ops + 25.0);
    const double round = esize == 8 ? 170.0 + 12.0 * w * P : 130.0 + 6.0 * w * P;
    const double exchange = M > 0 ? (1450.0 + 2.5 * h) / ((double)L * M) : 0.0;
    return level + round / L + exchange;
}

// The best shape for blocks that own `own` points each.  Returns its clocks per
// level, 0 when no tile holds them.
double best_shape(int eq, int esize, int own, ResidentShape* out)
{
    const int rad = eq == HEAT ? 1 : 2;
    const int* pts = esize == 8 ? kPoints64 : kPoints32;
    const int npts = esize == 8 ? (int)(sizeof(kPoints64) / sizeof(int)) : (int)(sizeof(kPoints32) / sizeof(int));
    double best = 0.0;
    for (int warps = 4; warps <= 16; warps += 4)
        for (int ip = 0; ip < npts; ++ip) {
            const int P = pts[ip];
            const bool vector = esize == 4 && P % 4 == 0;
            for (int step = 1; step <= 8; ++step) {
                // vector runs leave whole lanes stale
                const int L = vector ? step * P / rad : 2 * step;
                if (L & 1 || 2 * rad * L >= 32 * P - rad) continue;
                const int slots = slot_count(P, warps, rad, L);
                const int M = std::min(64, (slots - own) / (2 * rad * L));
                if (M < 1) continue;
                const int h = rad * L * M;
                if (resident_smem(esize, P, slots, h) > kResidentSmem) continue;
                const double cost = level_clocks(eq, esize, warps, P, L, M, h);
                if (best == 0.0 || cost < best) {
                    best = cost;
                    out->P = P;
                    out->warps = warps;
                    out->L = L;
                    out->M = M;
                }
            }
        }
    return best;
}

}  // namespace

bool resident_plan(int eq, int esize, int64_t N, int sms, ResidentShape* out)
{
    *out = ResidentShape();
    if (eq == EULER || N < 64 || sms < 1) return false;
    const double ops = eq == HEAT ? 3.0 : 7.0;
    // blocks of at least 16 points: with fewer the halos come from many blocks
    const int K = (int)std::min<int64_t>(sms, std::max<int64_t>(1, N / 16));
    if ((N + 1) * (K + 1) < (int64_t)1 << 31) {
        const int own = (int)((N + K - 1) / K);
        const double clocks = best_shape(eq, esize, own, out);
        // FP64 from 2^17 points: the swept dataflow launch spends about 700
        // clocks per level above its points' pipe time (KS 2^17: 3760 against
        // 3965 here, 2^20: 25530 against 25930; heat 2^17: 1995 against 1690)
        if (clocks > 0.0 &&
            (esize == 4 || N < ((int64_t)1 << 17) || clocks <= own / 128.0 * ops * 66.0 + 700.0)) {
            out->K = K;
            return true;
        }
    }
    if (esize == 8) return false;
    // FP32 beyond the chip: tiles of the same kind, a launch per exchange,
    // whole waves of one block per SM.  (FP64 there is at its pipe's rate in
    // the dataflow launch.)
    const int64_t waves = (N + (int64_t)sms * 14000 - 1) / ((int64_t)sms * 14000);
    const int64_t blocks = waves * sms;
    if (blocks >= (int64_t)1 << 30) return false;
    if (best_shape(eq, esize, (int)((N + blocks - 1) / blocks), out) == 0.0) return false;
    out->K = (int)blocks;
    out->waves = (int)std::min<int64_t>(waves, 1 << 20);
    return true;
}

size_t resident_words(int eq, int esize, int64_t N, const ResidentShape& s)
{
    const int rad = eq == HEAT ? 1 : 2;
    const int own = (int)((N + s.K - 1) / s.K);
    return (size_t)s.K * std::min(own, 2 * (rad * s.L * s.M + 1)) * (esize == 8 ? 2 : 1);
}

int64_t resident_exchanges(const ResidentShape& s, int64_t levels)
{
    const int64_t E = (int64_t)s.L * s.M;
    return (levels + E - 1) / E - 1;
}

template <typename R>
cudaError_t launch_swept_resident(int eq, int bc, const R* A, R* B, int64_t N, int64_t levels, const ResidentShape& s,
                                  const ResidentSync& y, const Coefs<R>& c, cudaStream_t st)
{
    const int rad = eq == HEAT ? 1 : 2;
    ResidentGeom g;
    g.N = N;
    g.K = s.K;
    g.L = s.L;
    g.E = s.L * s.M;
    g.h = rad * g.E;
    g.slots = slot_count(s.P, s.warps, rad, s.L);
    const int own = (int)((N + s.K - 1) / s.K);
    // the mirror image of a halo of h points reaches point h of the end block
    g.pub = g.h + 1;
    g.cap = std::min(own, 2 * g.pub);
    g.exchanges = resident_exchanges(s, levels);
    g.last = (int)(levels - g.exchanges * g.E);
    g.bc = bc;
    g.sync = y;
    g.parity_words = y.words ? (int64_t)resident_words(eq, (int)sizeof(R), N, s) : 0;
    const size_t smem = resident_smem((int)sizeof(R), s.P, g.slots, g.h);
    g.buf_elems = buffer_elems((int)sizeof(R), s.P, g.slots);
    const void* fn = kernel_of<R>(eq, s.P);
    if (!fn) return cudaErrorInvalidDeviceFunction;
    const cudaError_t e = allow_resident_smem(fn);
    if (e != cudaSuccess) return e;
    void* args[] = {(void*)&A, (void*)&B, (void*)&g, (void*)&c};
    const dim3 grid((unsigned)s.K), block((unsigned)(32 * s.warps));
    return s.waves > 1 ? cudaLaunchKernel(fn, grid, block, args, smem, st)
                       : cudaLaunchCooperativeKernel(fn, grid, block, args, smem, st);
}

template cudaError_t launch_swept_resident<double>(int, int, const double*, double*, int64_t, int64_t,
                                                   const ResidentShape&, const ResidentSync&, const Coefs<double>&,
                                                   cudaStream_t);
template cudaError_t launch_swept_resident<float>(int, int, const float*, float*, int64_t, int64_t,
                                                  const ResidentShape&, const ResidentSync&, const Coefs<float>&,
                                                  cudaStream_t);

}  // namespace swp
