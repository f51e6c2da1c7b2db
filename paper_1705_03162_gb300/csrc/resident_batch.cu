// Batched resident form: many heat and KS problems advanced in one cooperative
// launch, each tile on chip from its first level to its last.
//
// The dataflow batch (swept.cu) hands every node of every phase through global
// memory and a task table.  Here a block claims a tile of a problem and keeps it
// for the whole advance (resident_tile.cuh), exchanging halos with the problem's
// other tiles through published words.  Tiles are claimed in order, problem by
// problem, so a problem's tiles run together: the first problem in the list that
// has unfinished tiles has all of them claimed or next to be claimed, its
// predecessors need no later block to finish, and no problem has more tiles than
// the launch has blocks.  Longest advances come first, so the short ones fill
// the end.  Several blocks share an SM: while one waits for its halos or a
// barrier the others compute.
//
// What bounds it: FP32, instruction issue, plus the halos and the tiles' unused
// slots: 256 heat and KS problems of 2^10..2^16 points, 2000 to 10000 steps, dataflow
// launch 43.0 ms, this one 11.0.  FP64, for the batches that leave most of the chip
// idle (resident_batch_choose), the levels' chains and exchanges.
// A launch that the device refuses (too many blocks to hold at once) is the caller's
// sign to run the dataflow form.
#include <algorithm>
#include <vector>

#include "resident.h"
#include "resident_tile.cuh"

namespace swp {

namespace {

// Tiles: points per thread, stale points at each end of a warp's round (edge = rad
// L), rounds per exchange, threads, and blocks per SM.  FP64 blocks have two warps:
// smaller blocks lose less at their barriers when they share an SM.  FP32 rounds
// leave whole lanes of 8- or 16-point vectors stale.
//
// Long tiles do the least work beside their own points, short ones spread a small
// batch over more of the chip (resident_batch_choose).
template <typename R, int P_, int EDGE_, int M_, int THREADS_, int BLOCKS_PER_SM_> struct Tile {
    using Real = R;
    static constexpr int P = P_, EDGE = EDGE_, M = M_, THREADS = THREADS_, BLOCKS_PER_SM = BLOCKS_PER_SM_;
    static constexpr int SLOTS = THREADS / 32 * (32 * P - 2 * EDGE) + 2 * EDGE;
    static constexpr int HALO = EDGE * M;             // points per side of an exchange
    static constexpr int OWN = SLOTS - 2 * HALO;      // the most points a tile owns
};

template <typename T>
__global__ void __launch_bounds__(T::THREADS, T::BLOCKS_PER_SM)
    swept_resident_batch_kernel(const ResidentInst<typename T::Real>* insts, ResidentBatchWork w)
{
    using R = typename T::Real;
    constexpr int P = T::P;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int tile_s;
    for (;;) {
        if (threadIdx.x == 0) tile_s = atomicAdd(w.next_tile, 1);
        __syncthreads();
        const int t = tile_s;
        if (t >= w.ntiles) break;
        const int2 tk = w.tiles[t];
        const ResidentInst<R>& in = insts[tk.x];
        ResidentGeom g = in.g;
        g.sync.words = w.words + in.word_off;
        g.sync.seq = 1;
        g.sync.wait_offset = w.wait_offset;
        g.sync.wait_limit_ns = w.wait_limit_ns;
        g.sync.status = w.status;
        g.sync.claimed = w.next_tile;
        g.sync.last_tile = in.last_tile;
        bool ok;
        if (in.eq == HEAT) ok = resident_tile<R, HEAT, P, false, true>(in.A, in.B, g, tk.y, smem_raw, in.c);
        else ok = resident_tile<R, KS, P, false, true>(in.A, in.B, g, tk.y, smem_raw, in.c);
        if (!ok) break;
        __syncthreads();   // tile_s and the buffers are free again
    }
}

struct Variant {
    const void* kernel;
    int P, edge, M, threads, blocks_per_sm, slots, halo, own;
};
template <typename T>
Variant variant_of()
{
    return {(const void*)swept_resident_batch_kernel<T>, T::P, T::EDGE, T::M, T::THREADS, T::BLOCKS_PER_SM, T::SLOTS,
            T::HALO, T::OWN};
}

// The variants of a precision, longest tiles first.
const std::vector<Variant>& variants(int esize)
{
    static const std::vector<Variant> f32 = {variant_of<Tile<float, 16, 16, 3, 128, 4>>(),
                                             variant_of<Tile<float, 8, 16, 3, 128, 4>>()};
    static const std::vector<Variant> f64 = {variant_of<Tile<double, 4, 4, 4, 64, 8>>(),
                                             variant_of<Tile<double, 2, 4, 4, 64, 8>>()};
    return esize == 4 ? f32 : f64;
}

size_t smem_of(int esize, const Variant& v) { return resident_smem(esize, v.P, v.slots, v.halo); }

}  // namespace

// FP64, in ms, 300 to 1200 steps, P = 4 / 2 against the dataflow launch with its best
// node widths (points in all):
//   4 problems,    22 k     1.54 / 0.88   1.8
//   4 problems,    62 k     1.55 / 1.78   2.0
//   16 problems,   90 k     2.56 / 2.78   2.5
//   48 problems,  270 k      6.8 / 4.7    4.3
// and with the longest tiles that still even out (P = 12 for the larger ones):
//   48 problems,  1.2 M     17.7          15.4
//   256 problems, 3.9 M     47.0          44.3
//   4096 problems, 62.6 M   1290          1168
// So a batch whose P = 2 tiles the chip holds three to a sub-partition runs on chip,
// with the P that keeps a level of its busiest sub-partition shortest, and every other
// one as dataflow.  FP32 (P = 16 / 8, dataflow): 4 problems 0.20 / 0.15 / 1.1, 128
// problems of 2.0 M points 0.93 / 0.73 / 4.4, 256 of 4.0 M with 2000 to 10000 steps
// 11.0 / 12.6 / 43.
ResidentBatchFit resident_batch_choose(int esize, const std::vector<int64_t>& points, int sms, ResidentBatchShape* out)
{
    const auto& vs = variants(esize);
    std::vector<int64_t> tiles(vs.size(), 0);
    std::vector<bool> holds(vs.size(), true);   // no problem has more tiles than blocks
    for (const int64_t N : points)
        for (size_t i = 0; i < vs.size(); ++i) {
            const int64_t K = (N + vs[i].own - 1) / vs[i].own;
            tiles[i] += K;
            holds[i] = holds[i] && K <= (int64_t)vs[i].blocks_per_sm * sms;
        }
    auto waves = [&](size_t i) { return (double)tiles[i] / ((double)vs[i].blocks_per_sm * sms); };
    size_t pick = 0;
    if (esize == 4) {
        if (!holds[0]) return RESIDENT_TOO_LONG;
        pick = waves(0) < 2.5 && holds[1] ? 1 : 0;
    } else {
        if (waves(1) > 0.75) return RESIDENT_SLOWER;   // (below, every problem fits)
        auto level = [&](size_t i) {
            return vs[i].P * std::max(1.0, (double)tiles[i] * (vs[i].threads / 32) / (4.0 * sms));
        };
        pick = level(1) < level(0) ? 1 : 0;
    }
    out->variant = (int)pick;
    const Variant& v = vs[out->variant];
    const size_t smem = smem_of(esize, v);
    if (allow_resident_smem(v.kernel) != cudaSuccess) return RESIDENT_TOO_LONG;
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, v.kernel, v.threads, smem) != cudaSuccess ||
        nb < v.blocks_per_sm)
        return RESIDENT_TOO_LONG;
    out->blocks = v.blocks_per_sm * sms;
    return RESIDENT_FITS;
}

ResidentGeom resident_batch_geom(int eq, int esize, int bc, int64_t N, int64_t levels, const ResidentBatchShape& s)
{
    const Variant& v = variants(esize)[s.variant];
    ResidentGeom g{};
    g.N = N;
    g.K = (int)((N + v.own - 1) / v.own);
    g.L = v.edge / (eq == HEAT ? 1 : 2);
    g.E = g.L * v.M;
    g.h = v.halo;
    g.slots = v.slots;
    g.buf_elems = buffer_elems(esize, v.P, v.slots);
    g.pub = g.h + 1;
    g.cap = (int)std::min<int64_t>((N + g.K - 1) / g.K, 2 * g.pub);
    g.bc = bc;
    g.exchanges = (levels + g.E - 1) / g.E - 1;
    g.last = (int)(levels - g.exchanges * g.E);
    g.parity_words = (int64_t)g.K * g.cap * (esize == 8 ? 2 : 1);
    return g;
}

template <typename R>
cudaError_t launch_swept_resident_batch(const ResidentInst<R>* insts, const ResidentBatchWork& w,
                                        const ResidentBatchShape& shape, cudaStream_t s)
{
    const Variant& v = variants((int)sizeof(R))[shape.variant];
    void* args[] = {(void*)&insts, (void*)&w};
    return cudaLaunchCooperativeKernel(v.kernel, dim3((unsigned)std::min(shape.blocks, w.ntiles)),
                                       dim3((unsigned)v.threads), args, smem_of((int)sizeof(R), v), s);
}

template cudaError_t launch_swept_resident_batch<double>(const ResidentInst<double>*, const ResidentBatchWork&,
                                                         const ResidentBatchShape&, cudaStream_t);
template cudaError_t launch_swept_resident_batch<float>(const ResidentInst<float>*, const ResidentBatchWork&,
                                                        const ResidentBatchShape&, cudaStream_t);

}  // namespace swp
