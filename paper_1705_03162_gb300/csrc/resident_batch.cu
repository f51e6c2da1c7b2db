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
// What bounds it: the point updates' own pipe, FP64 (86 % of its peak with 4-warp
// blocks, whose barriers lost the rest) or FP32 issue, plus the halos and the
// tiles' unused slots.  256 heat and KS problems of 2^10..2^16 points, dataflow
// launch / this one: FP64, 400 to 1600 steps, 61.3 / 58.1 ms; FP32, 2000 to 10000
// steps, 43.0 / 11.1 ms.
#include <algorithm>

#include "resident.h"
#include "resident_tile.cuh"

namespace swp {

namespace {

// Points per thread, stale points at each end of a warp's round (edge = rad L),
// rounds per exchange, and blocks, by precision: the fastest of a sweep on 256
// heat and KS problems of 2^10..2^16 points.  Smaller blocks lose less at their
// barriers when they share an SM (FP64, P = 12: 58.1 ms with 2 warps, 61.2 with 4,
// 59.0 with 1, whose tiles have more halo); FP32 rounds stale whole lanes of
// 16-point vectors (P = 16: 11.1 ms; 8: 12.4, 12: 11.6, 20: 11.2, 28: 11.4; KS runs
// in pairs, which gain in the single launch, 12.2).
template <typename R> struct Tile;
template <> struct Tile<float> {
    static constexpr int P = 16, EDGE = 16, M = 3, THREADS = 128, BLOCKS_PER_SM = 4;
};
template <> struct Tile<double> {
    static constexpr int P = 12, EDGE = 4, M = 2, THREADS = 64, BLOCKS_PER_SM = 8;
};

template <typename R>
__global__ void __launch_bounds__(Tile<R>::THREADS, Tile<R>::BLOCKS_PER_SM)
    swept_resident_batch_kernel(const ResidentInst<R>* insts, ResidentBatchWork w)
{
    constexpr int P = Tile<R>::P;
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
        g.sync.wait_offset = 0;
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

template <typename R>
constexpr int kSlots = Tile<R>::THREADS / 32 * (32 * Tile<R>::P - 2 * Tile<R>::EDGE) + 2 * Tile<R>::EDGE;

// Halo points per side of the widest exchange, and the most points a tile owns.
template <typename R>
constexpr int kHalo = Tile<R>::EDGE * Tile<R>::M;
template <typename R>
constexpr int kOwn = kSlots<R> - 2 * kHalo<R>;

template <typename R>
size_t batch_smem()
{
    return resident_smem((int)sizeof(R), Tile<R>::P, kSlots<R>, kHalo<R>);
}

}  // namespace

int resident_batch_own(int esize) { return esize == 4 ? kOwn<float> : kOwn<double>; }

template <typename R>
ResidentGeom resident_batch_geom(int eq, int bc, int64_t N, int64_t levels)
{
    const int rad = eq == HEAT ? 1 : 2;
    ResidentGeom g{};
    g.N = N;
    g.K = (int)((N + kOwn<R> - 1) / kOwn<R>);
    g.L = Tile<R>::EDGE / rad;
    g.E = g.L * Tile<R>::M;
    g.h = kHalo<R>;
    g.slots = kSlots<R>;
    g.buf_elems = buffer_elems((int)sizeof(R), Tile<R>::P, kSlots<R>);
    g.pub = g.h + 1;
    g.cap = (int)std::min<int64_t>((N + g.K - 1) / g.K, 2 * g.pub);
    g.bc = bc;
    g.exchanges = (levels + g.E - 1) / g.E - 1;
    g.last = (int)(levels - g.exchanges * g.E);
    g.parity_words = (int64_t)g.K * g.cap * (sizeof(R) == 8 ? 2 : 1);
    return g;
}

template <typename R>
int resident_batch_blocks(int sms)
{
    const size_t smem = batch_smem<R>();
    if (smem > 48 * 1024 && cudaFuncSetAttribute((const void*)swept_resident_batch_kernel<R>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return 0;
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, swept_resident_batch_kernel<R>, Tile<R>::THREADS,
                                                      smem) !=
        cudaSuccess)
        return 0;
    return nb * sms;
}

template <typename R>
cudaError_t launch_swept_resident_batch(const ResidentInst<R>* insts, const ResidentBatchWork& w, int blocks,
                                        cudaStream_t s)
{
    void* args[] = {(void*)&insts, (void*)&w};
    return cudaLaunchCooperativeKernel((const void*)swept_resident_batch_kernel<R>, dim3((unsigned)blocks),
                                       dim3(Tile<R>::THREADS), args, batch_smem<R>(), s);
}

template ResidentGeom resident_batch_geom<double>(int, int, int64_t, int64_t);
template ResidentGeom resident_batch_geom<float>(int, int, int64_t, int64_t);
template int resident_batch_blocks<double>(int);
template int resident_batch_blocks<float>(int);
template cudaError_t launch_swept_resident_batch<double>(const ResidentInst<double>*, const ResidentBatchWork&, int,
                                                         cudaStream_t);
template cudaError_t launch_swept_resident_batch<float>(const ResidentInst<float>*, const ResidentBatchWork&, int,
                                                        cudaStream_t);

}  // namespace swp
