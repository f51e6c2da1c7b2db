// The resident form of a single advance (resident.cu, Euler: resident_euler.cu):
// launch interface between the C-ABI layer (api.cu) and the kernels.  Internal
// header.
#pragma once

#include <cstdint>
#include <vector>

#include <cuda_runtime.h>

#include "scheme.cuh"

namespace swp {

// Shared memory the resident kernels are allowed: always the same amount, so that
// launches from several threads with tiles of different sizes cannot undo each
// other's setting.
constexpr size_t kResidentSmem = 226 * 1024;
inline cudaError_t allow_resident_smem(const void* kernel)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResidentSmem);
}

// One cooperative launch of K blocks, each keeping its part of the grid on chip.
struct ResidentShape {
    int K = 0;        // blocks (0: N has no resident shape)
    int waves = 1;    // > 1: more blocks than the chip holds; no exchanges, a launch per L M levels
    int P = 0;        // points per thread
    int warps = 0;    // warps per block
    int L = 0, M = 0; // levels per warp round, rounds per exchange between blocks
    bool split = false;   // Euler: the sides of an interface are tasks of their own
};
// What a launch synchronises through: two sets of published words (one per
// exchange parity), each word carrying the exchange's sequence number, which
// no earlier launch on these words has used.
struct ResidentSync {
    uint64_t* words;
    uint32_t seq;          // of the launch's first exchange
    uint32_t wait_offset;  // 0; a test hook sets it so that no wait can succeed
    uint64_t wait_limit_ns;
    int* status;           // != 0: a wait gave up
    // batched form: tiles claimed so far, and the problem's last tile in the list.
    // Until it is claimed a wait is for another problem's tile to end (whose own
    // waits are bounded), and its limit has not begun.
    const int* claimed = nullptr;
    int last_tile = 0;
};
struct ResidentGeom {
    int64_t N;
    int K, L, E, h;        // blocks, levels per round, levels per exchange, halo points per side
    int slots, buf_elems;  // tile slots per block, elements of one shared-memory buffer
    int pub, cap;          // points published at each end of a block, words per block
    int bc, last;          // boundary; levels after the last exchange
    int64_t exchanges, parity_words;
    ResidentSync sync;
};
// The shape with the least estimated time per level, false when N does not fit.
bool resident_plan(int eq, int esize, int64_t N, int sms, ResidentShape* out);
// 8-byte words of one parity, and exchanges of an advance of `levels` levels.
size_t resident_words(int eq, int esize, int64_t N, const ResidentShape& s);
int64_t resident_exchanges(const ResidentShape& s, int64_t levels);
// A -> B (the state ends in row B).
template <typename R>
cudaError_t launch_swept_resident(int eq, int bc, const R* A, R* B, int64_t N, int64_t levels, const ResidentShape& s,
                                  const ResidentSync& y, const Coefs<R>& c, cudaStream_t st);

// Many heat and KS problems in one launch (resident_batch.cu): a block keeps a
// tile, (problem, k), for its whole advance.
template <typename R> struct ResidentInst {
    const R* A;
    R* B;
    int eq;
    int64_t word_off;      // of the problem's first published word
    int last_tile;         // the problem's last tile in the list
    ResidentGeom g;        // sync unset
    Coefs<R> c;
};
struct ResidentBatchWork {
    const int2* tiles;     // (problem, tile), a problem's tiles together
    int ntiles;
    int* next_tile;        // zeroed per launch
    uint64_t* words;       // zeroed per launch
    int* status;
    uint64_t wait_limit_ns;
    uint32_t wait_offset;  // 0; a test hook sets it so that no wait can succeed
};
struct ResidentBatchShape {
    int variant = 0;       // of the kernel's tiles
    int blocks = 0;        // resident at once
};
enum ResidentBatchFit { RESIDENT_FITS, RESIDENT_TOO_LONG, RESIDENT_SLOWER };
// The tiles for problems of these sizes; TOO_LONG when some problem has more tiles
// than the launch has blocks (or the launch cannot run), SLOWER when the dataflow
// launch with widths by the batch's size is the faster form.
ResidentBatchFit resident_batch_choose(int esize, const std::vector<int64_t>& points, int sms, ResidentBatchShape* out);
ResidentGeom resident_batch_geom(int eq, int esize, int bc, int64_t N, int64_t levels, const ResidentBatchShape& s);
template <typename R>
cudaError_t launch_swept_resident_batch(const ResidentInst<R>* insts, const ResidentBatchWork& w,
                                        const ResidentBatchShape& shape, cudaStream_t s);

// The same for Euler (FP64): cells in shared memory, L levels per exchange, M = 1; P and
// warps unused.
bool resident_euler_plan(int bc, int64_t N, int sms, ResidentShape* out);
size_t resident_euler_words(int64_t N, const ResidentShape& s);
cudaError_t launch_swept_resident_euler(int bc, const double* A, double* B, int64_t N, int64_t levels,
                                        const ResidentShape& s, const ResidentSync& y, const Coefs<double>& c,
                                        cudaStream_t st);

}  // namespace swp
