// Resident form of a single Euler advance: one launch, the cells in shared memory
// from the first step to the last (resident.cu has the idea and the exchange).
//
// Each block owns a contiguous part of the grid and holds it with h = 2 L halo
// cells on each side.  Level j of the L between two exchanges computes the
// cells [2 j, W - 2 j) of the tile's W = own + 4 L, in the four passes of the
// swept tiles: pressure per cell, the limiter per cell, one flux per interface,
// the update.  After L levels the owned cells are current and the halos are
// fetched again.  An update costs some hundred FP64 operations, so a level of
// even one cell per lane outlasts an exchange many times over and L is
// small; only the smallest grids, whose tiles do not fill the block's warps,
// take more levels per exchange.
//
// What bounds it: the FP64 pipe (93 % busy with 200000 cells limited everywhere); on
// small grids the chain of the passes and their barriers (Sod with 4096 cells: 5740
// clocks per level in the tile, pipe 27 %) and, at an exchange, the wait for the
// slowest tile.  A pass runs its rows of 32 cells on the SM's four sub-partitions in
// turn, so its time goes with ceil(rows / 4); a grid of 152 SMs x 128 cells or fewer
// has one row each, where the swept form took 2H - 1 dependent levels per H levels of
// progress.  Clocks (1/2.07 us) per level, Sod in its first hundred steps / limited
// everywhere, here (the dataflow launch when this form came): N = 4096 8100 / 8200
// (21200 / 22600), 65536 22500 / 32700 (28000 / 48700), 200000 54000 / 91000 (62200 /
// 115100).  Grids whose cells do not fit shared memory (N above about 330000), and
// Dirichlet ones above about 57000 cells (resident_euler_plan), keep that launch.
//
// Dirichlet ends: the tile's slots beyond an end hold that end's ghost state in
// both rows and are never updated (Appendix C's two ghost cells, and more of
// the same).  Periodic ends wrap.
#include <algorithm>

#include "geometry.cuh"
#include "resident.cuh"
#include "resident.h"

namespace swp {

namespace {

// Threads per block: 16 warps hide the latencies that 8 leave at each sub-partition
// (200000 cells limited everywhere: 91000 against 94800 clocks per level; 131072
// cells, Sod: 36800 against 38200); a SPLIT tile has work for few warps (N = 4096: 8240
// with 16, 8120 with 8).
template <bool SPLIT>
constexpr int kThreads = SPLIT ? 256 : 512;

// SPLIT: for tiles of at most two rows of cells, whose passes would leave
// sub-partitions idle: a cell's pressure and its sqrt(rho), and the two sides of
// an interface, are tasks of their own on different warps (N = 4096: 8100 against
// 10330 clocks per level).
template <bool SPLIT>
__global__ void __launch_bounds__(kThreads<SPLIT>)
    swept_resident_euler_kernel(const double* A, double* B, ResidentGeom g, Coefs<double> cp)
{
    using R = double;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Coefs<R> c = lane_coefs<R, EULER>(cp);
    const Units<R> ku = make_units<R, EULER>();
    constexpr int T = kThreads<SPLIT>;
    const int tid = threadIdx.x;
    const int k = blockIdx.x, K = g.K, h = g.h, cap = g.cap, pub = g.pub;
    const int64_t N = g.N;
    const int64_t b0 = k * N / K;
    const int own = (int)((k + 1) * N / K - b0), W = own + 2 * h, GW = W + 1;
    R* row0 = reinterpret_cast<R*>(smem_raw);   // [3][W], even levels
    R* row1 = row0 + 3 * W;                     // [3][W], odd levels
    R* P = row1 + 3 * W;                        // pressures
    R* Cc = P + W;                              // [3][W], kept values (euler_limit)
    R* G = Cc + 3 * W;                          // [3][W + 1]: interface between slots s - 1 and s
    R* S = G + 3 * GW;                          // SPLIT: [2][8][W + 1], the sides of every interface
    int* hoff = reinterpret_cast<int*>(S + (SPLIT ? 16 * GW : 0));   // published word of each halo cell, -1: a ghost
    // slots of the domain: all of them, or those between Dirichlet ends
    int c_lo = 0, c_hi = W;
    if (g.bc == DIRICHLET) {
        if (b0 < h) c_lo = h - (int)b0;
        if (N - (b0 - h) < W) c_hi = (int)(N - (b0 - h));
    }
    for (int s = tid; s < W; s += T) {
        const bool left = s < c_lo, ghost = left || s >= c_hi;
        const int64_t p = ghost ? 0 : fold(b0 - h + s, N, PERIODIC);
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            const R x = ghost ? (left ? c.ghost_l[v] : c.ghost_r[v]) : A[v * N + p];
            row0[v * W + s] = x;
            row1[v * W + s] = x;
        }
    }
    if (g.exchanges > 0) {
        for (int e = tid; e < 2 * h; e += T) {
            const int s = e < h ? e : own + e;
            hoff[e] = s < c_lo || s >= c_hi
                          ? -1
                          : word_of((int)fold(b0 - h + s, N, PERIODIC), (int)N, K, pub, cap);
        }
    }
    __syncthreads();
    for (int64_t x = 0;; ++x) {
        const int levels = x < g.exchanges ? g.E : g.last;
        for (int j = 1; j <= levels; ++j) {
            const bool odd = j & 1;
            const R* src = odd ? row0 : row1;
            R* dst = odd ? row1 : row0;
            const R kh = odd ? c.kh[0] : c.kh[1];
            const int lo = 2 * j, hi = W - 2 * j;
            if constexpr (SPLIT) {
                // whole warps for each, so that none runs both
                const int n = (hi - lo + 4 + 31) & ~31;
                for (int t = tid; t < 2 * n; t += T) {
                    const int s = lo - 2 + (t < n ? t : t - n);
                    if (s >= hi + 2) continue;
                    if (t < n) P[s] = euler_cell(src[s], src[W + s], src[2 * W + s], c.gm1, Cc[s], Cc[W + s], ku);
                    else Cc[2 * W + s] = Fp<R>::sqrt(src[s]);
                }
            } else {
                for (int s = lo - 2 + tid; s < hi + 2; s += T)
                    P[s] = euler_cell(src[s], src[W + s], src[2 * W + s], c.gm1, Cc[s], Cc[W + s], ku);
            }
            __syncthreads();
            for (int s = lo - 1 + tid; s < hi + 1; s += T)
                euler_limit<SPLIT>(P[s - 1], P[s], P[s + 1], src[s], Cc[s], Cc[W + s], Cc[2 * W + s], ku);
            __syncthreads();
            if constexpr (SPLIT) {
                const int n = hi - lo + 1;
                for (int t = tid; t < 2 * n; t += T) {
                    const int right = t >= n, s = lo + (right ? t - n : t);
                    const int a = s - 1 + right, b = s - right;   // the side's cell, and the other
                    const R qc[3] = {src[a], src[W + a], src[2 * W + a]};
                    const R qo[3] = {src[b], src[W + b], src[2 * W + b]};
                    const R cc[3] = {Cc[a], Cc[W + a], Cc[2 * W + a]};
                    R q[3], f1, f2, u, e, w;
                    euler_side(qc, qo, P[a], cc, right ? cc[1] : cc[0], c.gm1, q, f1, f2, u, e, w, ku);
                    R* o = S + right * 8 * GW + s;
                    o[0] = q[0];
                    o[GW] = q[1];
                    o[2 * GW] = q[2];
                    o[3 * GW] = f1;
                    o[4 * GW] = f2;
                    o[5 * GW] = right ? Fp<R>::mul(w, u, ku) : u;
                    o[6 * GW] = right ? Fp<R>::mul(w, e, ku) : e;
                    o[7 * GW] = w;
                }
                __syncthreads();
                for (int s = lo + tid; s <= hi; s += T) {
                    const R* l = S + s;
                    const R* r = l + 8 * GW;
                    const R ql[3] = {l[0], l[GW], l[2 * GW]}, qr[3] = {r[0], r[GW], r[2 * GW]};
                    R g3[3];
                    euler_join(ql, l[3 * GW], l[4 * GW], l[5 * GW], l[6 * GW], l[7 * GW], qr, r[3 * GW], r[4 * GW],
                               r[5 * GW], r[6 * GW], r[7 * GW], c.ggm1, g3, ku);
                    G[s] = g3[0];
                    G[GW + s] = g3[1];
                    G[2 * GW + s] = g3[2];
                }
            } else for (int s = lo + tid; s <= hi; s += T) {
                const R qa[3] = {src[s - 1], src[W + s - 1], src[2 * W + s - 1]};
                const R qb[3] = {src[s], src[W + s], src[2 * W + s]};
                const R ca[3] = {Cc[s - 1], Cc[W + s - 1], Cc[2 * W + s - 1]};
                const R cb[3] = {Cc[s], Cc[W + s], Cc[2 * W + s]};
                R g3[3];
                euler_interface(qa, qb, P[s - 1], P[s], ca, cb, c.gm1, c.ggm1, g3, ku);
                G[s] = g3[0];
                G[GW + s] = g3[1];
                G[2 * GW + s] = g3[2];
            }
            __syncthreads();
            const int end = min(hi, c_hi);
            for (int s = max(lo, c_lo) + tid; s < end; s += T) {
#pragma unroll
                for (int v = 0; v < 3; ++v)
                    dst[v * W + s] =
                        euler_update(G[v * GW + s + 1], G[v * GW + s], row0[v * W + s], kh, ku);   // base u^m
            }
            __syncthreads();
        }
        if (x >= g.exchanges) break;
        const uint32_t seq = g.sync.seq + (uint32_t)x;
        uint64_t* words = g.sync.words + (x & 1) * g.parity_words;
        const int words_here = 3 * min(own, 2 * pub);
        for (int i = tid; i < words_here; i += T) {
            const int cell = i / 3, v = i - 3 * cell;
            const int o = cell < pub || own <= 2 * pub ? cell : own - 2 * pub + cell;
            Word<R>::put(words + 2 * ((int64_t)k * cap * 3 + i), row0[v * W + h + o], seq);
        }
        int fail = 0;
        for (int i = tid; i < 6 * h; i += T) {
            const int e = i / 3, v = i - 3 * e;
            if (hoff[e] < 0) continue;
            R q;
            if (!wait_word<R>(words + 2 * ((int64_t)hoff[e] * 3 + v), seq + g.sync.wait_offset, g.sync, q)) {
                fail = 1;
                break;
            }
            row0[v * W + (e < h ? e : own + e)] = q;
        }
        if (__syncthreads_or(fail)) return;
    }
    for (int o = tid; o < own; o += T) {
#pragma unroll
        for (int v = 0; v < 3; ++v) B[v * N + b0 + o] = row0[v * W + h + o];
    }
}

size_t smem_of(int own, int L, bool split)
{
    const size_t W = (size_t)own + 4 * (size_t)L;
    return sizeof(double) * (6 * W + W + 3 * W + (split ? 19 : 3) * (W + 1)) + sizeof(int) * 4 * (size_t)L;
}

// Rows of 32 of n cells, in turns of the SM's four sub-partitions.
int turns(int n) { return ((n + 31) / 32 + 3) / 4; }

}  // namespace

bool resident_euler_plan(int bc, int64_t N, int sms, ResidentShape* out)
{
    *out = ResidentShape();
    if (N < 32 || sms < 1) return false;
    const int K = (int)std::min<int64_t>(sms, std::max<int64_t>(1, N / 8));
    if ((N + 1) * (K + 1) >= (int64_t)1 << 31) return false;
    const int own = (int)((N + K - 1) / K);
    // The blocks keep the pace of the slowest one, a tile limited everywhere, while the
    // dataflow launch's is the average of the grid.  Dirichlet ends are a tube whose
    // waves hold a part of it: beyond three turns of rows per pass (own + the shortest
    // halos; 57152 cells on 152 SMs) the dataflow launch is the faster form.  us per step
    // over 100 to 800 steps of the Sod tube, on chip / dataflow, at t = 0.03 / 0.1 / 0.2:
    //    55109   25.3 / 24.9   25.3 / 25.7    25.4 / 33.7
    //    60001   31.0 / 25.9   31.0 / 26.4    31.1 / 35.1
    //    77936   42.4 / 28.4   42.5 / 29.0    42.7 / 38.9
    //   131072   56.5 / 38.2   57.2 / 39.1    57.3 / 53.5
    //   300001  126.7 / 78.8  127.3 / 80.7   128.1 / 111
    // (its first steps, when hardly a cell is limited, are faster on chip: 131072 cells
    // 35.6 / 37.1 over 250 steps.)  Periodic flows are mostly limited everywhere (131072:
    // 57.5 / 68.9) and stay on chip.
    if (bc == DIRICHLET && turns(own + 8) > 3) return false;
    double best = 0.0;
    for (int split = 0; split < 2; ++split)
        for (int L = 2; L <= 48; L += 2) {
            const int W = own + 4 * L;
            if (smem_of(own, L, split) > kResidentSmem) break;
            // FP64 operations of the passes (limited on some interfaces), their
            // barriers and latencies, and an exchange
            double clocks = 1700.0 + 20.0 * L;
            for (int j = 1; j <= L; ++j) {
                const int n = W - 4 * j;
                const int flux = split ? 28 * turns(2 * n + 2) + 33 * turns(n + 1) : 82 * turns(n + 1);
                const int cell = split ? 10 * turns(2 * ((n + 4 + 31) & ~31)) + 12 * turns(n + 2)
                                       : 11 * turns(n + 4) + 20 * turns(n + 2);
                clocks += 66.0 * (cell + flux + 6 * turns(n)) + (split ? 700.0 : 500.0);
            }
            clocks /= L;
            if (best == 0.0 || clocks < best) {
                best = clocks;
                out->K = K;
                out->L = L;
                out->M = 1;
                out->split = split != 0;
            }
        }
    return best > 0.0;
}

size_t resident_euler_words(int64_t N, const ResidentShape& s)
{
    const int own = (int)((N + s.K - 1) / s.K);
    return (size_t)s.K * std::min(own, 2 * 2 * s.L) * 3 * 2;
}

cudaError_t launch_swept_resident_euler(int bc, const double* A, double* B, int64_t N, int64_t levels,
                                        const ResidentShape& s, const ResidentSync& y, const Coefs<double>& c,
                                        cudaStream_t st)
{
    ResidentGeom g{};
    g.N = N;
    g.K = s.K;
    g.L = g.E = s.L;
    g.h = 2 * s.L;
    const int own = (int)((N + s.K - 1) / s.K);
    g.pub = g.h;
    g.cap = std::min(own, 2 * g.pub);
    g.exchanges = resident_exchanges(s, levels);
    g.last = (int)(levels - g.exchanges * g.E);
    g.bc = bc;
    g.sync = y;
    g.parity_words = (int64_t)resident_euler_words(N, s);
    const size_t smem = smem_of(own, s.L, s.split);
    const void* fn = s.split ? (const void*)swept_resident_euler_kernel<true>
                             : (const void*)swept_resident_euler_kernel<false>;
    const cudaError_t e = allow_resident_smem(fn);
    if (e != cudaSuccess) return e;
    void* args[] = {(void*)&A, (void*)&B, (void*)&g, (void*)&c};
    return cudaLaunchCooperativeKernel(fn, dim3((unsigned)s.K), dim3(s.split ? kThreads<true> : kThreads<false>), args,
                                       smem, st);
}

}  // namespace swp
