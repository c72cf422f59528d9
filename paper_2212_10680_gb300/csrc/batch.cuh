// Batched lattices: many independent lattices (same component count and storage,
// any sizes, any mixtures) advanced together by one kernel per time step.
//
// Every lattice has a device-resident descriptor holding its StepArgs for both
// step parities (the ping-pong buffers swapped) and its own step counter.  A work list
// of (lattice, tile) items covers all lattices; a block copies the descriptor of its
// item's lattice into shared memory and runs the same phase functions as fused_step,
// so each lattice's arithmetic is exactly that of a single-lattice plain step: results
// are bit-identical alone and in any mix.  Two components in float or 16-bit storage take the
// packed step's tiles, with the descriptors in the launch's parameters (batch_pack).
#pragma once

#include "fmlbm_pack.cuh"

namespace fmlbm {

struct BatchLattice {
    StepArgs args[2];    // [step & 1]
    long long step;      // steps taken before the launches in flight (advanced by batch_advance)
    int active;          // 0: retired or not started
    int item0, nitems;   // its items in the work list
    int tile_y;          // the tile height its items were cut with
    int pad[3];
};

struct WorkItem {
    int lattice;
    int x0, y0;
};

// One step of every active lattice, `ahead` steps after the counters.
// Float storage capped at 64 registers (1024 threads per SM), as the single-lattice step.
template <int NC, int ST, int TY>
__global__ void __launch_bounds__(kTX* TY, ST == ST_F64 ? 1 : 1024 / (kTX * TY)) batch_step(BatchLattice* __restrict__ lat,
                                                      const WorkItem* __restrict__ work, int nwork, int ahead) {
    using Real = typename StoreTraits<ST>::Real;
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_batch[];
    auto& S = *reinterpret_cast<StepSmem<Real, NC, TY>*>(smem_batch);
    __shared__ __align__(16) StepArgs As;
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int tid = ty * kTX + tx;
    constexpr int NT = kTX * TY;
    constexpr int WORDS = sizeof(StepArgs) / 4;
    static_assert(sizeof(StepArgs) % 4 == 0, "StepArgs copied as words");
    for (int w = blockIdx.x; w < nwork; w += gridDim.x) {
        const WorkItem it = work[w];
        const BatchLattice* L = lat + it.lattice;
        if (!L->active) continue;  // uniform across the block
        const int* src = reinterpret_cast<const int*>(&L->args[(L->step + ahead) & 1]);
        int* dst = reinterpret_cast<int*>(&As);
        for (int k = tid; k < WORDS; k += NT) dst[k] = src[k];
        __syncthreads();
        const StepArgs& A = As;
        const MixConstT<Real>& m = mixc<Real>(A);
        const int nx = A.nx, ny = A.ny;
        const int x0 = it.x0, y0 = it.y0;
        const bool inner = x0 >= 3 && x0 + kTX + 3 <= nx && y0 >= 3 && y0 + TY + 3 <= ny;
        const int gxn = x0 + tx, gyn = y0 + ty;
        prefetch_force<Real, NC, TY>(A, S, tx, ty, gxn, gyn);
        Real g[NC][9], r[NC], jx, jy;
        phase1_global<NC, ST, TY>(A, m, S, g, r, jx, jy, x0, y0, inner, tx, ty, tid);
        __syncthreads();
        phase2<NC, TY, Real>(m, S, A.stencil, tid);
        __syncthreads();
        if (gxn < nx && gyn < ny) phase3<NC, ST, TY, false>(A, m, S, g, r, jx, jy, tx, ty, gxn, gyn);
        __syncthreads();  // As and the shared tiles are reused by the next item
    }
}

// One step of up to MAXL lattices of two components in float or 16-bit storage on 8-row tiles: the
// packed step's tiles, one block each, with the lattices' descriptors in the launch's parameters.
// A block finds its lattice by its index (the descriptors are in the order of their tiles) in
// registers that the whole warp shares, and reads plane addresses and mixture constants as
// constants, so that a block starts with its loads.  A step of 16 binaries of 88 to 484 nodes a side
// (971,000 nodes, FP32) takes 38.0 us, one of 12 of 64^2 to 184^2 9.8; with the descriptor copied from
// global to shared memory by every block 49.2 and 12.3 (two dependent reads and a barrier before
// the first load, and a shared-memory read for each address), with four blocks per multiprocessor
// 41.8 and 10.2.
struct PackLattice {
    int nx, ny, stencil, lagged;
    const void* Fin;
    void* Fout;
    ErrorLatch* err;
    const void* in[2 * 9];  // as Planes
    void* out[2 * 9];
    const float* g0in[2];
    float* g0out[2];
    MixConstT<float> mixf;
};
__device__ __forceinline__ bool checked_row(const PackLattice&, int) { return true; }
constexpr int kBatchGroup = 48;       // lattices in one launch (27 KB of parameters)
constexpr int kBatchGroupSmall = 16;  // fewer lattices take the launch with less to copy
constexpr int kBatchPackBlocks = 5;   // blocks per multiprocessor
template <int MAXL>
struct PackBatch {
    int n;
    int first[kBatchGroup];  // first block of each lattice
    PackLattice lat[MAXL];
};
template <int ST, bool SPEC, int MAXL>
__global__ void __launch_bounds__(kTX * 8, kBatchPackBlocks) batch_pack(const __grid_constant__ PackBatch<MAXL> B) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_batch_pack[];
    int l = 0;
#pragma unroll
    for (int s = MAXL > 32 ? 32 : MAXL / 2; s > 0; s >>= 1)
        if (l + s < B.n && B.first[l + s] <= (int)blockIdx.x) l += s;
    const PackLattice& L = B.lat[l];
    const int t = blockIdx.x - B.first[l], cols = (L.nx + kTX - 1) / kTX, row = t / cols;
    pack_tile<2, ST, SPEC, false>(L, L, *reinterpret_cast<PackSmem<2, 8>*>(smem_batch_pack), nullptr,
                                  (t - row * cols) * kTX, row * 8, 0, 0, 0);
}

// Counts n steps on every active lattice.
__global__ void batch_advance(BatchLattice* __restrict__ lat, int nlat, int n) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < nlat && lat[k].active) lat[k].step += n;
}

// Per-item partial sums (2 NC + 2 doubles: sum rho_i, sum (rho - rho_prev)^2, sum rho^2, then
// the phase measure's sum ln rho_i) over the item's tile of 32 x tile_y nodes, then
// rho_prev <- rho, with the node sums, the warp tree and the double strip sums of
// reduce_partial and lnrho_partial (the rows of a taller tile go through the same
// compensated sums before the tree).  The items of one lattice are contiguous, so
// batch_reduce_final sums each lattice in a fixed order.
template <int NC>
constexpr int kBatchSums = 2 * NC + 2;

template <int NC, int ST>
__global__ void __launch_bounds__(kTX* 8) batch_reduce(BatchLattice* __restrict__ lat, const WorkItem* __restrict__ work,
                                                       int nwork, void* const* __restrict__ rho_prev,
                                                       double* __restrict__ partial) {
    using Real = typename StoreTraits<ST>::Real;
    constexpr int K = kBatchSums<NC>;
    const int w = blockIdx.x;
    if (w >= nwork) return;
    const WorkItem it = work[w];
    const BatchLattice* L = lat + it.lattice;
    const StepArgs& A = L->args[L->step & 1];
    const int nx = A.nx, ny = A.ny, nxy = nx * ny;
    Real* prev = static_cast<Real*>(rho_prev[it.lattice]);
    Sum2<Real> acc[K];
#pragma unroll
    for (int k = 0; k < K; ++k) acc[k] = s2_of(Real(0));
    if (L->active) {
        for (int ry = threadIdx.y; ry < L->tile_y; ry += 8) {
            const int x = it.x0 + threadIdx.x, y = it.y0 + ry;
            if (x < nx && y < ny) {
                const bool inner = x >= 1 && x + 1 < nx && y >= 1 && y + 1 < ny;
                Real r[NC];
                pull_rho<NC, ST>(A, x, y, inner, nx, ny, nxy, r);
                const int node = y * nx + x;
                Real pv[NC];
#pragma unroll
                for (int i = 0; i < NC; ++i) pv[i] = prev[(size_t)i * nxy + node];
                Sum2<Real> a[NC + 2], l[NC];
                diag_node<NC, Real>(r, pv, 1, a);
                lnrho_node<NC, Real>(r, l);
#pragma unroll
                for (int k = 0; k < NC + 2; ++k) acc[k] = s2_add(acc[k], a[k]);
#pragma unroll
                for (int i = 0; i < NC; ++i) acc[NC + 2 + i] = s2_add(acc[NC + 2 + i], l[i]);
#pragma unroll
                for (int i = 0; i < NC; ++i) prev[(size_t)i * nxy + node] = r[i];
            }
        }
    }
    __shared__ Sum2<Real> red[8][K];
    sums_warp<K, Real>(acc, red[threadIdx.y]);
    __syncthreads();
    const int tid = threadIdx.y * kTX + threadIdx.x;
    if (tid < K) partial[(size_t)w * K + tid] = sums_strip<K, Real>(red, 0, tid, 0);
}

// One block per (lattice, sum), in the order of sum_columns (a thread per sum added a lattice's
// items one after the other: 80 us of every check of a 16-lattice sweep).
template <int NC>
__global__ void __launch_bounds__(kFinalThreads) batch_reduce_final(const BatchLattice* __restrict__ lat,
                                                                    const double* __restrict__ partial,
                                                                    double* __restrict__ out) {
    constexpr int K = kBatchSums<NC>;
    const int l = blockIdx.x / K, q = blockIdx.x - l * K;
    const double t = column_sum<K>(partial + (size_t)lat[l].item0 * K, lat[l].nitems, q);
    if (threadIdx.x == 0) out[blockIdx.x] = t;
}

// The two phases of a lattice from its densities rho[N][ny][nx] (mass, double), read as
// means over 2 x 2 blocks of nodes (block (bx, by) holds the nodes 2 bx, 2 bx + 1 in x and
// 2 by, 2 by + 1 in y, periodic at an odd edge).  The discrete force of Eqs. eqforcefinal and
// eq1stder differences a field over two nodes, so a field alternating from node to node (a
// checkerboard) feels no force, and at rest the well-balanced equilibrium (rho_0 = 0) holds
// every node's mass in its rest population, so nothing streams it away either: a checkerboard
// that the transient of a sharp interface excites stays in both bulk phases.  Each parity
// sublattice is then out of equilibrium on its own; the block mean is the thermodynamic state.
// out = the block-mean molar densities rho~_i at the block of largest total molar density
// sum_i rho_i / M_i (liquid) [N], then at the block of smallest (vapour) [N]; ties to the
// lowest block index (row-major): a choice, so the same however the node blocks are divided among
// thread blocks.  Bound by its double divisions (N for each node), hence many thread blocks: with one
// 350 us on average over 16 lattices of 8,600 to 171,000 nodes.
constexpr int kPhaseThreads = 512;
constexpr int kPhaseBlocks = 256;
struct PhaseNodes {      // the largest and smallest density seen and their node blocks (-1: none)
    double hi, lo;
    long long ih, il;
};
__device__ __forceinline__ void block_nodes(long long k, int nx, int ny, long long (&node)[4]) {
    const int bxn = (nx + 1) / 2;
    const int x0 = 2 * (int)(k % bxn), y0 = 2 * (int)(k / bxn);
    const int x1 = x0 + 1 < nx ? x0 + 1 : 0, y1 = y0 + 1 < ny ? y0 + 1 : 0;
    node[0] = (long long)y0 * nx + x0;
    node[1] = (long long)y0 * nx + x1;
    node[2] = (long long)y1 * nx + x0;
    node[3] = (long long)y1 * nx + x1;
}

// The block's choice from every thread's, in thread 0's result.
__device__ __forceinline__ PhaseNodes phase_reduce(const PhaseNodes& mine) {
    __shared__ PhaseNodes v[kPhaseThreads];
    const int t = threadIdx.x;
    v[t] = mine;
    __syncthreads();
    for (int w = kPhaseThreads / 2; w > 0; w >>= 1) {
        if (t < w) {
            const PhaseNodes o = v[t + w];
            if (o.ih >= 0 && (v[t].ih < 0 || o.hi > v[t].hi || (o.hi == v[t].hi && o.ih < v[t].ih))) {
                v[t].hi = o.hi;
                v[t].ih = o.ih;
            }
            if (o.il >= 0 && (v[t].il < 0 || o.lo < v[t].lo || (o.lo == v[t].lo && o.il < v[t].il))) {
                v[t].lo = o.lo;
                v[t].il = o.il;
            }
        }
        __syncthreads();
    }
    return v[0];
}

template <int NC>
__global__ void __launch_bounds__(kPhaseThreads) phase_nodes(const double* __restrict__ rho, int nx, int ny,
                                                             MixConstT<double> m, PhaseNodes* __restrict__ part) {
    const long long nxy = (long long)nx * ny;
    const long long nblk = (long long)((nx + 1) / 2) * ((ny + 1) / 2);
    double hi = -1.0, lo = 0.0;
    long long ih = -1, il = -1;
    for (long long k = (long long)blockIdx.x * kPhaseThreads + threadIdx.x; k < nblk;
         k += (long long)gridDim.x * kPhaseThreads) {
        long long node[4];
        block_nodes(k, nx, ny, node);
        double s = 0.0;
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int i = 0; i < NC; ++i) s += rho[i * nxy + node[q]] / m.M[i];
        if (ih < 0 || s > hi) { hi = s; ih = k; }          // k increases: first maximum kept
        if (il < 0 || s < lo) { lo = s; il = k; }
    }
    const PhaseNodes best = phase_reduce(PhaseNodes{hi, lo, ih, il});
    if (threadIdx.x == 0) part[blockIdx.x] = best;
}

template <int NC>
__global__ void __launch_bounds__(kPhaseThreads) phase_pick(const double* __restrict__ rho, int nx, int ny,
                                                            MixConstT<double> m, const PhaseNodes* __restrict__ part,
                                                            int nparts, double* __restrict__ out) {
    static_assert(kPhaseBlocks <= kPhaseThreads, "one thread per partial choice");
    const int t = threadIdx.x;
    const PhaseNodes best = phase_reduce(t < nparts ? part[t] : PhaseNodes{-1.0, 0.0, -1, -1});
    const long long nxy = (long long)nx * ny;
    if (t < 2 * NC) {
        const int i = t % NC;
        long long node[4];
        block_nodes(t < NC ? best.ih : best.il, nx, ny, node);
        double v = 0.0;
#pragma unroll
        for (int q = 0; q < 4; ++q) v += rho[i * nxy + node[q]] / m.M[i];
        out[t] = 0.25 * v;
    }
}

}  // namespace fmlbm
