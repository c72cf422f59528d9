// The split step: one time step in two launches, for the forms that evaluate ln f in double.
//
// GB300 issues one FP64 warp instruction per multiprocessor sub-partition every 64 cycles (19
// per warp instruction and multiprocessor with all four busy), whatever its active lanes, so
// these forms are bound by the number of FP64 warp instructions and by how many sub-partitions
// have some.  fused_step evaluates ln f on the halo ring of every tile (14 warps' worth of it for
// 8 warps of nodes) and gives a 64^2 lattice to 16 of the 152 multiprocessors.  Here
//
//   node_fields     computes rho_i, the first moment, rho~_i and ln f_i (steps 1-5) once per node
//                   and writes them to scratch planes;
//   collide_fields  reads rho~ and ln f of its tile with their halo, forms Phi (step 6) and
//                   collides (steps 7-9).
//
// The planes cost 2 x (3 N + 2) values of traffic per node, which these forms have to spare.  Both
// use the functions of fused_step on the same operands: same bits.
#pragma once

#include "fmlbm_kernels.cuh"

namespace fmlbm {

// Scratch planes per node: rho~ [N], ln f [N] and, in FP64 storage (whose sums are worth storing),
// rho [N] and the first moment [2].
template <int ST> constexpr bool kSplitStep = ST == ST_F64 || kLnf64<ST>;
constexpr int split_planes(int nc, bool f64) { return f64 ? 3 * nc + 2 : 2 * nc; }

template <int NC, int ST, int TY, bool DIAG>
__global__ void __launch_bounds__(kTX* TY) node_fields(const __grid_constant__ StepArgs A) {
    using Real = typename StoreTraits<ST>::Real;
    pdl_wait();
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int x = blockIdx.x * kTX + tx, y = blockIdx.y * TY + ty;
    const int nx = A.nx, ny = A.ny, nxy = nx * ny;
    const bool valid = x < nx && y < ny;
    extern __shared__ __align__(16) unsigned char smem_nf[];
    Real* pv_s = reinterpret_cast<Real*>(smem_nf);
    if constexpr (DIAG) {
        diag_prefetch<NC, Real, TY>(A, pv_s, tx, ty, x, y);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
    Real r[NC];
#pragma unroll
    for (int i = 0; i < NC; ++i) r[i] = Real(0);
    if (valid) {
        const MixConstT<Real>& m = mixc<Real>(A);
        const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
        const int ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
        Real g[NC][9], rt[NC], lnf[NC], jx, jy;
#pragma unroll
        for (int a = 0; a < 9; ++a) {
            const int src = pull_src(a, x, y, xm, xp, ym, yp, nx);
#pragma unroll
            for (int i = 0; i < NC; ++i) g[i][a] = load_g<ST>(A, i, a, (size_t)src, (size_t)nxy);
        }
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            r[i] = sum9(g[i]);
            if constexpr (ST == ST_F64) moment_j(g[i], i == 0, jx, jy);
            rt[i] = vmul(r[i], m.invM[i]);
        }
        const Real beta = node_lnf_st<NC, kLnf64<ST>, Real>(A, m, rt, lnf);
        domain_check<NC, Real>(A, rt, lnf, beta, x, 0, y, checked_row(A, y) ? 1u : 0u);
        Real* f = static_cast<Real*>(A.fields) + (size_t)y * nx + x;
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            f[(size_t)i * nxy] = rt[i];
            f[(size_t)(NC + i) * nxy] = lnf[i];
            if constexpr (ST == ST_F64) f[(size_t)(2 * NC + i) * nxy] = r[i];
        }
        if constexpr (ST == ST_F64) {
            f[(size_t)(3 * NC) * nxy] = jx;
            f[(size_t)(3 * NC + 1) * nxy] = jy;
        }
    }
    if constexpr (DIAG)
        diag_tile<NC, Real, TY>(A, r, pv_s, tx, ty, x, y, blockIdx.y * TY, blockIdx.y, blockIdx.x, gridDim.x);
}

template <int NC, int ST, int TY>
__global__ void __launch_bounds__(kTX* TY) collide_fields(const __grid_constant__ StepArgs A) {
    using Real = typename StoreTraits<ST>::Real;
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_cf[];
    auto& S = *reinterpret_cast<StepSmem<Real, NC, TY>*>(smem_cf);
    const MixConstT<Real>& m = mixc<Real>(A);
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * kTX + tx;
    const int x0 = blockIdx.x * kTX, y0 = blockIdx.y * TY;
    const int nx = A.nx, ny = A.ny, nxy = nx * ny;
    const int x = x0 + tx, y = y0 + ty;
    const bool valid = x < nx && y < ny;
    prefetch_force<Real, NC, TY>(A, S, tx, ty, x, y);
    const Real* f = static_cast<const Real*>(A.fields);
    // rho~ on the tile + 2 and ln f on the tile + 1
    constexpr int W2 = kTX + 4;
    for (int e = tid; e < W2 * (TY + 4); e += kTX * TY) {
        const int by = e / W2, bx = e - by * W2;
        const size_t node = (size_t)wrap(y0 - 2 + by, ny) * nx + wrap(x0 - 2 + bx, nx);
        const bool in = bx >= 1 && bx <= kTX + 2 && by >= 1 && by <= TY + 2;
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            S.rt.v[i][by][bx] = f[(size_t)i * nxy + node];
            if (in) S.lf.v[i][by - 1][bx - 1] = f[(size_t)(NC + i) * nxy + node];
        }
    }
    Real g[NC][9], r[NC], jx = Real(0), jy = Real(0);
    if (valid) {
        const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
        const int ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
#pragma unroll
        for (int a = 0; a < 9; ++a) {
            const int src = pull_src(a, x, y, xm, xp, ym, yp, nx);
#pragma unroll
            for (int i = 0; i < NC; ++i) g[i][a] = load_g<ST>(A, i, a, (size_t)src, (size_t)nxy);
        }
        if constexpr (ST == ST_F64) {
            const size_t node = (size_t)y * nx + x;
#pragma unroll
            for (int i = 0; i < NC; ++i) r[i] = f[(size_t)(2 * NC + i) * nxy + node];
            jx = f[(size_t)(3 * NC) * nxy + node];
            jy = f[(size_t)(3 * NC + 1) * nxy + node];
        } else {
#pragma unroll
            for (int i = 0; i < NC; ++i) {
                r[i] = sum9(g[i]);
                moment_j(g[i], i == 0, jx, jy);
            }
        }
    }
    __syncthreads();
    phase2<NC, TY, Real>(m, S, A.stencil, tid);
    __syncthreads();
    if (valid) phase3<NC, ST, TY, false>(A, m, S, g, r, jx, jy, tx, ty, x, y);
}

}  // namespace fmlbm
