// The packed step: the fused time step of fused_step on 32 x 8 tiles with two components per
// value (fmlbm_comps.cuh); the shared tiles hold a pair side by side, so that a stencil value of
// both is one 8-byte access.
#pragma once

#include "fmlbm_comps.cuh"

namespace fmlbm {

// Lattices of at least this many nodes take the packed step (two components; GB300, us per step,
// one component per value -> packed): 256^2 FP32 4.26 -> 4.20, 384^2 6.34 -> 5.93, 512^2 9.80 -> 9.20,
// 777x523 FP16 13.96 -> 12.76; below, the fewer registers only cost: 128^2 3.19 -> 3.29.  Three
// components spill or lose a block per multiprocessor: 512^2 FP32 13.5 -> 14.1.
constexpr size_t kPackNodes = 1 << 16;

// A field of the tile with a halo of H nodes, pairs of components side by side.
template <int NC, int TY, int H>
struct PackTile {
    static_assert(NC % 2 == 0, "components come in pairs");
    float2 p[NC / 2][TY + 2 * H][kTX + 2 * H];
};
template <int NC, int TY, int H>
__device__ __forceinline__ float2* tile_row(PackTile<NC, TY, H>& t, PairOf of, int cy) { return t.p[of.k][cy]; }

template <int NC, int TY>
struct PackSmem {
    PackTile<NC, TY, 2> rt;  // rho~ on tile + 2
    PackTile<NC, TY, 1> lf;  // ln f on tile + 1
    PackTile<NC, TY, 1> G;   // Phi on tile + 1
    float Fl[2][TY][kTX];    // stored total force at the tile's nodes (lagged reading)
};

// Finite differences at column cx of three consecutive rows (n above, c, s below): the
// operations of grad_at and lap_at.
__device__ __forceinline__ void grad_tile(const float2* rn, const float2* rc, const float2* rs, int cx, int stencil,
                                          float2& gx, float2& gy) {
    using V = float2;
    const V e = rc[cx + 1], w = rc[cx - 1], n = rn[cx], s = rs[cx];
    if (stencil == 1) {
        gx = vmul(vbc<V>(0.5f), vsub(e, w));
        gy = vmul(vbc<V>(0.5f), vsub(n, s));
    } else {
        const V ne = rn[cx + 1], nw = rn[cx - 1], sw = rs[cx - 1], se = rs[cx + 1];
        const V third = vbc<V>(float(1.0 / 3.0)), twelfth = vbc<V>(float(1.0 / 12.0));
        gx = vfma(vsub(e, w), third, vmul(vadd(vsub(ne, nw), vsub(se, sw)), twelfth));
        gy = vfma(vsub(n, s), third, vmul(vsub(vadd(ne, nw), vadd(sw, se)), twelfth));
    }
}
__device__ __forceinline__ float2 lap_tile(const float2* rn, const float2* rc, const float2* rs, int cx, int stencil) {
    using V = float2;
    const V c = rc[cx];
    const V ax = vadd(vadd(rc[cx + 1], rc[cx - 1]), vadd(rn[cx], rs[cx]));
    const V m4 = vbc<V>(-4.f);
    if (stencil == 1) return vfma(m4, c, ax);
    const V dg = vadd(vadd(rn[cx + 1], rn[cx - 1]), vadd(rs[cx - 1], rs[cx + 1]));
    return vfma(vfma(m4, c, ax), vbc<V>(float(2.0 / 3.0)), vmul(vfma(m4, c, dg), vbc<V>(float(1.0 / 6.0))));
}

// Phi at position (cx, cy) of the tile + 1 box (phase2_core).
template <int NC, int TY>
__device__ __forceinline__ void pack_phi(const MixConstT<float>& m, PackSmem<NC, TY>& S, int stencil, int cx, int cy) {
    Comps<NC> L;
    each_group<NC>([&](auto of) {
        of(L) = lap_tile(tile_row(S.rt, of, cy + 2), tile_row(S.rt, of, cy + 1), tile_row(S.rt, of, cy), cx + 1, stencil);
    });
    each_group<NC>([&](auto of) {
        float2 Gi = vmul(of.col(m.kap, 0), vbc<float2>(comp(L, 0)));
#pragma unroll
        for (int j = 1; j < NC; ++j) Gi = vfma(of.col(m.kap, j), vbc<float2>(comp(L, j)), Gi);
        tile_row(S.G, of, cy)[cx] = vfma(vbc<float2>(-m.RT), tile_row(S.lf, of, cy)[cx], Gi);
    });
}

// The pulled values of a node: the nine of component i through the plane base addresses.
template <int NC, int ST, typename PL>
__device__ __forceinline__ void pack_pull(const PL& P, bool inner, int wx, int wy, int nx, int ny, Comps<NC> (&g)[9]) {
    const int node = wy * nx + wx;
    int xm = wx - 1, xp = wx + 1, ym = wy - 1, yp = wy + 1;
    if (!inner) {
        xm = wx == 0 ? nx - 1 : xm;
        xp = wx == nx - 1 ? 0 : xp;
        ym = wy == 0 ? ny - 1 : ym;
        yp = wy == ny - 1 ? 0 : yp;
    }
#pragma unroll
    for (int a = 0; a < 9; ++a) {
        const int src = inner ? node - ey(a) * nx - ex(a) : pull_src(a, wx, wy, xm, xp, ym, yp, nx);
#pragma unroll
        for (int i = 0; i < NC; ++i) set_comp(g[a], i, load_gp<ST>(P, i, a, src));
    }
}

// Densities (step 1) of a node from its pulled values, and rho~.
template <int NC>
__device__ __forceinline__ void pack_rho(const MixConstT<float>& m, const Comps<NC> (&g)[9], Comps<NC>& r, Comps<NC>& rt) {
    each_group<NC>([&](auto of) {
        float2 s = of(g[0]);
#pragma unroll
        for (int a = 1; a < 9; ++a) s = vadd(s, of(g[a]));
        of(r) = s;
        of(rt) = vmul(s, of.of(m.invM));
    });
}

// One tile of the packed step: of a lattice's StepArgs and Planes, or of a batch's descriptor with
// the members used here.  DIAG: the sums of a diagnostics request where A asks for them, with pv_s
// their shared memory and the tile's place (row, col of cols) in their order.
// SPEC: the Peng-Robinson EOS, isotropic stencils and the lagged velocity as constants.
template <int NC, int ST, bool SPEC, bool DIAG, typename AT, typename PL>
__device__ __forceinline__ void pack_tile(const AT& A, const PL& P, PackSmem<NC, 8>& S, float* pv_s, int x0, int y0,
                                          int row, int col, int cols) {
    constexpr int TY = 8, NT = kTX * TY;
    const MixConstT<float>& m = A.mixf;
    const int nx = A.nx, ny = A.ny, nxy = nx * ny;
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * kTX + tx;
    const int x = x0 + tx, y = y0 + ty;
    const bool valid = x < nx && y < ny;
    const int eos = SPEC ? 0 : -1, stencil = SPEC ? 0 : A.stencil;
    const bool lagged = SPEC ? true : A.lagged != 0;
    if constexpr (DIAG) diag_prefetch<NC, float, TY>(A, pv_s, tx, ty, x, y);
    if (lagged && valid) {
        const float* Fin = static_cast<const float*>(A.Fin);
        const int node = y * nx + x;
        cp_async_elem(&S.Fl[0][ty][tx], Fin + node);
        cp_async_elem(&S.Fl[1][ty][tx], Fin + (size_t)nxy + node);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");

    Comps<NC> g[9], r;
    float jx, jy;
    // phase 1 (steps 1-5), as phase1_global: one owned node and at most one ring node per thread
    auto phase1 = [&](auto inner_c) {
        constexpr bool inner = decltype(inner_c)::value;
        constexpr int RING = 4 * (kTX + 4) + 4 * TY;
        static_assert(RING <= NT, "one ring node per thread");
        const bool has_ring = tid < RING;
        int bx = 0, by = 0;
        Comps<NC> rrt;
        auto pull_ring = [&]() {
            ring_position<TY>(tid, bx, by);
            const int wx = inner ? x0 - 2 + bx : wrap(x0 - 2 + bx, nx);
            const int wy = inner ? y0 - 2 + by : wrap(y0 - 2 + by, ny);
            Comps<NC> h[9], rr;
            pack_pull<NC, ST>(P, inner, wx, wy, nx, ny, h);
            pack_rho<NC>(m, h, rr, rrt);
        };
        auto put_ring = [&]() {
            each_group<NC>([&](auto of) { tile_row(S.rt, of, by)[bx] = of(rrt); });
            if (bx >= 1 && bx <= kTX + 2 && by >= 1 && by <= TY + 2) {
                Comps<NC> lnf;
                node_lnf_comps<NC>(m, rrt, lnf, eos);
                each_group<NC>([&](auto of) { tile_row(S.lf, of, by - 1)[bx - 1] = of(lnf); });
            }
        };
        if (has_ring) pull_ring();
        pack_pull<NC, ST>(P, inner, inner ? x : wrap(x, nx), inner ? y : wrap(y, ny), nx, ny, g);
        if (has_ring) put_ring();
        Comps<NC> rt, lnf;
        pack_rho<NC>(m, g, r, rt);
        each_group<NC>([&](auto of) {
            float2 h[9], jxi, jyi;
#pragma unroll
            for (int a = 0; a < 9; ++a) h[a] = of(g[a]);
            moment_j(h, true, jxi, jyi);
#pragma unroll
            for (int l = 0; l < 2; ++l) {
                jx = 2 * of.k + l == 0 ? lane(jxi, l) : vadd(jx, lane(jxi, l));
                jy = 2 * of.k + l == 0 ? lane(jyi, l) : vadd(jy, lane(jyi, l));
            }
            tile_row(S.rt, of, ty + 2)[tx + 2] = of(rt);
        });
        const float beta = node_lnf_comps<NC>(m, rt, lnf, eos);
        each_group<NC>([&](auto of) { tile_row(S.lf, of, ty + 1)[tx + 1] = of(lnf); });
        // the domain check; a sum of the ln f_i is finite only if each is
        float lo = comp(rt, 0), ls = comp(lnf, 0);
#pragma unroll
        for (int i = 1; i < NC; ++i) {
            lo = fminf(lo, comp(rt, i));
            ls = vadd(ls, comp(lnf, i));
        }
        if (!(beta < 1.f && lo > 0.f && fabsf(ls) < INFINITY) && valid && checked_row(A, y)) {
            float rr[NC], ll[NC];
#pragma unroll
            for (int i = 0; i < NC; ++i) {
                rr[i] = comp(rt, i);
                ll[i] = comp(lnf, i);
            }
            domain_check<NC, float>(A, rr, ll, beta, x, 0, y, 1u);
        }
    };
    // no periodic wrap anywhere in this block's reach (tile + 2 halo + 1 pull)
    if (x0 >= 3 && x0 + kTX + 3 <= nx && y0 >= 3 && y0 + TY + 3 <= ny) phase1(std::true_type());
    else phase1(std::false_type());
    __syncthreads();
    // phase 2 (step 6): whole warps on whole rows, the last warp also the two edge columns
    for (int cy = ty; cy < TY + 2; cy += TY) pack_phi<NC, TY>(m, S, stencil, tx, cy);
    if (ty == TY - 1)
        for (int e = tx; e < 2 * (TY + 2); e += kTX) pack_phi<NC, TY>(m, S, stencil, kTX + (e & 1), e >> 1);
    __syncthreads();
    // phase 3 (steps 7-9), as phase3_core
    if (valid) {
        const int node = y * nx + x;
        float rho_t = comp(r, 0);
#pragma unroll
        for (int i = 1; i < NC; ++i) rho_t = vadd(rho_t, comp(r, i));
        const float inv_rho = vrcp(rho_t);
        float Ftx = 0.f, Fty = 0.f, ux = 0.f, uy = 0.f;
        Comps<NC> Fx, Fy, grx, gry;
        auto force = [&](auto of) {
            float2 px, py, rx, ry;
            grad_tile(tile_row(S.G, of, ty + 2), tile_row(S.G, of, ty + 1), tile_row(S.G, of, ty), tx + 1, stencil, px, py);
            grad_tile(tile_row(S.rt, of, ty + 3), tile_row(S.rt, of, ty + 2), tile_row(S.rt, of, ty + 1), tx + 2, stencil, rx,
                      ry);
            const float2 rti = tile_row(S.rt, of, ty + 2)[tx + 2];
            of(grx) = vmul(rx, of.of(m.M));
            of(gry) = vmul(ry, of.of(m.M));
            of(Fx) = vmul(rti, px);
            of(Fy) = vmul(rti, py);
#pragma unroll
            for (int l = 0; l < 2; ++l) {
                Ftx = 2 * of.k + l == 0 ? lane(of(Fx), l) : vadd(Ftx, lane(of(Fx), l));
                Fty = 2 * of.k + l == 0 ? lane(of(Fy), l) : vadd(Fty, lane(of(Fy), l));
            }
        };
        auto collide = [&](auto of) {
            float2 h[9];
#pragma unroll
            for (int a = 0; a < 9; ++a) h[a] = of(g[a]);
            collide_node<false, float2, float>(m, h, of(r), vbc<float2>(ux), vbc<float2>(uy), of(Fx), of(Fy), of(grx), of(gry),
                                               [&](int a, float2 v) {
#pragma unroll
                                                   for (int l = 0; l < 2; ++l)
                                                       store_gp<ST>(P, 2 * of.k + l, a, node, lane(v, l));
                                               });
        };
        if (lagged) {
            asm volatile("cp.async.wait_all;\n" ::: "memory");
            ux = vmul(vfma(0.5f, S.Fl[0][ty][tx], jx), inv_rho);
            uy = vmul(vfma(0.5f, S.Fl[1][ty][tx], jy), inv_rho);
            each_group<NC>([&](auto of) {
                force(of);
                collide(of);
            });
        } else {
            each_group<NC>(force);
            ux = vmul(vfma(0.5f, Ftx, jx), inv_rho);
            uy = vmul(vfma(0.5f, Fty, jy), inv_rho);
            each_group<NC>(collide);
        }
        float* Fout = static_cast<float*>(A.Fout);
        Fout[node] = Ftx;
        Fout[(size_t)nxy + node] = Fty;
    }
    if constexpr (DIAG) {
        if (A.diag_partial != nullptr) {  // uniform: diagnostics of the state this step read
            float rr[NC];
#pragma unroll
            for (int i = 0; i < NC; ++i) rr[i] = comp(r, i);
            diag_tile<NC, float, TY>(A, rr, pv_s, tx, ty, x, y, y0, row, col, cols);
        }
    }
}
template <int NC, int ST, bool SPEC, int MINB>
__global__ void __launch_bounds__(kTX * 8, MINB) pack_step(const __grid_constant__ StepArgs A,
                                                          const __grid_constant__ Planes P) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_pack[];
    pack_tile<NC, ST, SPEC, true>(A, P, *reinterpret_cast<PackSmem<NC, 8>*>(smem_pack),
                                  reinterpret_cast<float*>(smem_pack + sizeof(PackSmem<NC, 8>)), blockIdx.x * kTX,
                                  blockIdx.y * 8, blockIdx.y, blockIdx.x, gridDim.x);
}
template <int NC>
constexpr size_t pack_smem_bytes() {
    return sizeof(PackSmem<NC, 8>) + (size_t)NC * 8 * kTX * sizeof(float);
}

}  // namespace fmlbm
