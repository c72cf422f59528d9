// The marching step: one full time step of the lattice (as fused_step) without a halo in y.
//
// A warp owns a strip of columns and a chunk of rows and marches over the rows.  At each row it
// pulls the 9N values of the row's nodes (step 9 of the previous step), sums them to the densities
// and ln f (steps 1-5), and, one and two rows behind, completes Phi (step 6) and the collision
// (steps 7-9): the three rows a stencil reads are rolling registers of the lane that owns the
// column, the neighbours in x come from the adjacent lanes by shuffles.  The pulled values wait in
// shared memory for the two rows between their sums and their collision (each lane reads back its
// own values, so there is no barrier; only they are parked, the sums are formed again: with the row
// sums and gradients beside them, 4096^2 ternary FP32 took 803 us instead of 760, as what a block
// parks is taken from the L1), and the loads of the next row are issued as soon as the row's values
// are parked, in flight during the row's arithmetic.  Two components share a packed value
// (fmlbm_comps.cuh).
//
// The tile step is bound by its blocks' phases: every block loads, then computes (6,000 of 14,700
// cycles of a block pass until its loads have come), its instructions (816 per node, binary FP32)
// are half halo work, and its shared tiles and halo pulls take 71 % of the L1 data pipe.  Here the
// loads stay in flight, a node takes 513 instructions, and 40 % of the L1 data pipe is used; what
// bounds it is the latency of the loads that 16 warps (12 with three components) keep in flight.  The
// first and last two columns of a warp are halo (28 of 32 owned), a chunk of H rows pulls H + 4 and
// evaluates ln f on H + 2.  Deeper prefetch (two rows), parking in registers (168 registers, 31.3 us
// on the 1024^2 binary), pulling twice instead of parking (38.5), 20 warps per multiprocessor (49)
// and copies by the bulk engine (7 cycles per 144-byte row) were all slower.
//
// Every operation is that of the tile kernels on the same operands (the row sums h(x+1) + h(x-1)
// and differences of the stencils are formed once per row and reused by the three rows that read
// them), so the results are bit-identical to fused_step.
#pragma once

#include "fmlbm_comps.cuh"

namespace fmlbm {

constexpr int kMarchCols = 28;  // columns a strip owns

// Where the marching step is the faster one (GB300, us per step, packed or tile step -> marching):
//   two components   768^2 FP32 19.6 -> 18.2, 1024^2 37.0 -> 31.0, 2048^2 132 -> 130;
//                    FP16 768^2 17.1 -> 16.8, 1024^2 29.9 -> 28.7, 2048^2 111 -> 104, 4096^2 433 -> 417
//   three components 768^2 FP32 33.3 -> 26.1, 1024^2 55.4 -> 50.0, 2048^2 201 -> 195, 4096^2 795 -> 760;
//                    BF16 768^2 26.1 -> 22.9, 1024^2 44.9 -> 38.1, 2048^2 165 -> 157, 4096^2 657 -> 619
// Below 2^19 nodes a chunk has so few rows that its four halo rows outweigh the rest (512^2 FP32
// 9.2 -> 9.8).
constexpr size_t kMarchNodes = 1 << 19;
// States up to this size stay in the 129 MB L2 from the step that writes them to the step that
// reads them; their loads then go without a place in L1, whose turnover cost more than its hits
// gave (1024^2 binary FP32 35.9 -> 31.0 us, 1280^2 FP16 43.7 -> 40.5).  From DRAM the sector-wise
// requests are slower (2048^2 FP32 130 -> 157).
constexpr size_t kMarchL2Bytes = 125000000;

template <int NC, int ST>
inline size_t march_state_bytes(const StepArgs& A) {  // distributions and stored force a step reads
    return (size_t)A.nx * A.ny * (ST == ST_F32 ? NC * 36 + 8 : NC * 20 + 8);
}
// Nor where the last strip is mostly empty: 64 columns take three strips (64 x 9000 ternary FP16 29.0 ->
// 29.9 us, binary FP32 22.8 -> 22.4); a quarter more columns than the lattice has is the limit.
inline bool march_applies(const StepArgs& A) {
    const long long cols = (A.nx + kMarchCols - 1) / kMarchCols * kMarchCols;
    return (size_t)A.nx * A.ny >= kMarchNodes && 4 * cols <= 5LL * A.nx;
}
// Rows per chunk: all warps resident at once (one wave of `capacity` warps) while that keeps a
// chunk below 96 rows; otherwise as many waves as bring it there (4096^2 BF16 binary, 256 rows in
// one wave 529 us, 125 rows in two 416 us).
inline int march_chunk_rows(int ny, int strips, int capacity) {
    const int per_wave = capacity / strips > 0 ? capacity / strips : 1;
    const int waves = (ny + 96 * per_wave - 1) / (96 * per_wave);
    const int chunks = per_wave * waves < ny ? per_wave * waves : ny;
    return (ny + chunks - 1) / chunks;
}

constexpr int kMarchWarps = 4;  // warps (neighbouring strips) per block
// Blocks per multiprocessor, and the warps of one wave.
constexpr int march_blocks(int nc) { return nc == 2 ? 4 : 3; }
inline int march_capacity(int nc, int sms) { return sms * march_blocks(nc) * kMarchWarps; }
// The share of its waves' row iterations that a march spends on the rows it owns: the rest are the
// four halo rows of a chunk and empty places in the last wave.
inline double march_fill(int nc, int nx, int ny, int sms) {
    const int strips = (nx + kMarchCols - 1) / kMarchCols, capacity = march_capacity(nc, sms);
    const int chunk = march_chunk_rows(ny, strips, capacity);
    const long long warps = (long long)strips * ((ny + chunk - 1) / chunk);
    const long long waves = (warps + capacity - 1) / capacity;
    return (double)strips * ny / ((double)waves * capacity * (chunk + 4));
}

// Words a lane parks per row: the pulled values (their sums are formed again at the collision:
// what a block parks is taken from the L1, whose size the step feels).
template <int NC> constexpr int kParkWords = 9 * NC;
template <int NC>
constexpr size_t march_smem_bytes() {
    return (size_t)kMarchWarps * 3 * kParkWords<NC> * 32 * sizeof(float);
}

// East and west neighbours of a value held by every lane (lane l of the warp: column l).  The
// outer neighbours of the strip's first and last column are not held: what those lanes get is
// unused.
__device__ __forceinline__ void lane_ew(float v, float& e, float& w) {
    e = __shfl_down_sync(0xffffffffu, v, 1);
    w = __shfl_up_sync(0xffffffffu, v, 1);
}
__device__ __forceinline__ void lane_ew(float2 v, float2& e, float2& w) {
    lane_ew(v.x, e.x, w.x);
    lane_ew(v.y, e.y, w.y);
}

// Finite differences at the middle one of three rows, from the rows' values c, their x-sums s =
// h(x+1) + h(x-1) and x-differences d = h(x+1) - h(x-1) (n: the row above, s: below): the
// operations of lap_at and grad_at.
template <typename V>
__device__ __forceinline__ V lap_rows(V cn, V cc, V cs, V sn, V sc, V ss, int stencil) {
    using E = LaneE<V>;
    const V ax = vadd(sc, vadd(cn, cs));
    const V m4 = vbc<V>(E(-4));
    if (stencil == 1) return vfma(m4, cc, ax);
    const V dg = vadd(sn, ss);
    return vfma(vfma(m4, cc, ax), vbc<V>(E(2.0 / 3.0)), vmul(vfma(m4, cc, dg), vbc<V>(E(1.0 / 6.0))));
}
template <typename V>
__device__ __forceinline__ void grad_rows(V cn, V cs, V sn, V ss, V dn, V dc, V ds, int stencil, V& gx, V& gy) {
    using E = LaneE<V>;
    if (stencil == 1) {
        gx = vmul(vbc<V>(E(0.5)), dc);
        gy = vmul(vbc<V>(E(0.5)), vsub(cn, cs));
    } else {
        const V third = vbc<V>(E(1.0 / 3.0)), twelfth = vbc<V>(E(1.0 / 12.0));
        gx = vfma(dc, third, vmul(vadd(dn, ds), twelfth));
        gy = vfma(vsub(cn, cs), third, vmul(vsub(sn, ss), twelfth));
    }
}

// A lane's W words to and from a slot: 16-byte vectors, then an 8-byte and a 4-byte remainder.
template <int W>
__device__ __forceinline__ void park_put(float* slot, int lane, const float (&w)[W]) {
#pragma unroll
    for (int q = 0; q < W / 4; ++q)
        reinterpret_cast<float4*>(slot)[q * 32 + lane] = make_float4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
    float* rest = slot + (W / 4) * 128;
    if constexpr (W % 4 >= 2) reinterpret_cast<float2*>(rest)[lane] = make_float2(w[W / 4 * 4], w[W / 4 * 4 + 1]);
    if constexpr (W % 2 == 1) rest[(W % 4 == 3 ? 64 : 0) + lane] = w[W - 1];
}
template <int W>
__device__ __forceinline__ void park_get(const float* slot, int lane, float (&w)[W]) {
#pragma unroll
    for (int q = 0; q < W / 4; ++q) {
        const float4 v = reinterpret_cast<const float4*>(slot)[q * 32 + lane];
        w[4 * q] = v.x; w[4 * q + 1] = v.y; w[4 * q + 2] = v.z; w[4 * q + 3] = v.w;
    }
    const float* rest = slot + (W / 4) * 128;
    if constexpr (W % 4 >= 2) {
        const float2 v = reinterpret_cast<const float2*>(rest)[lane];
        w[W / 4 * 4] = v.x; w[W / 4 * 4 + 1] = v.y;
    }
    if constexpr (W % 2 == 1) w[W - 1] = rest[(W % 4 == 3 ? 64 : 0) + lane];
}

// The pulled values as loaded: 16-bit values are widened where they are used, so that nothing
// waits for them at the load.  Volatile, so that the loads stay where they are issued, a row ahead
// of their use (the compiler sank them to their use: 4096^2 ternary BF16 990 us against 678).
// NOALLOC: without a place in L1.
template <bool NOALLOC>
__device__ __forceinline__ float ld_ahead(const float* p) {
    float v;
    if constexpr (NOALLOC) asm volatile("ld.global.nc.L1::no_allocate.f32 %0, [%1];" : "=f"(v) : "l"(p));
    else asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
template <bool NOALLOC, typename E>
__device__ __forceinline__ unsigned short ld_ahead16(const E* p) {
    unsigned short v;
    if constexpr (NOALLOC) asm volatile("ld.global.nc.L1::no_allocate.u16 %0, [%1];" : "=h"(v) : "l"(p));
    else asm volatile("ld.global.nc.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return v;
}
template <int ST> struct MarchRaw { using T = unsigned short; };
template <> struct MarchRaw<ST_F32> { using T = float; };

// One strip x chunk: columns x0 .. x0 + 27 (those below nx), rows y0 .. y0 + rows - 1, by one
// warp.  slots: the warp's three parking slots.
template <int NC, int ST, bool SPEC, bool NOALLOC>
__device__ __forceinline__ void march_chunk(const StepArgs& A, const Planes& P, const MixConstT<float>& m, float* slots,
                                            int x0, int y0, int rows) {
    using Elem = typename StoreTraits<ST>::Elem;
    using Raw = typename MarchRaw<ST>::T;
    constexpr bool F32 = ST == ST_F32;
    const int lane = threadIdx.x & 31;
    const int nx = A.nx, ny = A.ny, nxy = nx * ny;
    const int eos = SPEC ? 0 : -1, stencil = SPEC ? 0 : A.stencil;
    const bool lagged = SPEC ? true : A.lagged != 0;
    // the lane's column (wrapped), its x-neighbours, and whether the strip owns it
    const int x = x0 - 2 + lane;
    const int xc = wrap(x, nx);
    const int xm = xc == 0 ? nx - 1 : xc - 1, xp = xc == nx - 1 ? 0 : xc + 1;
    const bool own = lane >= 2 && lane < 30 && x < nx;
    // rows (uniform over the warp): the row to pull next, the ones below and above it
    const int yb = wrap(y0 - 2, ny);
    int rc = yb * nx, rm = (yb == 0 ? ny - 1 : yb - 1) * nx, rp = (yb == ny - 1 ? 0 : yb + 1) * nx;
    Raw g[NC][9];
    float g0[NC];  // 16-bit forms: the float plane a = 0
    auto load_row = [&]() {
#pragma unroll
        for (int a = 0; a < 9; ++a) {
            const int node = (ey(a) == 1 ? rm : (ey(a) == -1 ? rp : rc)) + (ex(a) == 1 ? xm : (ex(a) == -1 ? xp : xc));
#pragma unroll
            for (int i = 0; i < NC; ++i) {
                if constexpr (F32) g[i][a] = ld_ahead<NOALLOC>(static_cast<const float*>(P.in[i * 9 + a]) + node);
                else if (a == 0) g0[i] = ld_ahead<NOALLOC>(P.g0in[i] + node);
                else g[i][a] = ld_ahead16<NOALLOC>(static_cast<const Elem*>(P.in[i * 8 + a - 1]) + node);
            }
        }
        rm = rc;
        rc = rp;
        rp = rp + nx == nxy ? 0 : rp + nx;
    };
    auto pulled = [&](int i, int a) -> float {
        if constexpr (F32) return g[i][a];
        else if (a == 0) return g0[i];
        else if constexpr (std::is_same<Elem, __half>::value) return to_real(__ushort_as_half(g[i][a]));
        else return to_real(__ushort_as_bfloat16(g[i][a]));
    };
    const float* Fin = static_cast<const float*>(A.Fin);
    float* Fout = static_cast<float*>(A.Fout);
    float* snap = static_cast<float*>(A.rho_snap);
    load_row();
    // rolling rows, indexed by the iteration mod 3: rho~ with its x-sums and x-differences, Phi
    // likewise (one row behind), ln f of the last row, grad rho~ of the row to collide next
    Comps<NC> rt[3], rs[3], rd[3], ph[3], ps[3], pd[3], lf = {}, gx = {}, gy = {};
    const int T = rows + 4;
    auto row_step = [&](auto kc, int it) {
        constexpr int K = decltype(kc)::value, K1 = (K + 2) % 3, K2 = (K + 1) % 3;  // rows y, y - 1, y - 2
        // row y = y0 - 2 + it: densities and rho~ (steps 1-2); park the pulled values
        {
            float pk[kParkWords<NC>];
            each_group<NC>([&](auto of) {
                using V = typename decltype(of)::V;
                constexpr bool PAIR = std::is_same<V, float2>::value;
                int i0 = NC - 1;
                if constexpr (PAIR) i0 = 2 * of.k;
                V h[9];
#pragma unroll
                for (int a = 0; a < 9; ++a) {
                    if constexpr (PAIR) h[a] = make_float2(pulled(i0, a), pulled(i0 + 1, a));
                    else h[a] = pulled(i0, a);
                    // direction by direction within the group
#pragma unroll
                    for (int l = 0; l < (PAIR ? 2 : 1); ++l) pk[9 * i0 + (PAIR ? 2 * a + l : a)] = fmlbm::lane(h[a], l);
                }
                const V r = sum9(h);
                of(rt[K]) = vmul(r, of.of(m.invM));
                if (snap != nullptr && it >= 2 && it < rows + 2 && own) {
#pragma unroll
                    for (int l = 0; l < (PAIR ? 2 : 1); ++l)
                        snap[(size_t)(i0 + l) * nxy + (y0 + it - 2) * nx + xc] = fmlbm::lane(r, l);
                }
            });
            park_put(slots + K * kParkWords<NC> * 32, lane, pk);
        }
        // the next row's loads go out now, and the force of the row this iteration collides
        if (it + 1 < T) load_row();
        float Fpx = 0.f, Fpy = 0.f;
        if (lagged && it >= 4) {
            const int node = (y0 + it - 4) * nx + xc;
            Fpx = ld_ahead<NOALLOC>(Fin + node);
            Fpy = ld_ahead<NOALLOC>(Fin + nxy + node);
        }
        // ln f (steps 2-5) on the rows Phi needs
        Comps<NC> lnew = {};
        if (it >= 1 && it <= rows + 2) {
            const float beta = node_lnf_comps<NC>(m, rt[K], lnew, eos);
            // the domain check; a sum of the ln f_i is finite only if each is
            float lo = comp(rt[K], 0), ls = comp(lnew, 0);
#pragma unroll
            for (int i = 1; i < NC; ++i) {
                lo = fminf(lo, comp(rt[K], i));
                ls = vadd(ls, comp(lnew, i));
            }
            if (!(beta < 1.f && lo > 0.f && fabsf(ls) < INFINITY) && own && it >= 2 && it < rows + 2 &&
                checked_row(A, y0 + it - 2)) {
                float rr[NC], ll[NC];
#pragma unroll
                for (int i = 0; i < NC; ++i) {
                    rr[i] = comp(rt[K], i);
                    ll[i] = comp(lnew, i);
                }
                domain_check<NC, float>(A, rr, ll, beta, x, 0, y0 + it - 2, 1u);
            }
        }
        each_group<NC>([&](auto of) {
            typename decltype(of)::V e, w;
            lane_ew(of(rt[K]), e, w);
            of(rs[K]) = vadd(e, w);
            of(rd[K]) = vsub(e, w);
        });
        if (it >= 2) {
            // Phi of row y - 1 (step 6)
            Comps<NC> L;
            each_group<NC>([&](auto of) {
                using V = typename decltype(of)::V;
                of(L) = lap_rows<V>(of(rt[K]), of(rt[K1]), of(rt[K2]), of(rs[K]), of(rs[K1]), of(rs[K2]), stencil);
            });
            each_group<NC>([&](auto of) {
                using V = typename decltype(of)::V;
                V Gi = vmul(of.col(m.kap, 0), vbc<V>(comp(L, 0)));
#pragma unroll
                for (int j = 1; j < NC; ++j) Gi = vfma(of.col(m.kap, j), vbc<V>(comp(L, j)), Gi);
                of(ph[K]) = vfma(vbc<V>(-m.RT), of(lf), Gi);
                V e, w;
                lane_ew(of(ph[K]), e, w);
                of(ps[K]) = vadd(e, w);
                of(pd[K]) = vsub(e, w);
            });
            if (it >= 4 && own) {
                // collision of row y - 2 (steps 7-9): the operations of phase3_core
                float pk[kParkWords<NC>];
                park_get(slots + K2 * kParkWords<NC> * 32, lane, pk);
                const int node = (y0 + it - 4) * nx + xc;
                auto group_h = [&](auto of, auto (&h)[9]) {
                    constexpr bool PAIR = std::is_same<typename decltype(of)::V, float2>::value;
                    int i0 = NC - 1;
                    if constexpr (PAIR) i0 = 2 * of.k;
#pragma unroll
                    for (int a = 0; a < 9; ++a) {
                        if constexpr (PAIR) h[a] = make_float2(pk[9 * i0 + 2 * a], pk[9 * i0 + 2 * a + 1]);
                        else h[a] = pk[9 * i0 + a];
                    }
                };
                // densities and first moment (step 1)
                Comps<NC> rho;
                float jx = 0.f, jy = 0.f, rho_t = 0.f;
                each_group<NC>([&](auto of) {
                    using V = typename decltype(of)::V;
                    constexpr bool PAIR = std::is_same<V, float2>::value;
                    int i0 = NC - 1;
                    if constexpr (PAIR) i0 = 2 * of.k;
                    V h[9], jxi, jyi;
                    group_h(of, h);
                    of(rho) = sum9(h);
                    moment_j(h, true, jxi, jyi);
#pragma unroll
                    for (int l = 0; l < (PAIR ? 2 : 1); ++l) {
                        jx = i0 + l == 0 ? fmlbm::lane(jxi, l) : vadd(jx, fmlbm::lane(jxi, l));
                        jy = i0 + l == 0 ? fmlbm::lane(jyi, l) : vadd(jy, fmlbm::lane(jyi, l));
                        rho_t = i0 + l == 0 ? fmlbm::lane(of(rho), l) : vadd(rho_t, fmlbm::lane(of(rho), l));
                    }
                });
                const float inv_rho = vrcp(rho_t);
                float Ftx = 0.f, Fty = 0.f, ux = 0.f, uy = 0.f;
                Comps<NC> Fx, Fy;
                auto force = [&](auto of) {
                    using V = typename decltype(of)::V;
                    constexpr bool PAIR = std::is_same<V, float2>::value;
                    int i0 = NC - 1;
                    if constexpr (PAIR) i0 = 2 * of.k;
                    V px, py;
                    grad_rows<V>(of(ph[K]), of(ph[K2]), of(ps[K]), of(ps[K2]), of(pd[K]), of(pd[K1]), of(pd[K2]), stencil,
                                 px, py);
                    const V rti = of(rt[K2]);
                    of(Fx) = vmul(rti, px);
                    of(Fy) = vmul(rti, py);
#pragma unroll
                    for (int l = 0; l < (PAIR ? 2 : 1); ++l) {
                        Ftx = i0 + l == 0 ? fmlbm::lane(of(Fx), l) : vadd(Ftx, fmlbm::lane(of(Fx), l));
                        Fty = i0 + l == 0 ? fmlbm::lane(of(Fy), l) : vadd(Fty, fmlbm::lane(of(Fy), l));
                    }
                };
                auto collide = [&](auto of) {
                    using V = typename decltype(of)::V;
                    constexpr bool PAIR = std::is_same<V, float2>::value;
                    int i0 = NC - 1;
                    if constexpr (PAIR) i0 = 2 * of.k;
                    V h[9];
                    group_h(of, h);
                    const V grx = vmul(of(gx), of.of(m.M)), gry = vmul(of(gy), of.of(m.M));
                    const V u_x = vbc<V>(ux), u_y = vbc<V>(uy);
                    collide_node<false, V, float>(m, h, of(rho), u_x, u_y, of(Fx), of(Fy), grx, gry, [&](int a, V v) {
#pragma unroll
                        for (int l = 0; l < (PAIR ? 2 : 1); ++l) store_gp<ST>(P, i0 + l, a, node, fmlbm::lane(v, l));
                    });
                };
                if (lagged) {
                    ux = vmul(vfma(0.5f, Fpx, jx), inv_rho);
                    uy = vmul(vfma(0.5f, Fpy, jy), inv_rho);
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
                Fout[node] = Ftx;
                Fout[nxy + node] = Fty;
            }
            // grad rho~ of row y - 1, for its collision in the next iteration
            each_group<NC>([&](auto of) {
                using V = typename decltype(of)::V;
                grad_rows<V>(of(rt[K]), of(rt[K2]), of(rs[K]), of(rs[K2]), of(rd[K]), of(rd[K1]), of(rd[K2]), stencil, of(gx),
                             of(gy));
            });
        }
        lf = lnew;
    };
    for (int it = 0; it < T; it += 3) {
        row_step(std::integral_constant<int, 0>(), it);
        if (it + 1 < T) row_step(std::integral_constant<int, 1>(), it + 1);
        if (it + 2 < T) row_step(std::integral_constant<int, 2>(), it + 2);
    }
}

// The warp index is broadcast from lane 0 so that the rows and the loop are uniform for the
// compiler.
template <int NC, int ST, bool SPEC, bool NOALLOC, int MINB>
__global__ void __launch_bounds__(32 * kMarchWarps, MINB)
    march_step(const __grid_constant__ StepArgs A, const __grid_constant__ Planes P, int strips, int chunk) {
    extern __shared__ __align__(16) float smem_march[];
    pdl_wait();
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
    const int w = blockIdx.x * kMarchWarps + warp;
    const int cy = w / strips, y0 = cy * chunk;
    if (y0 >= A.ny) return;
    const int x0 = (w - cy * strips) * kMarchCols;
    march_chunk<NC, ST, SPEC, NOALLOC>(A, P, A.mixf, smem_march + warp * 3 * kParkWords<NC> * 32, x0, y0, min(chunk, A.ny - y0));
}

}  // namespace fmlbm
