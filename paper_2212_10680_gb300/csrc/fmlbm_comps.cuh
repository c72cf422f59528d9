// Component-packed values: the float arithmetic of components 2k and 2k + 1 of a node runs as packed
// two-lane instructions (add.f32x2 and the like: one issue slot for both); an odd last component
// stays scalar.  A pair of components, unlike a pair of nodes (fmlbm_pair.cuh), costs no registers.
// Every operation is that of the one-node kernels on the same operands: same bits.
#pragma once

#include "fmlbm_kernels.cuh"

namespace fmlbm {

// One value per component: pairs of components in float2, an odd last one in a float.
template <int NC>
struct Comps {
    float2 p[NC >= 2 ? NC / 2 : 1];
    float s;
};
struct PairOf {  // components 2k, 2k + 1
    using V = float2;
    int k;
    template <int NC> __device__ __forceinline__ float2& operator()(Comps<NC>& c) const { return c.p[k]; }
    template <int NC> __device__ __forceinline__ const float2& operator()(const Comps<NC>& c) const { return c.p[k]; }
    __device__ __forceinline__ float2 of(const float* v) const { return make_float2(v[2 * k], v[2 * k + 1]); }
    // column j of a matrix with row stride kMaxC
    __device__ __forceinline__ float2 col(const float* v, int j) const {
        return make_float2(v[2 * k * kMaxC + j], v[(2 * k + 1) * kMaxC + j]);
    }
};
template <int I>
struct LastOf {  // component I alone
    using V = float;
    template <int NC> __device__ __forceinline__ float& operator()(Comps<NC>& c) const { return c.s; }
    template <int NC> __device__ __forceinline__ const float& operator()(const Comps<NC>& c) const { return c.s; }
    __device__ __forceinline__ float of(const float* v) const { return v[I]; }
    __device__ __forceinline__ float col(const float* v, int j) const { return v[I * kMaxC + j]; }
};
template <int NC, typename F>
__device__ __forceinline__ void each_group(F&& f) {
#pragma unroll
    for (int k = 0; k < NC / 2; ++k) f(PairOf{k});
    if constexpr (NC & 1) f(LastOf<NC - 1>{});
}
template <int NC>
__device__ __forceinline__ float comp(const Comps<NC>& c, int i) {
    if ((NC & 1) && i == NC - 1) return c.s;
    return (i & 1) ? c.p[i / 2].y : c.p[i / 2].x;
}
template <int NC>
__device__ __forceinline__ void set_comp(Comps<NC>& c, int i, float v) {
    if ((NC & 1) && i == NC - 1) c.s = v;
    else if (i & 1) c.p[i / 2].y = v;
    else c.p[i / 2].x = v;
}

// ln f of a node (node_lnf, the same operations) with the per-component parts packed.
template <int NC>
__device__ __forceinline__ float node_lnf_comps(const MixConstT<float>& m, const Comps<NC>& rt, Comps<NC>& lnf,
                                                int eos) {
    const int kind = eos >= 0 ? eos : m.eos;
    float rtot = comp(rt, 0), beta = vmul(m.b[0], comp(rt, 0));
#pragma unroll
    for (int i = 1; i < NC; ++i) {
        rtot = vadd(rtot, comp(rt, i));
        beta = vfma(m.b[i], comp(rt, i), beta);
    }
    const float inv = vrcp(rtot);
    Comps<NC> S;
    each_group<NC>([&](auto of) {
        using V = typename decltype(of)::V;
        V s = vmul(of.col(m.aij, 0), vbc<V>(comp(rt, 0)));
#pragma unroll
        for (int j = 1; j < NC; ++j) s = vfma(of.col(m.aij, j), vbc<V>(comp(rt, j)), s);
        of(S) = s;
    });
    float aam_rt2 = vmul(comp(rt, 0), comp(S, 0));
#pragma unroll
    for (int i = 1; i < NC; ++i) aam_rt2 = vfma(comp(rt, i), comp(S, i), aam_rt2);
    const float invomb = vrcp(vsub(1.f, beta));
    const float lead = vmul(m.RT, invomb);
    if (kind == 2) {
        const float rb1 = vmul(rtot, invomb), m2rt = -2.f * m.invRT;
        each_group<NC>([&](auto of) {
            using V = typename decltype(of)::V;
            of(lnf) = vfma(of(S), vbc<V>(m2rt), vfma(of.of(m.b), vbc<V>(rb1), vln(vmul(of(rt), vbc<V>(lead)))));
        });
        return beta;
    }
    const float att = vmul(vmul(aam_rt2, inv), m.invRT);
    float rep, lr, pref;
    if (kind == 0) {
        const float s2 = float(1.4142135623730950488);
        const float den = vfma(beta, vsub(2.f, beta), 1.f);
        rep = vfma(-att, vrcp(den), vmul(beta, invomb));
        lr = vln(vmul(vfma(1.f + s2, beta, 1.f), vrcp(vfma(1.f - s2, beta, 1.f))));
        pref = m.invRT * float(0.35355339059327376220);
    } else {
        rep = vfma(-att, vrcp(vadd(1.f, beta)), vmul(beta, invomb));
        lr = vlog1p(beta);
        pref = m.invRT;
    }
    const float rb = vmul(rtot, vrcp(beta));
    const float aam = vmul(vmul(aam_rt2, inv), inv);
    const float plr = vmul(vmul(pref, rb), lr);
    const float m2inv = vmul(-2.f, inv);
    each_group<NC>([&](auto of) {
        using V = typename decltype(of)::V;
        const V bi = vmul(of.of(m.b), vbc<V>(rb));
        const V t = vfma(vbc<V>(aam), bi, vmul(of(S), vbc<V>(m2inv)));
        of(lnf) = vfma(vbc<V>(plr), t, vfma(bi, vbc<V>(rep), vln(vmul(of(rt), vbc<V>(lead)))));
    });
    return beta;
}

}  // namespace fmlbm
