// The collisions of the plain steps on pairs of nodes (float2 lanes), with Blackwell's paired FP32
// instructions.  Every operation is an explicitly rounded one, so a kernel that takes several
// steps at once gives, bit for bit, what the one-step kernels give:
//   SCALAR_FORM: the grouping of step_node (lbm_kernels.cuh), including which products the
//     compiler contracts there (measured by comparing the bits): t = 3 cu + (4.5 cu) cu - 1.5 u.u,
//     feq = w (rho' + (1 + rho') t), f + omega (feq - f), as chains of fused multiply-adds;
//   PAIR_FORM: the grouping of step_pair (lbm_pair.cuh), that of plain coupled steps in FP16 storage.
#pragma once

#include "lbm_pair.cuh"

namespace mfc {

// A product that must not be contracted with the sum that takes it (the compiler contracts paired
// products and sums, but not these).
__device__ __forceinline__ float2 p_rounded_mul(float2 a, float2 b)
{
    return make_float2(__fmul_rn(a.x, b.x), __fmul_rn(a.y, b.y));
}

enum : int { SCALAR_FORM = 0, PAIR_FORM = 1 };

// u.u as the one-step kernels round it (which of the products are contracted differs between them):
//   CHAIN_01: fma(u1, u1, u0 u0); CHAIN_10: fma(u0, u0, u1 u1); SUM: u0 u0 + u1 u1 with both
//   products rounded.  In 3-D the third term is fma(u2, u2, .), or with SUM a rounded product too.
enum : int { UU_CHAIN_01 = 0, UU_CHAIN_10 = 1, UU_SUM = 2 };
template <int DIM, typename ST, bool COUPLED, int AQ, int SINK> struct UuForm {
    static constexpr bool f32 = std::is_same<ST, float>::value;
    static constexpr bool first_order_2d = DIM == 2 && AQ == 5 && SINK == SINK_LINEAR;
    // in the collision, and in the outlet values along the axis and along the diagonals
    static constexpr int collision = f32 && (!COUPLED || first_order_2d) ? UU_SUM : UU_CHAIN_01;
    static constexpr int outlet_axis = f32 && (!COUPLED || first_order_2d) ? UU_SUM : UU_CHAIN_10;
    static constexpr int outlet_diagonal = f32 && !COUPLED ? UU_SUM : UU_CHAIN_10;
};
// Batches (whose kernels choose the consumption at run time) take the reader form of the open boundaries
// for every storage type.
template <int DIM, typename ST, int AQ, int SINK> struct ReaderForm {
    static constexpr bool value = SINK == SINK_RUNTIME || ReaderBoundaries<DIM, ST, AQ>::step;
};
template <int DIM, int FORM> __device__ __forceinline__ float2 p_uu(const float2 (&u)[3])
{
    const float2 m0 = FORM == UU_SUM ? p_rounded_mul(u[0], u[0]) : p_mul(u[0], u[0]);
    const float2 m1 = FORM == UU_SUM ? p_rounded_mul(u[1], u[1]) : p_mul(u[1], u[1]);
    float2 r = FORM == UU_SUM ? p_add(m0, m1) : (FORM == UU_CHAIN_01 ? p_fma(u[1], u[1], m0) : p_fma(u[0], u[0], m1));
    if (DIM == 3) r = FORM == UU_SUM ? p_add(r, p_rounded_mul(u[2], u[2])) : p_fma(u[2], u[2], r);
    return r;
}
template <int DIM, int FORM> __device__ __forceinline__ float s_uu(float u0, float u1, float u2)
{
    const float m0 = __fmul_rn(u0, u0), m1 = __fmul_rn(u1, u1);
    float r = FORM == UU_SUM ? __fadd_rn(m0, m1) : (FORM == UU_CHAIN_01 ? __fmaf_rn(u1, u1, m0) : __fmaf_rn(u0, u0, m1));
    if (DIM == 3) r = FORM == UU_SUM ? __fadd_rn(r, __fmul_rn(u2, u2)) : __fmaf_rn(u2, u2, r);
    return r;
}

// The value a store of v keeps (see kept() in lbm_lattice.cuh).
__device__ __forceinline__ float2 p_kept(const float *, float2 v) { return v; }
__device__ __forceinline__ float2 p_kept(const __half *, float2 v) { return __half22float2(__float22half2_rn(v)); }

// c_i . u with the components added in axis order, up to the sign of the first of the pair (i,
// opposite): the caller takes i with the lower index and negates for the opposite (exact).
template <typename SET, int DIM> __device__ __forceinline__ float2 p_cu(int i, const float2 (&u)[3])
{
    float2 r = p_all(0.0f);
    bool any = false;
#pragma unroll
    for (int ax = 0; ax < DIM; ++ax) {
        const int c = SET::c(i, ax);
        if (c == 0) continue;
        if (!any) r = c > 0 ? u[ax] : p_mul(p_all(-1.0f), u[ax]);
        else r = c > 0 ? p_add(r, u[ax]) : p_sub(r, u[ax]);
        any = true;
    }
    return r;
}

// Flow moments (Eqs. 9-10) and BGK relaxation (Eqs. 4-5) of two nodes: d holds the gathered
// populations (deviations) and receives the post-collision ones as a store keeps them; u and rp
// (rho - 1) are the moments.
template <int DIM, typename ST, int FORM, int UU>
__device__ __forceinline__ void collide_flow(float2 (&d)[FlowSet<DIM>::Q], float omega, float2 (&u)[3], float2 &rp)
{
    using F = FlowSet<DIM>;
    const ST *tag = nullptr;
    rp = d[0];
#pragma unroll
    for (int i = 1; i < F::Q; ++i) rp = p_add(rp, d[i]);
    const float2 opr = p_add(p_all(1.0f), rp);
    const float2 inv = make_float2(recip(opr.x), recip(opr.y));
    float2 moved = p_all(0.0f);
    if constexpr (FORM == SCALAR_FORM) {
#pragma unroll
        for (int ax = 0; ax < DIM; ++ax) {
            float2 j = p_all(0.0f);
            bool any = false;
#pragma unroll
            for (int i = 1; i < F::Q; ++i) {
                const int c = F::c(i, ax);
                if (c == 0) continue;
                if (!any) j = c > 0 ? d[i] : p_mul(p_all(-1.0f), d[i]);
                else j = c > 0 ? p_add(j, d[i]) : p_sub(j, d[i]);
                any = true;
            }
            u[ax] = p_mul(j, inv);
        }
        const float2 uu = p_uu<DIM, UU>(u);
        const float2 om = p_all(-omega);
        float2 v[F::Q];
#pragma unroll
        for (int i = 1; i < F::Q; ++i) {
            const int o = F::opp(i);
            if (o < i) continue;  // taken with its opposite: c_o . u = -(c_i . u)
            const float2 cu = p_cu<F, DIM>(i, u);
            const float2 sq = p_mul(p_mul(p_all(4.5f), cu), cu);
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const int k = s ? o : i;
                const float2 t = p_fma(p_all(-1.5f), uu, p_fma(p_all(s ? -3.0f : 3.0f), cu, sq));
                const float2 nd = p_fma(p_all(-F::w(k)), p_fma(opr, t, rp), d[k]);  // f - feq
                v[k] = p_kept(tag, p_fma(om, nd, d[k]));
            }
        }
        moved = v[1];
        d[1] = v[1];
#pragma unroll
        for (int i = 2; i < F::Q; ++i) {
            moved = p_add(moved, v[i]);
            d[i] = v[i];
        }
    } else {
#pragma unroll
        for (int ax = 0; ax < DIM; ++ax)
            u[ax] = p_mul(p_sub(p_sum_where<F>(d, ax, 1), p_sum_where<F>(d, ax, -1)), inv);
        float2 uu = p_mul(u[0], u[0]);
#pragma unroll
        for (int ax = 1; ax < DIM; ++ax) uu = p_fma(u[ax], u[ax], uu);
        const float2 muu = p_mul(p_all(-1.5f), uu);
        const float2 om = p_all(omega);
        // w (1 + rho') and w rho' of the two moving weight classes (faces; diagonals or edges)
        constexpr int IE = DIM == 2 ? 5 : 7;
        const float2 wo_f = p_mul(p_all(F::w(1)), opr), wr_f = p_mul(p_all(F::w(1)), rp);
        const float2 wo_e = p_mul(p_all(F::w(IE)), opr), wr_e = p_mul(p_all(F::w(IE)), rp);
#pragma unroll
        for (int i = 1; i < F::Q; ++i) {
            float s;
            const float2 m = p_cdot<F, DIM>(i, u, s);
            // 3 cu + 9/2 cu^2 - 3/2 u.u = m (9/2 m + 3 s) - 3/2 u.u
            const float2 t = p_fma(m, p_fma(p_all(4.5f), m, p_all(3.0f * s)), muu);
            const float2 feq = i < IE ? p_fma(wo_f, t, wr_f) : p_fma(wo_e, t, wr_e);
            d[i] = p_kept(tag, p_fma(om, p_sub(feq, d[i]), d[i]));
            moved = i == 1 ? d[i] : p_add(moved, d[i]);
        }
    }
    d[0] = p_kept(tag, p_sub(rp, moved));
}

// Substrate moment (Eq. 13), relaxation (Eq. 12) and consumption of two nodes in the velocity u
// (already scaled).  sinks: whether either node may consume (its rate k0, k1 is 0 where it does
// not); without, the consumption is exactly zero and its terms are left out.
template <int DIM, typename ST, int AQ, int SINK, int FORM>
__device__ __forceinline__ void collide_ade(float2 (&e)[AdeSet<DIM, AQ>::Q], const float2 (&u)[3], float omega_c,
                                            float c_ref, float k_half, bool sinks, float k0, float k1)
{
    using A = AdeSet<DIM, AQ>;
    const ST *tag = nullptr;
    float2 cp = e[0];
#pragma unroll
    for (int i = 1; i < A::Q; ++i) cp = p_add(cp, e[i]);
    const float2 Cs = p_add(p_all(c_ref), cp);
    float2 sink = p_all(0.0f);
    if (sinks) {  // Eq. 16's substrate factor: k C, or k C K_s / (K_s + C)
        sink = p_mul(make_float2(k0, k1), Cs);
        if (SINK == SINK_MONOD || (SINK == SINK_RUNTIME && k_half > 0.0f)) {
            if (k0 != 0.0f) sink.x = sink.x * k_half * recip(k_half + Cs.x);
            if (k1 != 0.0f) sink.y = sink.y * k_half * recip(k_half + Cs.y);
        }
    }
    float2 moved = p_all(0.0f);
    if constexpr (FORM == SCALAR_FORM) {
        float2 uu = p_all(0.0f);
        if (A::quadratic) uu = p_fma(u[1], u[1], p_mul(u[0], u[0]));
        const float2 om = p_all(-omega_c);
        float2 v[A::Q];
#pragma unroll
        for (int i = 1; i < A::Q; ++i) {
            const int o = A::opp(i);
            if (o < i) continue;
            const float2 cu = p_cu<A, DIM>(i, u);
            const float2 sq = A::quadratic ? p_mul(p_mul(p_all(4.5f), cu), cu) : p_mul(cu, p_all(A::inv_cs2));
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const int k = s ? o : i;
                float2 X;
                if (A::quadratic) X = p_fma(Cs, p_fma(p_all(-1.5f), uu, p_fma(p_all(s ? -3.0f : 3.0f), cu, sq)), cp);
                else X = p_fma(s ? p_mul(p_all(-1.0f), Cs) : Cs, sq, cp);
                const float2 nd = p_fma(p_all(-A::w(k)), X, e[k]);
                float2 w = p_fma(om, nd, e[k]);
                if (sinks) w = p_fma(p_all(-A::w(k)), sink, w);
                v[k] = p_kept(tag, w);
            }
        }
        moved = v[1];
        e[1] = v[1];
#pragma unroll
        for (int i = 2; i < A::Q; ++i) {
            moved = p_add(moved, v[i]);
            e[i] = v[i];
        }
    } else {
        // the moving directions share one weight: w C (1 + c_i.u / cs^2) as deviations is
        // w cp +/- (w / cs^2) C u_a
        constexpr float W = A::w(1);
        const float2 wcp = p_mul(p_all(W), cp), wsink = p_mul(p_all(W), sink);
        const float2 wc_pos = p_mul(p_all(W * A::inv_cs2), Cs), wc_neg = p_mul(p_all(-W * A::inv_cs2), Cs);
        const float2 omc = p_all(omega_c);
#pragma unroll
        for (int i = 1; i < A::Q; ++i) {
            float s;
            const float2 m = p_cdot<A, DIM>(i, u, s);
            const float2 geq = p_fma(s > 0.0f ? wc_pos : wc_neg, m, wcp);
            e[i] = p_kept(tag, p_sub(p_fma(omc, p_sub(geq, e[i]), e[i]), wsink));
            moved = i == 1 ? e[i] : p_add(moved, e[i]);
        }
    }
    e[0] = p_kept(tag, p_sub(p_sub(cp, sink), moved));
}

// The flow outlet value along c_i (Eq. 5 at rho_out with the last layer's velocity), rounded as
// flow_ghosts rounds it.
template <int DIM, typename FORMS>
__device__ __forceinline__ float outlet_value(int i, float rho_out, float u0, float u1, float u2)
{
    using F = FlowSet<DIM>;
    const float uu = i < 2 * DIM + 1 ? s_uu<DIM, FORMS::outlet_axis>(u0, u1, u2) : s_uu<DIM, FORMS::outlet_diagonal>(u0, u1, u2);
    const float uv[3] = {u0, u1, u2};
    float cu = 0.0f;
    bool any = false;
#pragma unroll
    for (int ax = 0; ax < DIM; ++ax) {
        const int c = F::c(i, ax);
        if (c == 0) continue;
        const float t = c > 0 ? uv[ax] : -uv[ax];
        cu = any ? __fadd_rn(cu, t) : t;
        any = true;
    }
    const float t = __fmaf_rn(-1.5f, uu, __fmaf_rn(3.0f, cu, __fmul_rn(__fmul_rn(4.5f, cu), cu)));
    return __fmul_rn(F::w(i), __fmaf_rn(rho_out, t, __fsub_rn(rho_out, 1.0f)));
}

}  // namespace mfc
