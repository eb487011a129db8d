// 2-D plain coupled steps in FP16 with two nodes per thread: node (x, y) and (x, y + 1), the same
// stream-collide as step_node (Eqs. 4, 5, 9-13 with the bounce-back of Eq. 11), with the
// collision of both nodes carried out by Blackwell's paired FP32 instructions (one FFMA2, FADD2 or
// FMUL2 for the two lanes).  In FP16 storage the single-node step spends its issue slots on
// arithmetic, not on HBM (the conversions and the collision per population, at half the bytes of
// FP32); pairing halves the collision's instructions and gives every thread twice the loads in
// flight.  Loads, stores, link bits and boundary work stay per node.
//
// Pairs run along y, never along the inlet/outlet axis, so the inlet and
// outlet tests are the same for both nodes of a pair.  Every lane rounds as an FP32 instruction
// does, but the operations are grouped differently from step_node's (the equilibrium is formed as
// w (1 + rho') t + w rho', the momentum as the sum over c = +1 less the sum over c = -1), so the
// two forms agree to FP32 rounding, not bit for bit.  Single plain steps use the pairs (and lattices
// whose steps cannot go several per launch: a periodic axis, a cut face); lbm_sweep.cuh takes
// several steps in the same grouping and rounding (PAIR_FORM).  Check steps and stored-field steps stay on
// step_node, which reads and writes the same buffers.
#pragma once

#include "lbm_kernels.cuh"

namespace mfc {

__device__ __forceinline__ float2 p_all(float s) { return make_float2(s, s); }
__device__ __forceinline__ float2 p_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 p_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 p_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// a - b, rounded once: the product b * -1 is exact
__device__ __forceinline__ float2 p_sub(float2 a, float2 b) { return __ffma2_rn(b, p_all(-1.0f), a); }

// Sum of v[i] over the directions with c_i[ax] == s, in index order (the loops unroll, so the
// direction tests are resolved at compile time).
template <typename SET, int N>
__device__ __forceinline__ float2 p_sum_where(const float2 (&v)[N], int ax, int s)
{
    float2 r = p_all(0.0f);
    bool any = false;
#pragma unroll
    for (int i = 0; i < SET::Q; ++i) {
        if (SET::c(i, ax) != s) continue;
        r = any ? p_add(r, v[i]) : v[i];
        any = true;
    }
    return r;
}

// c_i . u with unit velocity components, as s m: m is the sum of the u[ax] with c_i[ax] = +1
// less those with -1 when both signs occur, else the sum over the one sign present, s its sign.
template <typename SET, int DIM>
__device__ __forceinline__ float2 p_cdot(int i, const float2 (&u)[3], float &s)
{
    float2 pos = p_all(0.0f), neg = p_all(0.0f);
    bool hp = false, hn = false;
#pragma unroll
    for (int ax = 0; ax < DIM; ++ax) {
        if (SET::c(i, ax) == 1) {
            pos = hp ? p_add(pos, u[ax]) : u[ax];
            hp = true;
        } else if (SET::c(i, ax) == -1) {
            neg = hn ? p_add(neg, u[ax]) : u[ax];
            hn = true;
        }
    }
    s = (hp || !hn) ? 1.0f : -1.0f;
    return (hp && hn) ? p_sub(pos, neg) : (hp ? pos : neg);
}

// Store the two lanes (lane 1 only where it exists); returns the values the stores keep.
__device__ __forceinline__ float2 p_store(__half *p0, __half *p1, bool has1, float2 v)
{
    const __half2 h = __float22half2_rn(v);
    *p0 = __low2half(h);
    if (has1) *p1 = __high2half(h);
    return __half22float2(h);
}

// Which plain steps have this grouping: FP16 storage (2-D here, 3-D in lbm_row.cuh).  They must be the
// ones whose single-node steps take the reader-side boundary form.
template <int DIM, typename ST> struct PairedStep {
    static constexpr bool value = std::is_same<ST, __half>::value;
    static_assert(!value || ReaderBoundaries<DIM, ST>::step, "paired and single-node steps share one boundary form");
};

// Resident blocks of 256 threads per SM (48 registers; 4096x1024 anode: 58.7 us at 5 blocks, 62.6 at 4).
enum : int { PAIR_BLOCKS = 5 };

// The link words of nodes (x, y) and (x, y + 1) (the second repeats the first where y + 1 = ny).
template <typename ST>
__device__ __forceinline__ void pair_links(const StepArgs<2, ST> &a, int x, int y, uint32_t (&L)[2])
{
    const Geo &g = a.geo;
    const int k0 = (int)g.row0 + y * g.px + x;
    const int k1 = y + 1 < g.ny ? k0 + g.px : k0;
    L[0] = __ldg(a.link + MFC_IDX(k0, g.plane));
    L[1] = __ldg(a.link + MFC_IDX(k1, g.plane));
}

// One plain coupled step of nodes (x, y + l), l = 0, 1 (lane 1 absent where y + 1 = ny; x < nx), given
// their link words, with 32-bit element offsets and the default transport set, in the reader form of the
// open boundaries.  BOUNDARY: the block's tile touches one.
template <typename ST, bool BOUNDARY, int SINK>
__device__ __forceinline__ void step_pair(const StepArgs<2, ST> &a, int x, int y, const uint32_t (&L)[2])
{
    using F = FlowSet<2>;
    using A = AdeSet<2>;
    using LK = Links<2>;
    static_assert(std::is_same<ArithT<ST>, float>::value, "paired FP32 arithmetic");
    static_assert(!A::quadratic, "linear transport equilibrium");
    const Geo g = a.geo;
    const bool has1 = y + 1 < g.ny;
    const int P = (int)g.plane;
    const int k0 = (int)g.row0 + y * g.px + x;
    const int k[2] = {k0, has1 ? k0 + g.px : k0};
    bool ghosts[2];
#pragma unroll
    for (int l = 0; l < 2; ++l) ghosts[l] = BOUNDARY && (l == 0 || has1) && step_writes_ghosts<2>(g, a.bc, x, y + l, 0);
    const bool inout = BOUNDARY && a.bc[0] == BC_INOUT;
    const bool at_in = inout && x == 0 && !a.cut[0];
    const bool at_out = inout && x == g.nx - 1 && !a.cut[1];

    // ---- flow: gather (bounce-back and inlet per node), moments, BGK ----
    float2 u[3] = {p_all(0.0f), p_all(0.0f), p_all(0.0f)};
    {
        float2 d[F::Q];
#pragma unroll
        for (int i = 0; i < F::Q; ++i) {
            const int off = F::c(i, 0) + F::c(i, 1) * g.px;
            float v[2];
#pragma unroll
            for (int l = 0; l < 2; ++l) {
                // bounce-back, or the moving-wall value entering across the inlet
                const bool bb = i > 0 && ((L[l] >> i) & 1u);
                const bool inj = F::c(i, 0) == 1 && at_in && !bb;
                const int o = (bb || inj) ? F::opp(i) * P : i * P - off;
                v[l] = ld(a.fsrc + MFC_IDX(k[l] + o, F::Q * P));
                if (F::c(i, 0) == 1 && inj) v[l] += a.bb_in[i];
            }
            d[i] = make_float2(v[0], v[1]);
        }
        const bool open0 = !(L[0] & (1u << LK::FLOW_SELF)), open1 = !(L[1] & (1u << LK::FLOW_SELF));
#pragma unroll
        for (int i = 0; i < F::Q; ++i)  // blocked nodes hold no populations
            d[i] = make_float2(open0 ? d[i].x : 0.0f, open1 ? d[i].y : 0.0f);
        float2 rp = d[0];
#pragma unroll
        for (int i = 1; i < F::Q; ++i) rp = p_add(rp, d[i]);
        const float2 opr = p_add(p_all(1.0f), rp);
        const float2 inv = make_float2(recip(opr.x), recip(opr.y));
#pragma unroll
        for (int ax = 0; ax < 2; ++ax)
            u[ax] = p_mul(p_sub(p_sum_where<F>(d, ax, 1), p_sum_where<F>(d, ax, -1)), inv);
        const float2 uu = p_fma(u[1], u[1], p_mul(u[0], u[0]));
        const float2 muu = p_mul(p_all(-1.5f), uu);
        const float2 om = p_all(a.omega);
        // w (1 + rho') and w rho' of the two moving weight classes (faces; diagonals)
        constexpr int IE = 5;
        const float2 wo_f = p_mul(p_all(F::w(1)), opr), wr_f = p_mul(p_all(F::w(1)), rp);
        const float2 wo_e = p_mul(p_all(F::w(IE)), opr), wr_e = p_mul(p_all(F::w(IE)), rp);
        float2 moved = p_all(0.0f);
#pragma unroll
        for (int i = 1; i < F::Q; ++i) {
            float s;
            const float2 m = p_cdot<F, 2>(i, u, s);
            // 3 cu + 9/2 cu^2 - 3/2 u.u = m (9/2 m + 3 s) - 3/2 u.u
            const float2 t = p_fma(m, p_fma(p_all(4.5f), m, p_all(3.0f * s)), muu);
            const float2 feq = i < IE ? p_fma(wo_f, t, wr_f) : p_fma(wo_e, t, wr_e);
            const float2 v = p_fma(om, p_sub(feq, d[i]), d[i]);
            const float2 vk = p_store(a.fdst + MFC_IDX(i * P + k[0], F::Q * P),
                                      a.fdst + MFC_IDX(i * P + k[1], F::Q * P), has1, v);
            moved = i == 1 ? vk : p_add(moved, vk);
        }
        p_store(a.fdst + MFC_IDX(k[0], F::Q * P), a.fdst + MFC_IDX(k[1], F::Q * P), has1, p_sub(rp, moved));
#pragma unroll
        for (int l = 0; l < 2; ++l) {
            const bool open = l == 0 ? open0 : open1;
            if (!(ghosts[l] && open)) continue;
            const float u0 = l == 0 ? u[0].x : u[0].y, u1 = l == 0 ? u[1].x : u[1].y;
            flow_ghosts_step<2, ST>(a, a.fdst, x, y + l, 0, k[l], u0, u1, 0.0f);
        }
    }

    // ---- transport: gather (zero flux, inlet, outlet per node), linear equilibrium, sink ----
    {
        const float2 us = p_all(a.u_scale);
#pragma unroll
        for (int ax = 0; ax < 2; ++ax) u[ax] = p_mul(u[ax], us);  // 0 on flow-blocked nodes
        float2 e[A::Q];
#pragma unroll
        for (int i = 0; i < A::Q; ++i) {
            const int off = A::c(i, 0) + A::c(i, 1) * g.px;
            float v[2];
#pragma unroll
            for (int l = 0; l < 2; ++l) {
                const bool bb = i > 0 && ((L[l] >> (LK::ADE_SELF + i)) & 1u);
                const bool in_v = A::c(i, 0) == 1 && at_in && !bb;
                const bool out_v = A::c(i, 0) == -1 && at_out && !bb;
                const int o = bb ? A::opp(i) * P : i * P - (out_v ? 0 : off);
                v[l] = ld(a.gsrc + MFC_IDX(k[l] + o, A::Q * P));
                if (A::c(i, 0) == 1 && in_v) v[l] = a.gin_dev[i];
                if (A::c(i, 0) == -1 && out_v && a.ade_dirichlet) v[l] = a.gout_dev[i];
            }
            e[i] = make_float2(v[0], v[1]);
        }
        const bool open0 = !(L[0] & (1u << LK::ADE_SELF)), open1 = !(L[1] & (1u << LK::ADE_SELF));
#pragma unroll
        for (int i = 0; i < A::Q; ++i) e[i] = make_float2(open0 ? e[i].x : 0.0f, open1 ? e[i].y : 0.0f);
        float2 cp = e[0];
#pragma unroll
        for (int i = 1; i < A::Q; ++i) cp = p_add(cp, e[i]);
        const float2 Cs = p_add(p_all(a.c_ref), cp);
        // consumption (Eq. 16's substrate factor): k C, or k C K_s / (K_s + C)
        float2 sink = p_mul(make_float2((L[0] & (1u << LK::SINK)) ? a.k_sink : 0.0f,
                                        (L[1] & (1u << LK::SINK)) ? a.k_sink : 0.0f), Cs);
        if constexpr (SINK == SINK_MONOD) {
            if (L[0] & (1u << LK::SINK)) sink.x = sink.x * a.k_half * recip(a.k_half + Cs.x);
            if (L[1] & (1u << LK::SINK)) sink.y = sink.y * a.k_half * recip(a.k_half + Cs.y);
        }
        // the moving directions share one weight: w C (1 + c_i.u / cs^2) as deviations is
        // w cp +/- (w / cs^2) C u_a
        constexpr float W = A::w(1);
        const float2 wcp = p_mul(p_all(W), cp), wsink = p_mul(p_all(W), sink);
        const float2 wc_pos = p_mul(p_all(W * A::inv_cs2), Cs), wc_neg = p_mul(p_all(-W * A::inv_cs2), Cs);
        const float2 omc = p_all(a.omega_c);
        float2 moved = p_all(0.0f);
#pragma unroll
        for (int i = 1; i < A::Q; ++i) {
            float s;
            const float2 m = p_cdot<A, 2>(i, u, s);
            const float2 geq = p_fma(s > 0.0f ? wc_pos : wc_neg, m, wcp);
            const float2 v = p_sub(p_fma(omc, p_sub(geq, e[i]), e[i]), wsink);
            const float2 vk = p_store(a.gdst + MFC_IDX(i * P + k[0], A::Q * P),
                                      a.gdst + MFC_IDX(i * P + k[1], A::Q * P), has1, v);
            moved = i == 1 ? vk : p_add(moved, vk);
        }
        p_store(a.gdst + MFC_IDX(k[0], A::Q * P), a.gdst + MFC_IDX(k[1], A::Q * P), has1,
                p_sub(p_sub(cp, sink), moved));
#pragma unroll
        for (int l = 0; l < 2; ++l) {
            const bool open = l == 0 ? open0 : open1;
            if (!(ghosts[l] && open)) continue;
            ade_ghosts_step<2, ST>(a, a.gdst, x, y + l, 0, k[l]);
        }
    }
}

// Plain coupled step, two rows per thread: grid (row / block, ceil(ny / 2)), in the reader-side
// boundary form (tiles that touch no open boundary run code with no boundary handling).  The
// single-node steps of the same storage type take it too (ReaderBoundaries), so that the forms
// never mix on one lattice.
// (A loop over several row pairs per thread, loading the next pair's link words ahead, measured
// slower at every depth tried.)
template <typename ST, int SINK>
__global__ void __launch_bounds__(256, PAIR_BLOCKS) lbm_pair_kernel(const StepArgs<2, ST> a)
{
    const int x0 = blockIdx.x * blockDim.x;
    const int x = x0 + (int)threadIdx.x;
    if (x >= a.geo.nx) return;
    const int y = 2 * (int)blockIdx.y;
    uint32_t L[2];
    pair_links(a, x, y, L);
    const int y1 = y + 1 < a.geo.ny ? y + 1 : y;
    if (tile_on_open_boundary<2>(a.geo, a.bc, x0, blockDim.x, y, 0) || tile_on_open_boundary<2>(a.geo, a.bc, x0, blockDim.x, y1, 0))
        step_pair<ST, true, SINK>(a, x, y, L);
    else
        step_pair<ST, false, SINK>(a, x, y, L);
}

}  // namespace mfc
