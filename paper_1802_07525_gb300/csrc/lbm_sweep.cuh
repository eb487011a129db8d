// Several plain steps per sweep of a 2-D lattice.
//
// One plain step per launch reads and writes every population once per step: 112 B per node in
// FP32, which bounds it by HBM on large lattices and by launches and memory latency on small
// ones.  Here a warp marches up a strip of rows, 64 columns wide (two neighbouring columns per
// lane), and carries T steps through its registers: on reading row q it takes step 1 at row q - 1,
// step 2 at row q - 2, ..., and writes the populations after step T at row q - T.  Every
// population is read and written once per T steps; nothing passes through shared memory and no
// warp waits on another.
//   - Along y, a row's pulls are in rows the warp already holds; along x, a pull is the lane's own
//     other column or one shuffle.  Half-way bounce-back (Eq. 11) selects between the pulled
//     value and the node's own opposite population, both in registers; warps whose row has no
//     link to any wall or sink skip the selects.
//   - Each step loses one column at either end of the warp's 64 and one row at either end of its
//     strip: 64 - 2T columns are written, and neighbouring strips recompute 2(T - 1) rows.
//   - The collision runs on the two columns of a lane at once with paired FP32 instructions, in
//     the rounding of the one-step kernel (lbm_collide.cuh): T steps of a sweep give the bits of
//     T one-step launches.
// Inlet and outlet: a node takes its inlet values and its transport outlet value itself when it
// gathers (the reader form of step_node); between the steps of a sweep, the flow outlet values are
// formed in the column beyond the outlet.  What the sweep leaves in the ghost cells of the written
// buffer is what the one-step kernels of the lattice need: in the writer form the inlet and
// transport outlet values too.
//
// For lattices with walls across the flow axis, and walls or inlet/outlet along it, whole
// (no cut faces), with 32-bit element offsets; the others take the one-step kernels.
#pragma once

#include "lbm_collide.cuh"

namespace mfc {

// Columns: a warp's 64 columns begin sweep_halo<T>() before the first one written (even, so that the
// pairs are aligned), and T are lost at either end.
template <int T> __host__ __device__ constexpr int sweep_halo() { return (T + 1) & ~1; }
template <int T> __host__ __device__ constexpr int sweep_width() { return (64 - sweep_halo<T>() - T) & ~1; }

template <int AQ, bool FLOW, bool ADE> struct SweepRow {
    float2 f[FLOW ? 9 : 1];
    float2 g[ADE ? AQ : 1];
};

// The values of two neighbouring columns (x, x + 1) pulled along cx from the row values s.
__device__ __forceinline__ float2 pull_x(int cx, float2 s)
{
    if (cx == 0) return s;
    if (cx > 0) return make_float2(__shfl_up_sync(0xffffffffu, s.y, 1), s.x);
    return make_float2(s.y, __shfl_down_sync(0xffffffffu, s.x, 1));
}

// A pair as it is stored, and its value.
__device__ __forceinline__ float2 ld_pair(const float *p) { return __ldg(reinterpret_cast<const float2 *>(p)); }
__device__ __forceinline__ __half2 ld_pair(const __half *p) { return __ldg(reinterpret_cast<const __half2 *>(p)); }
__device__ __forceinline__ float2 pair_value(float2 v) { return v; }
__device__ __forceinline__ float2 pair_value(__half2 v) { return __half22float2(v); }
// link words of two neighbouring nodes (even x)
__device__ __forceinline__ uint2 ld_links(const uint16_t *p)
{
    const uint32_t v = __ldg(reinterpret_cast<const uint32_t *>(p));
    return make_uint2(v & 0xffffu, v >> 16);
}
__device__ __forceinline__ uint2 ld_links(const uint32_t *p) { return __ldg(reinterpret_cast<const uint2 *>(p)); }
__device__ __forceinline__ void st_pair(float *p, float2 v) { *reinterpret_cast<float2 *>(p) = v; }
__device__ __forceinline__ void st_pair(__half *p, float2 v) { *reinterpret_cast<__half2 *>(p) = __float22half2_rn(v); }

// The inlet or outlet value v as a gathering node sees it: as it is in the reader form, as its
// ghost cell would keep it in the writer form.
template <int AQ, int SINK, typename ST> __device__ __forceinline__ float ghost_value(const ST *tag, float v)
{
    return ReaderForm<2, ST, AQ, SINK>::value ? v : kept(tag, v);
}

// Column state of a lane in tiles that hold the inlet or the outlet.
struct SweepEdge {
    bool inlet;    // the lane's first column is column 0 of an inlet
    int last;      // which of the lane's columns is the last one (0, 1), or -1
    int beyond;    // which of the lane's columns is the one beyond the outlet, or -1
};

// What a stage keeps of the row it steps next until the row above arrives: the populations already
// gathered (the directions along the row and going up), and in `up` the row's own populations going up
// (pulled by the row above, and bounced back by the row itself where the ones going down are blocked).
template <int AQ, bool FLOW, bool ADE> struct SweepStage {
    SweepRow<AQ, FLOW, ADE> got, up;
    uint2 L;       // links of the row
    bool links;    // any in the warp (uniform)
    float2 uf[2];  // frozen velocity (transport without flow)
};

// Gather the populations along c_i with c_iy < 0 (DOWN: from the row above, `above`) or >= 0 (from
// the row itself, `own`, and the row below, `below`) of one set into d.
template <typename ST, int AQ, int SINK, int Q, bool FLOWSET, bool DOWN, bool EDGE, typename D, typename FB, typename FO,
          typename FA>
__device__ __forceinline__ void sweep_gather(const StepArgs<2, ST, AQ> &a, D &d, const FB &below, const FO &own,
                                             const FA &above, uint2 L, bool links, const SweepEdge &edge)
{
    using F = FlowSet<2>;  // the transport sets are its first directions
    const ST *tag = nullptr;
    constexpr int SELF = FLOWSET ? 0 : Links<2, AQ>::ADE_SELF;
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        const int cx = F::c(i, 0), cy = F::c(i, 1);
        if ((cy < 0) != DOWN) continue;
        const float2 s = cy > 0 ? below(i) : (cy < 0 ? above(i) : own(i));
        d[i] = pull_x(cx, s);
        if (EDGE && !FLOWSET && cx == -1 && edge.last >= 0) {  // outlet: zero gradient, or the Dirichlet value
            const float v = a.ade_dirichlet ? ghost_value<AQ, SINK>(tag, a.gout_dev[i < AQ ? i : 0]) : (edge.last ? s.y : s.x);
            if (edge.last) d[i].y = v;
            else d[i].x = v;
        }
        if (EDGE && cx == 1 && edge.inlet) {  // moving-wall bounce-back, or the transport inlet value
            if constexpr (!FLOWSET) d[i].x = ghost_value<AQ, SINK>(tag, a.gin_dev[i < AQ ? i : 0]);
            else d[i].x = ghost_value<AQ, SINK>(tag, own(F::opp(i)).x + a.bb_in[i]);
        }
    }
    if (links) {
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            if ((F::c(i, 1) < 0) != DOWN) continue;
            const float2 o = own(F::opp(i));
            d[i] = make_float2((L.x >> (SELF + i)) & 1u ? o.x : d[i].x, (L.y >> (SELF + i)) & 1u ? o.y : d[i].y);
        }
    }
}

// The next row of a stage arrives: v, its populations after the step before, with links L.  The row the
// stage holds is gathered completely into out (not yet collided); then the stage holds the new row.
template <typename ST, bool FLOW, bool ADE, int AQ, int SINK, bool EDGE>
__device__ __forceinline__ void sweep_arrive(const StepArgs<2, ST, AQ> &a, SweepStage<AQ, FLOW, ADE> &st,
                                             const SweepRow<AQ, FLOW, ADE> &v, uint2 L, const SweepEdge &edge,
                                             SweepRow<AQ, FLOW, ADE> &out)
{
    using F = FlowSet<2>;
    const bool links = __any_sync(0xffffffffu, (L.x | L.y) != 0u);
    if constexpr (FLOW) {
        auto none = [&](int) { return p_all(0.0f); };
        auto held = [&](int i) { return st.up.f[i]; };
        auto now = [&](int i) { return v.f[i]; };
#pragma unroll
        for (int i = 0; i < 9; ++i)
            if (F::c(i, 1) >= 0) out.f[i] = st.got.f[i];
        sweep_gather<ST, AQ, SINK, 9, true, true, EDGE>(a, out.f, none, held, now, st.L, st.links, edge);
        st.got.f[0] = v.f[0];
        sweep_gather<ST, AQ, SINK, 9, true, false, EDGE>(a, st.got.f, held, now, none, L, links, edge);
#pragma unroll
        for (int i = 1; i < 9; ++i)
            if (F::c(i, 1) > 0) st.up.f[i] = v.f[i];
    }
    if constexpr (ADE) {
        auto none = [&](int) { return p_all(0.0f); };
        auto held = [&](int i) { return st.up.g[i]; };
        auto now = [&](int i) { return v.g[i]; };
#pragma unroll
        for (int i = 0; i < AQ; ++i)
            if (F::c(i, 1) >= 0) out.g[i] = st.got.g[i];
        sweep_gather<ST, AQ, SINK, AQ, false, true, EDGE>(a, out.g, none, held, now, st.L, st.links, edge);
        st.got.g[0] = v.g[0];
        sweep_gather<ST, AQ, SINK, AQ, false, false, EDGE>(a, st.got.g, held, now, none, L, links, edge);
#pragma unroll
        for (int i = 1; i < AQ; ++i)
            if (F::c(i, 1) > 0) st.up.g[i] = v.g[i];
    }
    st.L = L;
    st.links = links;
}

// Collide the gathered row d (links L) in place; u: the flow velocity.
template <typename ST, bool FLOW, bool ADE, int AQ, int SINK, int FORM>
__device__ __forceinline__ void sweep_collide(const StepArgs<2, ST, AQ> &a, SweepRow<AQ, FLOW, ADE> &d, uint2 L, bool links,
                                              const float2 (&uf)[2], float2 (&u)[3])
{
    using LK = Links<2, AQ>;
    u[0] = u[1] = u[2] = p_all(0.0f);
    if constexpr (FLOW) {
        float2 rp;
        collide_flow<2, ST, FORM, UuForm<2, ST, ADE, AQ, SINK>::collision>(d.f, a.omega, u, rp);
    }
    if constexpr (ADE) {
        float2 v[3] = {uf[0], uf[1], p_all(0.0f)};
        float k0 = 0.0f, k1 = 0.0f;
        if constexpr (FLOW) {
            v[0] = u[0];
            v[1] = u[1];
        }
        if (links) {
            if constexpr (!FLOW) {  // at rest on flow-blocked nodes
                if (L.x & (1u << LK::FLOW_SELF)) v[0].x = v[1].x = 0.0f;
                if (L.y & (1u << LK::FLOW_SELF)) v[0].y = v[1].y = 0.0f;
            }
            k0 = L.x & (1u << LK::SINK) ? a.k_sink : 0.0f;
            k1 = L.y & (1u << LK::SINK) ? a.k_sink : 0.0f;
        }
        const float2 us = p_all(a.u_scale);
        v[0] = p_mul(v[0], us);
        v[1] = p_mul(v[1], us);
        collide_ade<2, ST, AQ, SINK, FORM>(d.g, v, a.omega_c, a.c_ref, a.k_half, links, k0, k1);
    }
}

// Flow outlet values in the column beyond the outlet (the directions entering from it), between the
// steps of a sweep.
template <typename ST, bool FLOW, bool ADE, int AQ, int SINK>
__device__ __forceinline__ void sweep_outlet(const StepArgs<2, ST, AQ> &a, const SweepEdge &edge, const float2 (&u)[3],
                                             SweepRow<AQ, FLOW, ADE> &out)
{
    using F = FlowSet<2>;
    const ST *tag = nullptr;
    const float l0 = __shfl_up_sync(0xffffffffu, u[0].y, 1), l1 = __shfl_up_sync(0xffffffffu, u[1].y, 1);
    if (edge.beyond < 0) return;
    const float u0 = edge.beyond ? u[0].x : l0, u1 = edge.beyond ? u[1].x : l1;
#pragma unroll
    for (int i = 1; i < F::Q; ++i) {
        if (F::c(i, 0) != -1) continue;
        const float v = kept(tag, outlet_value<2, UuForm<2, ST, ADE, AQ, SINK>>(i, a.rho_out, u0, u1, 0.0f));
        if (edge.beyond) out.f[i].y = v;
        else out.f[i].x = v;
    }
}

// Ghost cells of the written buffer that belong to the nodes of one row at the inlet or outlet.
template <typename ST, bool FLOW, bool ADE, int AQ, int SINK>
__device__ __forceinline__ void sweep_ghosts(const StepArgs<2, ST, AQ> &a, const SweepEdge &edge, int y, int k, uint2 L,
                                             const float2 (&u)[3], const SweepRow<AQ, FLOW, ADE> &v)
{
    using F = FlowSet<2>;
    using S = AdeSet<2, AQ>;
    using LK = Links<2, AQ>;
    constexpr bool WRITER = !ReaderForm<2, ST, AQ, SINK>::value;
    const int P = (int)a.geo.plane, px = a.geo.px;
    if (WRITER && edge.inlet) {
        if constexpr (FLOW) {
            if (!(L.x & (1u << LK::FLOW_SELF))) {
#pragma unroll
                for (int i = 1; i < F::Q; ++i)
                    if (F::c(i, 0) == 1 && !((L.x >> i) & 1u))
                        st(a.fdst + MFC_IDX(i * P + k - 1 - F::c(i, 1) * px, F::Q * P), v.f[F::opp(i)].x + a.bb_in[i]);
            }
        }
        if constexpr (ADE) {
            if (!(L.x & (1u << LK::ADE_SELF))) {
#pragma unroll
                for (int i = 1; i < S::Q; ++i)
                    if (S::c(i, 0) == 1 && !((L.x >> (LK::ADE_SELF + i)) & 1u))
                        st(a.gdst + MFC_IDX(i * P + k - 1 - S::c(i, 1) * px, S::Q * P), a.gin_dev[i]);
            }
        }
    }
    if (edge.last >= 0) {
        const uint32_t l = edge.last ? L.y : L.x;
        const int q = k + edge.last + 1;
        if constexpr (FLOW) {
            if (!(l & (1u << LK::FLOW_SELF))) {
                const float u0 = edge.last ? u[0].y : u[0].x, u1 = edge.last ? u[1].y : u[1].x;
#pragma unroll
                for (int i = 1; i < F::Q; ++i)
                    if (F::c(i, 0) == -1 && y + F::c(i, 1) >= 0 && y + F::c(i, 1) < a.geo.ny)
                        st(a.fdst + MFC_IDX(i * P + q, F::Q * P), outlet_value<2, UuForm<2, ST, ADE, AQ, SINK>>(i, a.rho_out, u0, u1, 0.0f));
            }
        }
        if constexpr (ADE) {
            if (WRITER && !(l & (1u << LK::ADE_SELF))) {
#pragma unroll
                for (int i = 1; i < S::Q; ++i)
                    if (S::c(i, 0) == -1 && y + S::c(i, 1) >= 0 && y + S::c(i, 1) < a.geo.ny)
                        st(a.gdst + MFC_IDX(i * P + q, S::Q * P),
                           a.ade_dirichlet ? a.gout_dev[i] : (edge.last ? v.g[i].y : v.g[i].x));
            }
        }
    }
}

// T steps of rows [y0, y1), columns [x0, x1) by one warp.
template <typename ST, bool FLOW, bool ADE, int AQ, int SINK, int FORM, int T, bool EDGE>
__device__ __forceinline__ void sweep_strip(const StepArgs<2, ST, AQ> &a, int x0, int x1, int y0, int y1)
{
    using Row = SweepRow<AQ, FLOW, ADE>;
    const Geo &g = a.geo;
    const int nx = g.nx, ny = g.ny, px = g.px;
    const int P = (int)g.plane, row0 = (int)g.row0;
    const int X = x0 - sweep_halo<T>() + 2 * (int)threadIdx.x;
    // columns beyond the ghost column are not needed: repeat the last pair that holds it
    const int Xc = EDGE ? min(X, nx & ~1) : X;
    SweepEdge edge = {false, -1, -1};
    if (EDGE && a.bc[0] == BC_INOUT) {
        edge.inlet = X == 0;
        edge.last = X == nx - 1 ? 0 : (X + 1 == nx - 1 ? 1 : -1);
        edge.beyond = X == nx ? 0 : (X + 1 == nx ? 1 : -1);
    }
    const bool store = X >= x0 && X < x1, both = !EDGE || X + 1 < nx;

    using Pair = typename std::conditional<std::is_same<ST, __half>::value, __half2, float2>::type;
    struct Raw {
        Pair f[FLOW ? 9 : 1], g[ADE ? AQ : 1];
        uint2 L;
        float2 uf[2];
    };
    auto load = [&](Raw &r, int q) {
        const int kr = row0 + min(max(q, -1), ny) * px + Xc;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            if constexpr (FLOW) r.f[i] = ld_pair(a.fsrc + MFC_IDX(i * P + kr, 9 * P - 1));
        }
#pragma unroll
        for (int i = 0; i < AQ; ++i) {
            if constexpr (ADE) r.g[i] = ld_pair(a.gsrc + MFC_IDX(i * P + kr, AQ * P - 1));
        }
        r.L = ld_links(a.link + MFC_IDX(kr, P - 1));
        if constexpr (!FLOW) {
#pragma unroll
            for (int ax = 0; ax < 2; ++ax) r.uf[ax] = ld_pair(a.fld_u + MFC_IDX(ax * P + kr, 2 * P - 1));
        }
    };

    // turn q: raw row q arrives at stage 1, which steps row q - 1, which arrives at stage 2, ...; stage
    // T steps row q - T, which is written.  Row q + 1 is loaded as soon as row q has been gathered from.
    // The stages start from zeros, although what the first turns gather from them is dropped: from an
    // indeterminate start the compiler may take a held value for the arriving one in every turn (it did,
    // for the inlet value of the direction going down).
    SweepStage<AQ, FLOW, ADE> st[T];
#pragma unroll
    for (int s = 0; s < T; ++s) {
#pragma unroll
        for (int i = 0; i < (FLOW ? 9 : 0); ++i) st[s].got.f[i] = st[s].up.f[i] = p_all(0.0f);
#pragma unroll
        for (int i = 0; i < (ADE ? AQ : 0); ++i) st[s].got.g[i] = st[s].up.g[i] = p_all(0.0f);
        st[s].L = make_uint2(0, 0);
        st[s].links = false;
        st[s].uf[0] = st[s].uf[1] = p_all(0.0f);
    }
    Raw in = {};
    const int q_last = y1 - 1 + T;
    auto turn = [&](int q) {
        Row v;
        uint2 L = in.L;
        float2 uf[2] = {in.uf[0], in.uf[1]}, u[3];
#pragma unroll
        for (int s = 0; s < T; ++s) {
            // stage s + 1 steps row q - s - 1, needed from row y0 - T + s + 1 on
            const uint2 Ls = st[s].L;
            const bool ls = st[s].links;
            const float2 us[2] = {st[s].uf[0], st[s].uf[1]};
            Row out;
            if (s == 0) {
#pragma unroll
                for (int i = 0; i < (FLOW ? 9 : 0); ++i) v.f[i] = pair_value(in.f[i]);
#pragma unroll
                for (int i = 0; i < (ADE ? AQ : 0); ++i) v.g[i] = pair_value(in.g[i]);
            }
            sweep_arrive<ST, FLOW, ADE, AQ, SINK, EDGE>(a, st[s], v, L, edge, out);
            st[s].uf[0] = uf[0];
            st[s].uf[1] = uf[1];
            if (s == 0 && q < q_last) load(in, q + 1);
            if (q < y0 - T + 2 * (s + 1)) return;
            v = out;
            sweep_collide<ST, FLOW, ADE, AQ, SINK, FORM>(a, v, Ls, ls, us, u);
            if constexpr (FLOW && EDGE) {
                if (s < T - 1) sweep_outlet<ST, FLOW, ADE, AQ, SINK>(a, edge, u, v);
            }
            L = Ls;
            uf[0] = us[0];
            uf[1] = us[1];
        }
        const int y = q - T;
        const int k = row0 + y * px + X;
        if (store) {
            if (both) {
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    if constexpr (FLOW) st_pair(a.fdst + MFC_IDX(i * P + k, 9 * P - 1), v.f[i]);
                }
#pragma unroll
                for (int i = 0; i < AQ; ++i) {
                    if constexpr (ADE) st_pair(a.gdst + MFC_IDX(i * P + k, AQ * P - 1), v.g[i]);
                }
            } else {
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    if constexpr (FLOW) mfc::st(a.fdst + MFC_IDX(i * P + k, 9 * P), v.f[i].x);
                }
#pragma unroll
                for (int i = 0; i < AQ; ++i) {
                    if constexpr (ADE) mfc::st(a.gdst + MFC_IDX(i * P + k, AQ * P), v.g[i].x);
                }
            }
            if (EDGE) sweep_ghosts<ST, FLOW, ADE, AQ, SINK>(a, edge, y, k, L, u, v);
        }
    };
    load(in, y0 - T);
    for (int q = y0 - T; q <= q_last; ++q) turn(q);
}

// Steps per sweep and resident warps per SM, measured: two steps with 12 warps (164 registers) for
// D2Q9 + D2Q5 (2048x1024 FP32: 24 us per step; with 13 warps, where it spills, 37; with 10, 28; three
// steps with 8 warps 26).  D2Q9 transport, 8 warps: two steps coupled (240 registers; 2048x1024 FP32 31.5 us, FP16
// 36.5; three steps spill 112 bytes: 38.0 and 40.7), three for flow alone and transport alone (2048x1024 in the
// paper's order 32.2 and 38.0 us; two steps 41.1 and 39.8).
template <int AQ, bool COUPLED> struct SweepSteps {
    static constexpr int value = AQ == 9 && !COUPLED ? 3 : 2;
};
template <int T, int AQ> struct SweepOccupancy {
    static constexpr int blocks = T == 2 && AQ != 9 ? 12 : 8;
};

// One warp per block, so that everything that depends on the strip is uniform: one column tile of one
// strip each, the tiles of a strip first.
template <typename ST, bool FLOW, bool ADE, int AQ, int SINK, int FORM, int T>
__global__ void __launch_bounds__(32, SweepOccupancy<T, AQ>::blocks)
    lbm_sweep_kernel(const StepArgs<2, ST, AQ> a, const SweepShape s)
{
    const int x0 = blockIdx.x * s.width, y0 = blockIdx.y * s.rows;
    const int x1 = min(x0 + s.width, a.geo.nx), y1 = min(y0 + s.rows, a.geo.ny);
    // tiles whose 64 columns hold the first, the last column or the one beyond
    if (x0 == 0 || x0 + 64 - sweep_halo<T>() >= a.geo.nx)
        sweep_strip<ST, FLOW, ADE, AQ, SINK, FORM, T, true>(a, x0, x1, y0, y1);
    else
        sweep_strip<ST, FLOW, ADE, AQ, SINK, FORM, T, false>(a, x0, x1, y0, y1);
}

// ---- small lattices ---------------------------------------------------------------------------
// A lattice that does not fill the GPU is bound by launches and by the latency of a step's loads, not
// by bandwidth.  Here a block takes a tile of rows T steps at a time: one warp per row (64 columns) loads
// it once, and between the steps the rows exchange the populations that cross them through shared memory
// (a row's own stay in registers).  Each step loses one row at either end of the tile: a block of w warps
// writes w - 2 T rows.  The rows lost are recomputed by the neighbouring tiles, which an idle GPU affords.
// T is a launch parameter: any number of steps up to TILE_STEPS goes in one launch.
// Measured (solve blocks, FP32 D2Q9 + D2Q5): 128x64 5.1 us per step with one-step launches, 2.9 with
// strips of two steps, 1.1 with tiles of four; 611x293 4.5, 4.1 and 2.9; 1024x512 11.5, 7.4 and 7.0;
// 2048x1024 41, 23.6 and 25.4 (there the recomputed rows cost more than the strips' waits).
// (Two register rows that swap roles, to save the copies of v, spill: 9 to 40% slower.)
enum : int { TILE_STEPS = 8, TILE_WARPS = 28 };  // 28 warps: at most 72 registers, which the kernel needs

template <bool FLOW, bool ADE, int AQ> struct TileExchange {
    static constexpr int per = (FLOW ? 3 : 0) + (ADE ? (AQ == 9 ? 3 : 1) : 0);  // populations going up, and down
    static constexpr int row = 2 * per * 32;                                  // float2 per row
    // place of a population that crosses rows among those of its direction of y
    __host__ __device__ static constexpr int place(bool ade, int i)
    {
        const int k = i == 2 || i == 4 ? 0 : (i == 5 || i == 7 ? 1 : 2);
        return (ade && FLOW ? 3 : 0) + k + (FlowSet<2>::c(i, 1) < 0 ? per : 0);
    }
};

template <typename ST, bool FLOW, bool ADE, int AQ, int SINK, int FORM, bool EDGE>
__device__ __forceinline__ void tile_steps(const StepArgs<2, ST, AQ> &a, float2 *sh, int x0, int x1, int y0, int rows, int T)
{
    using X = TileExchange<FLOW, ADE, AQ>;
    using F = FlowSet<2>;
    const Geo &g = a.geo;
    const int nx = g.nx, ny = g.ny;
    const int P = (int)g.plane;
    const int lane = (int)(threadIdx.x & 31), warps = rows + 2 * T;
    const int w = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int y = y0 - T + w;
    const int x = x0 - ((T + 1) & ~1) + 2 * lane;
    const int xc = EDGE ? min(max(x, -2), nx & ~1) : x;
    SweepEdge edge = {false, -1, -1};
    if (EDGE && a.bc[0] == BC_INOUT) {
        edge.inlet = x == 0;
        edge.last = x == nx - 1 ? 0 : (x + 1 == nx - 1 ? 1 : -1);
        edge.beyond = x == nx ? 0 : (x + 1 == nx ? 1 : -1);
    }
    SweepRow<AQ, FLOW, ADE> v;
    uint2 L = make_uint2(0, 0);
    float2 uf[2] = {p_all(0.0f), p_all(0.0f)}, u[3];
#pragma unroll
    for (int i = 0; i < (FLOW ? 9 : 0); ++i) v.f[i] = p_all(0.0f);
#pragma unroll
    for (int i = 0; i < (ADE ? AQ : 0); ++i) v.g[i] = p_all(0.0f);
    const bool inside = y >= 0 && y < ny;
    if (inside) {
        const int k = (int)g.row0 + y * g.px + xc;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            if constexpr (FLOW) v.f[i] = pair_value(ld_pair(a.fsrc + MFC_IDX(i * P + k, 9 * P - 1)));
        }
#pragma unroll
        for (int i = 0; i < AQ; ++i) {
            if constexpr (ADE) v.g[i] = pair_value(ld_pair(a.gsrc + MFC_IDX(i * P + k, AQ * P - 1)));
        }
        L = ld_links(a.link + MFC_IDX(k, P - 1));
        if constexpr (!FLOW) {
#pragma unroll
            for (int ax = 0; ax < 2; ++ax) uf[ax] = ld_pair(a.fld_u + MFC_IDX(ax * P + k, 2 * P - 1));
        }
    }
    const bool links = __any_sync(0xffffffffu, (L.x | L.y) != 0u);
    for (int s = 1; s <= T; ++s) {
        // two buffers in turn: one barrier per step
        float2 *mine = sh + ((s & 1) * warps + w) * X::row + lane;
#pragma unroll
        for (int i = 1; i < 9; ++i) {
            if (F::c(i, 1) == 0) continue;
            if constexpr (FLOW) mine[X::place(false, i) * 32] = v.f[i];
            if constexpr (ADE) {
                if (i < AQ) mine[X::place(true, i) * 32] = v.g[i];
            }
        }
        __syncthreads();
        // rows that this step loses, or outside the lattice, only take part in the exchange
        if (!inside || w < s || w >= warps - s) continue;
        const float2 *below_row = mine - X::row, *above_row = mine + X::row;
        SweepRow<AQ, FLOW, ADE> d;
        if constexpr (FLOW) {
            auto below = [&](int i) { return below_row[X::place(false, i) * 32]; };
            auto above = [&](int i) { return above_row[X::place(false, i) * 32]; };
            auto own = [&](int i) { return v.f[i]; };
            d.f[0] = v.f[0];
            sweep_gather<ST, AQ, SINK, 9, true, false, EDGE>(a, d.f, below, own, above, L, links, edge);
            sweep_gather<ST, AQ, SINK, 9, true, true, EDGE>(a, d.f, below, own, above, L, links, edge);
        }
        if constexpr (ADE) {
            auto below = [&](int i) { return below_row[X::place(true, i) * 32]; };
            auto above = [&](int i) { return above_row[X::place(true, i) * 32]; };
            auto own = [&](int i) { return v.g[i]; };
            d.g[0] = v.g[0];
            sweep_gather<ST, AQ, SINK, AQ, false, false, EDGE>(a, d.g, below, own, above, L, links, edge);
            sweep_gather<ST, AQ, SINK, AQ, false, true, EDGE>(a, d.g, below, own, above, L, links, edge);
        }
        v = d;
        sweep_collide<ST, FLOW, ADE, AQ, SINK, FORM>(a, v, L, links, uf, u);
        if constexpr (FLOW && EDGE) {
            if (s < T) sweep_outlet<ST, FLOW, ADE, AQ, SINK>(a, edge, u, v);
        }
    }
    if (!inside || w < T || w >= warps - T || x < x0 || x >= x1) return;
    const int k = (int)g.row0 + y * g.px + x;
    if (!EDGE || x + 1 < nx) {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            if constexpr (FLOW) st_pair(a.fdst + MFC_IDX(i * P + k, 9 * P - 1), v.f[i]);
        }
#pragma unroll
        for (int i = 0; i < AQ; ++i) {
            if constexpr (ADE) st_pair(a.gdst + MFC_IDX(i * P + k, AQ * P - 1), v.g[i]);
        }
    } else {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            if constexpr (FLOW) st(a.fdst + MFC_IDX(i * P + k, 9 * P), v.f[i].x);
        }
#pragma unroll
        for (int i = 0; i < AQ; ++i) {
            if constexpr (ADE) st(a.gdst + MFC_IDX(i * P + k, AQ * P), v.g[i].x);
        }
    }
    if (EDGE) sweep_ghosts<ST, FLOW, ADE, AQ, SINK>(a, edge, y, k, L, u, v);
}

template <typename ST, bool FLOW, bool ADE, int AQ, int SINK, int FORM>
__global__ void __launch_bounds__(TILE_WARPS * 32, 1) lbm_tile_kernel(const StepArgs<2, ST, AQ> a, const SweepShape s)
{
    extern __shared__ __align__(16) char tile_sh[];  // two buffers of a row per warp
    float2 *sh = reinterpret_cast<float2 *>(tile_sh);
    const int x0 = blockIdx.x * s.width, y0 = blockIdx.y * s.rows;
    const int x1 = min(x0 + s.width, a.geo.nx);
    if (x0 == 0 || x0 + 64 - ((s.steps + 1) & ~1) >= a.geo.nx)
        tile_steps<ST, FLOW, ADE, AQ, SINK, FORM, true>(a, sh, x0, x1, y0, s.rows, s.steps);
    else
        tile_steps<ST, FLOW, ADE, AQ, SINK, FORM, false>(a, sh, x0, x1, y0, s.rows, s.steps);
}

// Tiles of many lattices (batches): one launch of T plain steps for every instance that can sweep.  A fixed
// grid walks the table of tiles; the argument block of a tile's instance is copied to shared memory.  Every
// launch uses one tile height and the column tiles of BATCH_STEPS steps, so that one table serves launches
// of any T up to that (12 anodes of 2.2 million nodes together, FP32: 35.6 us per step with four steps of 8
// rows, 36.9 with three; 52.9 with one step per launch).
template <typename ST> struct BatchSweep {
    static constexpr int steps = sizeof(ST) == 4 ? 4 : 3, rows = 8;
    static constexpr int warps = rows + 2 * steps;
    static constexpr int exchange = 2 * warps * TileExchange<true, true, 5>::row * (int)sizeof(float2);
};

template <typename ST>
__global__ void __launch_bounds__(BatchSweep<ST>::warps * 32, 2) lbm_batch_tile_kernel(const BatchArgs<2, ST> b, int T)
{
    static_assert(sizeof(StepArgs<2, ST>) % 4 == 0, "argument block copied as 32-bit words");
    __shared__ StepArgs<2, ST> sa;
    extern __shared__ __align__(16) char batch_sh[];
    float2 *sh = reinterpret_cast<float2 *>(batch_sh);
    constexpr int WORDS = (int)(sizeof(StepArgs<2, ST>) / 4);
    const int n = *b.ntiles;
    int cur = -1;
    for (int t = blockIdx.x; t < n; t += gridDim.x) {
        const Tile tile = b.tiles[t];  // x0, first row (y), end of the columns (z)
        __syncthreads();               // the tile before: its exchange buffers and arguments are no longer read
        if (tile.slot != cur) {
            const uint32_t *src = reinterpret_cast<const uint32_t *>(b.inst + 2 * tile.slot + b.parity);
            uint32_t *dst = reinterpret_cast<uint32_t *>(&sa);
            for (int w = threadIdx.x; w < WORDS; w += blockDim.x) dst[w] = src[w];
            __syncthreads();
            cur = tile.slot;
        }
        if (tile.x0 == 0 || tile.x0 + 64 - ((T + 1) & ~1) >= sa.geo.nx)
            tile_steps<ST, true, true, 5, SINK_RUNTIME, SCALAR_FORM, true>(sa, sh, tile.x0, tile.z, tile.y, BatchSweep<ST>::rows, T);
        else
            tile_steps<ST, true, true, 5, SINK_RUNTIME, SCALAR_FORM, false>(sa, sh, tile.x0, tile.z, tile.y, BatchSweep<ST>::rows, T);
    }
}

}  // namespace mfc
