// Two plain coupled steps per sweep of a 3-D lattice in FP32.
//
// One plain step per launch reads and writes every population once per step: 208 B per node.  Here a block
// marches up a column of planes, MARCH_ROWS rows of 64 columns (one warp per row, two neighbouring columns per
// lane), and carries two steps through registers: on plane p it takes step 1, which arrives at step 2, which
// finishes plane p - 1.  Every population is read and written once per two steps.
//   - Between the steps, a pull along x is a shuffle, along z the values are in registers, and along y they
//     pass through shared memory (three planes of the directions that cross rows; one barrier per plane).
//   - The next plane's loads are issued before step 2's collision, which hides their latency.
//   - A block loses one row at either edge, a warp two columns at either end; a column's first and last planes
//     are stepped once more by its neighbours.
// Bound by latency at 8 warps of 252 registers per SM (no spills): 39% of issue slots used, 880 MB of DRAM traffic
// per two 256x128x128 steps at 3.4 TB/s; a turn of a plane takes 2.6 us, a third of it for the edges.  The rows
// are what the registers allow (12 rows at 168 registers: 168 us per 256x128x128 step instead of 134; rings of
// planes in shared memory instead of registers: 156 to 170).  us per step, one step per launch and two:
// 120x120x120 57.4 and 53.3, 256x128x128 135.7 and 134.3, 256x256x128 268 and 250, 300x200x150 307 and 248.
// The rule for which lattices is march_shape's.  (Flow or transport alone, and FP16 storage, are faster in the
// row kernel at every size.)
// The rounding is that of the one-step kernels (lbm_collide.cuh): two steps here give the bits of two launches
// of lbm_row_kernel, and leave the same ghost cells.
//
// For lattices with walls across x and y, walls or inlet/outlet along z, whole (no cut faces), with 32-bit
// element offsets.
#pragma once

#include "lbm_row.cuh"

namespace mfc {

enum : int { MARCH_ROWS = 8, MARCH_WIDTH = 60 };

struct MarchRow {
    float2 f[19], g[7];
};

// Exchange across rows: the directions with c_y != 0 of one plane, a pair per lane.
struct MarchExchange {
    static constexpr int row = 12 * 32, plane = MARCH_ROWS * row;  // float2
    static constexpr int bytes = 3 * plane * (int)sizeof(float2);
    __host__ __device__ static constexpr int place(bool ade, int i)
    {
        int n = ade ? 10 : 0;
        for (int k = 0; k < i; ++k) n += FlowSet<3>::c(k, 1) != 0 ? 1 : 0;
        return n;
    }
};

// A warp's raw row of one plane: gathered where the row has links, else the pairs at the source rows, still to
// be shifted along x.
__device__ __forceinline__ void march_load(const StepArgs<3, float> &a, MarchRow &v, int k, uint2 L, bool links)
{
    using F = FlowSet<3>;
    const int P = (int)a.geo.plane, px = a.geo.px, zs = (int)a.geo.zs;
    if (links) {
        row_gather<19, 0, true, false>(a, a.fsrc, v.f, k, L, true, false, false);
        row_gather<7, Links<3>::ADE_SELF, false, false>(a, a.gsrc, v.g, k, L, true, false, false);
    } else {
#pragma unroll
        for (int i = 0; i < 19; ++i) {
            const int o = k + i * P - F::c(i, 1) * px - F::c(i, 2) * zs;
            v.f[i] = ld_pair(a.fsrc + MFC_IDX(o, 19 * P - 1));
            if (i < 7) v.g[i] = ld_pair(a.gsrc + MFC_IDX(o, 7 * P - 1));
        }
    }
}

template <int SINK>
__device__ __forceinline__ void march_collide(const StepArgs<3, float> &a, MarchRow &d, uint2 L, bool links, float2 (&u)[3])
{
    using LK = Links<3>;
    float2 rp, v[3];
    collide_flow<3, float, SCALAR_FORM, UuForm<3, float, true, 7, SINK>::collision>(d.f, a.omega, u, rp);
    const float2 us = p_all(a.u_scale);
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) v[ax] = p_mul(u[ax], us);
    collide_ade<3, float, 7, SINK, SCALAR_FORM>(d.g, v, a.omega_c, a.c_ref, a.k_half, links,
                                                L.x & (1u << LK::SINK) ? a.k_sink : 0.0f, L.y & (1u << LK::SINK) ? a.k_sink : 0.0f);
}

// Step 2's gather of one set.  v: plane p after step 1 (own row); now / before: the exchanged planes p and
// p - 1.  Finishes plane p - 1 in d (its directions going down arrive from plane p) and leaves plane p's other
// directions in got; up: the row's own populations going up, plane p - 1 on entry, p on return.
template <int Q, int SELF, bool FLOWSET>
__device__ __forceinline__ void march_arrive(const StepArgs<3, float> &a, float2 (&d)[Q], float2 (&got)[Q], float2 (&up)[Q],
                                             const float2 (&v)[Q], const float2 *now, const float2 *before, uint2 Lr, uint2 L,
                                             bool inlet, bool outlet_r)
{
    using F = FlowSet<3>;
    using X = MarchExchange;
    auto sel = [&](int i, uint2 l, float2 own, float2 w) {
        return make_float2((l.x >> (SELF + i)) & 1u ? own.x : w.x, (l.y >> (SELF + i)) & 1u ? own.y : w.y);
    };
    auto crossed = [&](const float2 *plane, int i) { return plane[X::place(!FLOWSET, i) * 32 - F::c(i, 1) * X::row]; };
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        if (F::c(i, 2) >= 0) {
            d[i] = got[i];
            continue;
        }
        float2 w = F::c(i, 1) != 0 ? crossed(now, i) : v[i];
        w = pull_x(F::c(i, 0), w);
        // the transport outlet: got[i] holds the row's own population of plane p - 1
        if (!FLOWSET && outlet_r) w = a.ade_dirichlet ? p_all(a.gout_dev[i < 7 ? i : 0]) : got[i];
        d[i] = sel(i, Lr, up[F::opp(i)], w);
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const int cz = F::c(i, 2);
        if (cz < 0) {
            if (!FLOWSET) got[i] = v[i];
            continue;
        }
        if (i == 0) {
            got[0] = v[0];
            continue;
        }
        float2 w = F::c(i, 1) != 0 ? crossed(cz > 0 ? before : now, i) : (cz > 0 ? up[i] : v[i]);
        w = pull_x(F::c(i, 0), w);
        if (cz > 0 && inlet) {  // moving-wall bounce-back, or the transport inlet value
            if constexpr (FLOWSET) w = make_float2(v[F::opp(i)].x + a.bb_in[i], v[F::opp(i)].y + a.bb_in[i]);
            else w = p_all(a.gin_dev[i < 7 ? i : 0]);
        }
        got[i] = sel(i, L, v[F::opp(i)], w);
    }
#pragma unroll
    for (int i = 1; i < Q; ++i)
        if (F::c(i, 2) > 0) up[i] = v[i];
}

template <int SINK>
__global__ void __launch_bounds__(MARCH_ROWS * 32, 1) lbm_march_kernel(const StepArgs<3, float> a, const SweepShape s)
{
    using X = MarchExchange;
    using F = FlowSet<3>;
    using LK = Links<3>;
    using UU = UuForm<3, float, true, 7, SINK>;
    extern __shared__ __align__(16) char march_sh[];
    float2 *sh = reinterpret_cast<float2 *>(march_sh);
    const Geo &g = a.geo;
    const int nx = g.nx, ny = g.ny, nz = g.nz, zs = (int)g.zs;
    const int lane = (int)(threadIdx.x & 31);
    const int w = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int x0 = blockIdx.x * s.width, y = (int)blockIdx.y * (MARCH_ROWS - 2) - 1 + w;
    const int z0 = blockIdx.z * s.rows, z1 = min(z0 + s.rows, nz);
    const int x = x0 - 2 + 2 * lane;
    const int xc = min(x, (nx - 1) & ~1);  // columns beyond the lattice are not needed
    const bool inside = y >= 0 && y < ny;
    const bool writes = inside && w > 0 && w < MARCH_ROWS - 1;
    const bool inout = a.bc[2] == BC_INOUT;
    const int krow = (int)g.row0 + (inside ? y : 0) * g.px + xc;
    MarchRow v, d, got, up;
    float2 u[3] = {p_all(0.0f), p_all(0.0f), p_all(0.0f)};
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        got.f[i] = up.f[i] = v.f[i] = p_all(0.0f);
        if (i < 7) got.g[i] = up.g[i] = v.g[i] = p_all(0.0f);
    }
    // planes p0 .. z1 take step 1 (z1 only inside the lattice); L: links of plane p, Ln of the next, Lr of p - 1
    const int p0 = max(z0 - 1, 0);
    uint2 L = make_uint2(0, 0), Ln = make_uint2(0, 0), Lr = make_uint2(0, 0);
    if (inside) {
        L = ld_links(a.link + MFC_IDX(krow + p0 * zs, (int)g.plane - 1));
        if (p0 + 1 < nz) Ln = ld_links(a.link + MFC_IDX(krow + (p0 + 1) * zs, (int)g.plane - 1));
        march_load(a, v, krow + p0 * zs, L, __any_sync(0xffffffffu, (L.x | L.y) != 0u));
    }
    for (int p = p0; p <= z1; ++p) {
        // three buffers: a warp that is a turn ahead writes neither of the planes still being read
        float2 *mine = sh + p % 3 * X::plane + w * X::row + lane;
        const float2 *before = sh + (p + 2) % 3 * X::plane + w * X::row + lane;
        if (inside && p < nz) {
            const bool links = __any_sync(0xffffffffu, (L.x | L.y) != 0u);
            if (!links) {
#pragma unroll
                for (int i = 1; i < 19; ++i) {
                    v.f[i] = pull_x(F::c(i, 0), v.f[i]);
                    if (i < 7) v.g[i] = pull_x(F::c(i, 0), v.g[i]);
                }
            }
            march_collide<SINK>(a, v, L, links, u);
        } else if (inside && inout) {
            // beyond the outlet: the flow values from the velocity of the last plane (the turn before)
#pragma unroll
            for (int i = 1; i < 19; ++i)
                if (F::c(i, 2) == -1)
                    v.f[i] = make_float2(outlet_value<3, UU>(i, a.rho_out, u[0].x, u[1].x, u[2].x),
                                         outlet_value<3, UU>(i, a.rho_out, u[0].y, u[1].y, u[2].y));
        }
#pragma unroll
        for (int i = 1; i < 19; ++i) {
            if (F::c(i, 1) == 0) continue;
            mine[X::place(false, i) * 32] = v.f[i];
            if (i < 7) mine[X::place(true, i) * 32] = v.g[i];
        }
        __syncthreads();
        const int r = p - 1;
        if (writes) {
            march_arrive<19, 0, true>(a, d.f, got.f, up.f, v.f, mine, before, Lr, L, inout && p == 0, inout && r == nz - 1);
            march_arrive<7, LK::ADE_SELF, false>(a, d.g, got.g, up.g, v.g, mine, before, Lr, L, inout && p == 0, inout && r == nz - 1);
        }
        // the next plane's loads, under step 2's collision
        const uint2 Lq = Lr;
        Lr = L;
        L = Ln;
        if (inside && p + 1 <= z1 && p + 1 < nz) {
            march_load(a, v, krow + (p + 1) * zs, L, __any_sync(0xffffffffu, (L.x | L.y) != 0u));
            if (p + 2 < nz) Ln = ld_links(a.link + MFC_IDX(krow + (p + 2) * zs, (int)g.plane - 1));
        }
        if (writes && r >= z0) {
            float2 u2[3];
            march_collide<SINK>(a, d, Lq, true, u2);
            if (x >= x0 && x < min(x0 + s.width, nx)) {
                const int k = krow - xc + x + r * zs;
                const bool both = x + 1 < nx;
                row_store<19>(a, a.fdst, d.f, k, both);
                row_store<7>(a, a.gdst, d.g, k, both);
                if (inout && (r == 0 || r == nz - 1)) {
                    if (!(Lq.x & (1u << LK::FLOW_SELF)))
                        row_flow_ends<float, UU, true, false>(a, x, y, r, k, Lq.x, [&](int i) { return d.f[i].x; }, u2[0].x, u2[1].x, u2[2].x);
                    if (both && !(Lq.y & (1u << LK::FLOW_SELF)))
                        row_flow_ends<float, UU, true, false>(a, x + 1, y, r, k + 1, Lq.y, [&](int i) { return d.f[i].y; }, u2[0].y, u2[1].y, u2[2].y);
                    if (!(Lq.x & (1u << LK::ADE_SELF))) row_ade_ends<float, true>(a, r, k, Lq.x, d.g[6].x);
                    if (both && !(Lq.y & (1u << LK::ADE_SELF))) row_ade_ends<float, true>(a, r, k + 1, Lq.y, d.g[6].y);
                }
            }
        }
    }
}

}  // namespace mfc
