// Plain steps of 3-D lattices, two neighbouring nodes of a row per thread.
//
// The one-node kernel (step_node) spends its time on instructions and latency as much as on memory: 695
// warp instructions per 32 nodes in FP32, an address and a load per population and node.  Here a thread
// takes nodes (x, x + 1): populations that stay in their column come with one 64-bit load (32-bit in FP16
// storage) and all leave with one, and the collision runs on both nodes at once with paired FP32
// instructions, in the rounding of the kernels that it replaces (lbm_collide.cuh).  Threads are numbered
// through the pairs of a plane, so a row that is no multiple of a warp leaves no lanes idle.
// A warp with no link to a wall or a sink and no consumption node skips the selection of bounced-back
// sources; a warp with one takes every population with one load per node, from the source node or from the
// node's own opposite population.
#pragma once

#include "lbm_sweep.cuh"

namespace mfc {

enum : int { ROW_BLOCK = 128 };

// Planes are taken in alternating order (RowPairs::back) where a step reads and writes more than this, three
// quarters of the L2; below, all of it stays there in any order, and the outlet plane is better taken first
// (64x40x48 6.04 us per step, 6.16 in turn; 97x71x83 in FP16, 60 MB, the same).
constexpr long long BACK_BYTES = 96ll << 20;

// Resident blocks per SM.  FP32 coupled steps gather both sets before the first collision (102 registers, 5
// blocks: 137.4 us per 256x128x128 step, against 141.3 one set after the other at 8 blocks; the one-node
// kernel took 140); FP16 ones do better with more warps and one set at a time (99.6 us against 104 with
// both at 6 blocks; two rows per thread took 108.8), as do flow and transport alone (128x64x96: 30.5 us for
// the two, against 31.5 at 5 blocks and 33.5 with one node per thread).  Small lattices gain the most, from
// ghost values written from registers: 24x16x16 10.6 -> 4.6 us, 64x40x48 11.4 -> 5.9.
template <typename ST, bool COUPLED> struct RowOccupancy {
    static constexpr bool both_sets = COUPLED && sizeof(ST) == 4;
    static constexpr int blocks = both_sets ? 5 : 8;
};

// Gather one set's populations of nodes k and k + 1.  at_in, at_out: the nodes are on the inlet or outlet
// layer and take its values themselves (reader form).
template <int Q, int SELF, bool FLOWSET, bool READER, typename ST, typename D>
__device__ __forceinline__ void row_gather(const StepArgs<3, ST> &a, const ST *src, D &d, int k, uint2 L, bool links,
                                           bool at_in, bool at_out)
{
    using F = FlowSet<3>;  // the transport set is its first directions
    const int P = (int)a.geo.plane, px = a.geo.px, zs = (int)a.geo.zs;
    if (links) {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const int off = F::c(i, 0) + F::c(i, 1) * px + F::c(i, 2) * zs;
            const bool inj = READER && F::c(i, 2) == 1 && at_in;
            const bool out_v = READER && !FLOWSET && F::c(i, 2) == -1 && at_out;
            const int own = F::opp(i) * P;
            const int from = inj ? own : i * P - (out_v ? 0 : off);
            const bool b0 = i > 0 && ((L.x >> (SELF + i)) & 1u), b1 = i > 0 && ((L.y >> (SELF + i)) & 1u);
            float v0 = ld(src + MFC_IDX(k + (b0 ? own : from), Q * P)), v1 = ld(src + MFC_IDX(k + 1 + (b1 ? own : from), Q * P));
            if (inj) {
                if constexpr (FLOWSET) {
                    v0 = b0 ? v0 : v0 + a.bb_in[i];
                    v1 = b1 ? v1 : v1 + a.bb_in[i];
                } else {
                    v0 = b0 ? v0 : a.gin_dev[i < 7 ? i : 0];
                    v1 = b1 ? v1 : a.gin_dev[i < 7 ? i : 0];
                }
            }
            if (out_v && a.ade_dirichlet) {
                v0 = b0 ? v0 : a.gout_dev[i < 7 ? i : 0];
                v1 = b1 ? v1 : a.gout_dev[i < 7 ? i : 0];
            }
            d[i] = make_float2(v0, v1);
        }
    } else {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const int off = F::c(i, 0) + F::c(i, 1) * px + F::c(i, 2) * zs;
            const bool inj = READER && F::c(i, 2) == 1 && at_in;
            const bool out_v = READER && !FLOWSET && F::c(i, 2) == -1 && at_out;
            const int o = k + (inj ? F::opp(i) * P : i * P - (out_v ? 0 : off));
            if (F::c(i, 0) == 0) {
                d[i] = pair_value(ld_pair(src + MFC_IDX(o, Q * P - 1)));
            } else {  // from the columns (x - 1, x) or (x + 1, x + 2): unaligned
                const float v0 = ld(src + MFC_IDX(o, Q * P - 1));
                d[i] = make_float2(v0, ld(src + MFC_IDX(o + 1, Q * P)));
            }
            if (inj) {
                if constexpr (FLOWSET) d[i] = make_float2(d[i].x + a.bb_in[i], d[i].y + a.bb_in[i]);
                else d[i] = p_all(a.gin_dev[i < 7 ? i : 0]);
            }
            if (out_v && a.ade_dirichlet) d[i] = p_all(a.gout_dev[i < 7 ? i : 0]);
        }
    }
}

// Store one set's pairs (the second node only where it exists).
template <int Q, typename ST, typename D>
__device__ __forceinline__ void row_store(const StepArgs<3, ST> &a, ST *dst, const D &d, int k, bool both)
{
    const int P = (int)a.geo.plane;
    if (both) {
#pragma unroll
        for (int i = 0; i < Q; ++i) st_pair(dst + MFC_IDX(i * P + k, Q * P - 1), d[i]);
    } else {
#pragma unroll
        for (int i = 0; i < Q; ++i) st(dst + MFC_IDX(i * P + k, Q * P), d[i].x);
    }
}

// Ghost cells of the written flow populations that belong to node (x, y, z) at the inlet or the outlet, from
// its post-collision populations v and velocity in registers: reading them back after the store costs a
// round trip to L2 per value, which a small lattice's step waits for.
template <typename ST, typename FORMS, bool WRITER, typename V>
__device__ __forceinline__ void row_flow_ends(const StepArgs<3, ST> &a, int x, int y, int z, int k, uint32_t L, const V &v,
                                              float u0, float u1, float u2)
{
    using F = FlowSet<3>;
    const Geo &g = a.geo;
    const int P = (int)g.plane, px = g.px, zs = (int)g.zs;
    if (WRITER && z == 0 && !a.cut[0]) {
#pragma unroll
        for (int i = 1; i < F::Q; ++i)
            if (F::c(i, 2) == 1 && !((L >> i) & 1u))  // the node's own next pull
                st(a.fdst + MFC_IDX(i * P + k - F::c(i, 0) - F::c(i, 1) * px - zs, F::Q * P), v(F::opp(i)) + a.bb_in[i]);
    }
    if (z == g.nz - 1 && !a.cut[1]) {
#pragma unroll
        for (int i = 1; i < F::Q; ++i) {
            if (F::c(i, 2) != -1) continue;
            const int rx = x + F::c(i, 0), ry = y + F::c(i, 1);
            if (rx >= 0 && rx < g.nx && ry >= 0 && ry < g.ny)
                st(a.fdst + MFC_IDX(i * P + k + zs, F::Q * P), outlet_value<3, FORMS>(i, a.rho_out, u0, u1, u2));
        }
    }
}

// The same for the transport populations (v6: the node's population leaving the outlet inwards).
template <typename ST, bool WRITER>
__device__ __forceinline__ void row_ade_ends(const StepArgs<3, ST> &a, int z, int k, uint32_t L, float v6)
{
    const int P = (int)a.geo.plane, zs = (int)a.geo.zs;
    if (!WRITER) return;
    if (z == 0 && !a.cut[0] && !((L >> (Links<3>::ADE_SELF + 5)) & 1u)) st(a.gdst + MFC_IDX(5 * P + k - zs, 7 * P), a.gin_dev[5]);
    if (z == a.geo.nz - 1 && !a.cut[1]) st(a.gdst + MFC_IDX(6 * P + k + zs, 7 * P), a.ade_dirichlet ? a.gout_dev[6] : v6);
}

// Lattices with a periodic axis: the periodic images of node (x, y, z), and the images of the outlet values,
// read back from the node's stored populations.  SET: the velocity set, Q planes at pop.
template <typename SET, typename ST, typename FORMS, bool FLOWSET, bool WRITER>
__device__ __noinline__ void row_images(const StepArgs<3, ST> &a, ST *pop, int x, int y, int z, int k, float u0, float u1,
                                        float u2)
{
    const Geo &g = a.geo;
    const bool images = on_periodic_boundary<3>(g, a.bc, x, y, z);
    const bool outlet = a.bc[2] == BC_INOUT && z == g.nz - 1 && !a.cut[1] && (FLOWSET || WRITER);
#pragma unroll
    for (int i = 1; i < SET::Q; ++i) {
        if (images) ghost_images<3, SET, ST>(g, a.bc, pop, i, x, y, z, false, ldplain(pop + (long long)i * g.plane + k));
        if (outlet && SET::c(i, 2) == -1) {
            float v;
            if constexpr (FLOWSET) v = outlet_value<3, FORMS>(i, a.rho_out, u0, u1, u2);
            else v = a.ade_dirichlet ? a.gout_dev[i] : ldplain(pop + (long long)i * g.plane + k);
            ghost_images<3, SET, ST>(g, a.bc, pop, i, x, y, g.nz, true, v);
        }
    }
}

// Pairs per row and the multiplier ceil(2^32 / n) of the division by it: the quotient's estimate is at
// most one too large (q < 2^31), and never too small.
struct RowPairs {
    int n;       // pairs per row
    uint32_t m;  // ceil(2^32 / n)
    // Planes from the last to the first, in every other step: the step before wrote its last planes last, and
    // reading those first finds them in the L2.  us per step, always upwards and in turn: 97x71x83 27.3 and
    // 23.4, 128x64x96 30.1 and 27.7, 128x128x128 73.0 and 70.3 (FP16 58.5 and 53.6), 256x128x128 138.1 and
    // 135.7 (FP16 100.8 and 97.3).  (Loads marked evict-first besides lose more: neighbours' rows share lines.)
    int back;
};

// One plain step of pair q (numbered along the rows) of plane z.
template <typename ST, bool FLOW, bool ADE, int SINK, int FORM>
__device__ __forceinline__ void row_step(const StepArgs<3, ST> &a, const RowPairs &rp, int q, int z)
{
    using F = FlowSet<3>;
    using LK = Links<3>;
    using UU = UuForm<3, ST, ADE, 7, SINK>;
    constexpr bool READER = ReaderForm<3, ST, 7, SINK>::value, BOTH = RowOccupancy<ST, FLOW && ADE>::both_sets;
    const Geo &g = a.geo;
    const int P = (int)g.plane;
    int y = rp.n > 1 ? (int)__umulhi((uint32_t)q, rp.m) : q;
    if (y * rp.n > q) --y;
    const bool valid = y < g.ny;
    y = valid ? y : g.ny - 1;  // the last warp's idle lanes repeat the last pair and store nothing
    const int x = valid ? 2 * (q - y * rp.n) : 2 * (rp.n - 1);
    const int k = (int)g.row0 + z * (int)g.zs + y * g.px + x;
    const bool both = x + 1 < g.nx;
    const uint2 L = __ldg(reinterpret_cast<const uint2 *>(a.link + MFC_IDX(k, P - 1)));
    const bool links = __any_sync(0xffffffffu, (L.x | L.y) != 0u);
    const bool at_in = READER && a.bc[2] == BC_INOUT && z == 0 && !a.cut[0];
    const bool at_out = READER && a.bc[2] == BC_INOUT && z == g.nz - 1 && !a.cut[1];
    // the node's ghost cells: at the ends of an inlet/outlet axis, and on any boundary of a lattice with a
    // periodic axis
    const bool periodic = a.bc[0] == BC_PERIODIC || a.bc[1] == BC_PERIODIC || a.bc[2] == BC_PERIODIC;
    const bool ends = valid && a.bc[2] == BC_INOUT && (z == 0 || z == g.nz - 1);
    float2 u[3] = {p_all(0.0f), p_all(0.0f), p_all(0.0f)};
    float2 e[7];
    if constexpr (FLOW) {
        float2 d[F::Q], rho;
        row_gather<F::Q, 0, true, READER>(a, a.fsrc, d, k, L, links, at_in, at_out);
        if constexpr (BOTH) row_gather<7, LK::ADE_SELF, false, READER>(a, a.gsrc, e, k, L, links, at_in, at_out);
        collide_flow<3, ST, FORM, UU::collision>(d, a.omega, u, rho);
        if (valid) row_store<F::Q>(a, a.fdst, d, k, both);
        const bool o0 = valid && !(L.x & (1u << LK::FLOW_SELF)), o1 = valid && both && !(L.y & (1u << LK::FLOW_SELF));
        if (ends) {
            if (o0) row_flow_ends<ST, UU, !READER>(a, x, y, z, k, L.x, [&](int i) { return d[i].x; }, u[0].x, u[1].x, u[2].x);
            if (o1) row_flow_ends<ST, UU, !READER>(a, x + 1, y, z, k + 1, L.y, [&](int i) { return d[i].y; }, u[0].y, u[1].y, u[2].y);
        }
        if (periodic) {
            if (o0) row_images<F, ST, UU, true, !READER>(a, a.fdst, x, y, z, k, u[0].x, u[1].x, u[2].x);
            if (o1) row_images<F, ST, UU, true, !READER>(a, a.fdst, x + 1, y, z, k + 1, u[0].y, u[1].y, u[2].y);
        }
    }
    if constexpr (ADE) {
        if constexpr (!BOTH) row_gather<7, LK::ADE_SELF, false, READER>(a, a.gsrc, e, k, L, links, at_in, at_out);
        if constexpr (!FLOW) {  // the frozen velocity, at rest on flow-blocked nodes
#pragma unroll
            for (int ax = 0; ax < 3; ++ax) {
                u[ax] = ld_pair(a.fld_u + MFC_IDX(ax * P + k, 3 * P - 1));
                if (L.x & (1u << LK::FLOW_SELF)) u[ax].x = 0.0f;
                if (L.y & (1u << LK::FLOW_SELF)) u[ax].y = 0.0f;
            }
        }
        const float2 us = p_all(a.u_scale);
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) u[ax] = p_mul(u[ax], us);
        collide_ade<3, ST, 7, SINK, FORM>(e, u, a.omega_c, a.c_ref, a.k_half, links, L.x & (1u << LK::SINK) ? a.k_sink : 0.0f,
                                          L.y & (1u << LK::SINK) ? a.k_sink : 0.0f);
        if (valid) row_store<7>(a, a.gdst, e, k, both);
        const bool o0 = valid && !(L.x & (1u << LK::ADE_SELF)), o1 = valid && both && !(L.y & (1u << LK::ADE_SELF));
        if (ends) {
            if (o0) row_ade_ends<ST, !READER>(a, z, k, L.x, e[6].x);
            if (o1) row_ade_ends<ST, !READER>(a, z, k + 1, L.y, e[6].y);
        }
        if (periodic) {
            if (o0) row_images<AdeSet<3>, ST, UU, false, !READER>(a, a.gdst, x, y, z, k, 0.0f, 0.0f, 0.0f);
            if (o1) row_images<AdeSet<3>, ST, UU, false, !READER>(a, a.gdst, x + 1, y, z, k + 1, 0.0f, 0.0f, 0.0f);
        }
    }
}

// One plain step of a lattice: grid (pairs of a plane / block, nz); the outlet plane first, whose ghost work is
// longest.
template <typename ST, bool FLOW, bool ADE, int SINK, int FORM>
__global__ void __launch_bounds__(ROW_BLOCK, RowOccupancy<ST, FLOW && ADE>::blocks)
    lbm_row_kernel(const StepArgs<3, ST> a, const RowPairs rp)
{
    const int z = rp.back ? (int)(gridDim.y - 1 - blockIdx.y) : blockIdx.y == 0 ? (int)gridDim.y - 1 : (int)blockIdx.y - 1;
    const int b = (int)(rp.back ? gridDim.x - 1 - blockIdx.x : blockIdx.x);
    row_step<ST, FLOW, ADE, SINK, FORM>(a, rp, b * ROW_BLOCK + (int)threadIdx.x, z);
}

__host__ __device__ __forceinline__ RowPairs row_pairs(int nx, int back = 0)
{
    const int n = (nx + 1) / 2;
    return {n, n > 1 ? (uint32_t)(((1ull << 32) + n - 1) / n) : 0u, back};
}

// One plain coupled step of many lattices (batches): a fixed grid walks the table of chunks of ROW_BLOCK pairs
// (slot, first pair, -, plane); the argument block of a chunk's instance is copied to shared memory.
template <typename ST>
__global__ void __launch_bounds__(ROW_BLOCK, RowOccupancy<ST, true>::blocks) lbm_batch_row_kernel(const BatchArgs<3, ST> b)
{
    static_assert(sizeof(StepArgs<3, ST>) % 4 == 0, "argument block copied as 32-bit words");
    __shared__ StepArgs<3, ST> sa;
    constexpr int WORDS = (int)(sizeof(StepArgs<3, ST>) / 4);
    const int n = *b.ntiles;
    // the order of RowPairs::back (a mix of 3.4 million nodes, FP32: 83.5 -> 79.0 ms for 800 steps)
    const bool back = b.parity && n > (int)(BACK_BYTES / (2 * ROW_BLOCK * 26 * 2 * sizeof(ST)));
    int cur = -1;
    RowPairs rp = {1, 0, 0};
    for (int t = blockIdx.x; t < n; t += gridDim.x) {
        const Tile tile = b.tiles[back ? n - 1 - t : t];
        if (tile.slot != cur) {  // uniform over the block
            __syncthreads();     // the previous instance's arguments are no longer read
            const uint32_t *src = reinterpret_cast<const uint32_t *>(b.inst + 2 * tile.slot + b.parity);
            uint32_t *dst = reinterpret_cast<uint32_t *>(&sa);
            for (int w = threadIdx.x; w < WORDS; w += ROW_BLOCK) dst[w] = src[w];
            __syncthreads();
            cur = tile.slot;
            rp = row_pairs(sa.geo.nx);
        }
        row_step<ST, true, true, SINK_RUNTIME, SCALAR_FORM>(sa, rp, tile.x0 + (int)threadIdx.x, tile.z);
    }
}

}  // namespace mfc
