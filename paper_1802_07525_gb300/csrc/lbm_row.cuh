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

// Resident blocks per SM.  FP32 coupled steps gather both sets before the first collision (96 registers, 5
// blocks: 137.4 us per 256x128x128 step, against 141.3 one set after the other at 8 blocks; the one-node
// kernel took 140); FP16 ones do better with more warps and one set at a time (99.6 us against 104 with
// both at 6 blocks; two rows per thread took 108.8), as do flow and transport alone (128x64x96: 30.5 us for
// the two, against 31.5 at 5 blocks and 33.5 with one node per thread).  At 8 blocks FP32 flow alone spills 16
// bytes (256x128x128 98.9 us per step; at 6, without spills, 101.8), the FP16 batch kernel 32.  Small lattices gain the most, from
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

// The sides of the lattice that a node lies on, and what a population that leaves across one of them meets.
// On a periodic axis the neighbour that receives it pulls it through the ghost cell one lattice length away
// (its image: at most one per direction, shifted along every axis that the direction leaves by); other sides
// have no image.
struct RowSides {
    uint32_t at, shut;  // bit 2 axis + (0: low, 1: high): the node is on that side; the side is not periodic
    int nx, ny, nz;     // shifts along the axes in elements
};
template <typename ST> __device__ __forceinline__ RowSides row_sides(const StepArgs<3, ST> &a, int x, int y, int z)
{
    const Geo &g = a.geo;
    RowSides s;
    s.at = (x == 0 ? 1u : 0u) | (x == g.nx - 1 ? 2u : 0u) | (y == 0 ? 4u : 0u) | (y == g.ny - 1 ? 8u : 0u) |
           (z == 0 ? 16u : 0u) | (z == g.nz - 1 ? 32u : 0u);
    s.shut = (a.bc[0] == BC_PERIODIC ? 0u : 3u) | (a.bc[1] == BC_PERIODIC ? 0u : 12u) | (a.bc[2] == BC_PERIODIC ? 0u : 48u);
    s.nx = g.nx;
    s.ny = g.ny * g.px;
    s.nz = g.nz * (int)g.zs;
    return s;
}
// the sides that direction i leaves by, as in RowSides::at
__host__ __device__ constexpr uint32_t row_exits(int i)
{
    uint32_t m = 0;
    for (int ax = 0; ax < 3; ++ax) {
        if (FlowSet<3>::c(i, ax) < 0) m |= 1u << (2 * ax);
        if (FlowSet<3>::c(i, ax) > 0) m |= 2u << (2 * ax);
    }
    return m;
}
// Offset from a node to the cell through which its population i is pulled next: out is those of the
// direction's exits that the node is on.
__device__ __forceinline__ int row_shift(const RowSides &s, int i, uint32_t out)
{
    using F = FlowSet<3>;  // the transport set is its first directions
    int o = 0;
    if (F::c(i, 0) != 0 && (out & 3u)) o -= F::c(i, 0) * s.nx;
    if (F::c(i, 1) != 0 && (out & 12u)) o -= F::c(i, 1) * s.ny;
    if (F::c(i, 2) != 0 && (out & 48u)) o -= F::c(i, 2) * s.nz;
    return o;
}

// Ghost cells of one set's written populations across periodic axes, from the node's post-collision populations
// v in registers.  (Written back from memory by the general loops of ghost_images, and asked for at every node
// by a call, they cost more than the step: us per step of 128x128x128, before and now, periodic along y 105.5 and
// 71.9 in FP32, 87.0 and 57.4 in FP16, along x and y 281 and 74.4, 230 and 57.5; between walls 67.2 and 51.7.)
template <int Q, typename ST, typename V>
__device__ __forceinline__ void row_images(const StepArgs<3, ST> &a, ST *pop, const RowSides &s, int k, const V &v)
{
    const int P = (int)a.geo.plane;
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        const uint32_t out = row_exits(i) & s.at;
        if (out && !(out & s.shut)) st(pop + MFC_IDX(i * P + k + row_shift(s, i, out), Q * P), v(i));
    }
}

// Ghost cells of the written flow populations that belong to node (x, y, z) at the inlet or the outlet, from
// its post-collision populations v and velocity in registers: reading them back after the store costs a
// round trip to L2 per value, which a small lattice's step waits for.
template <typename ST, typename FORMS, bool WRITER, bool PERIODIC, typename V>
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
            if constexpr (PERIODIC) {
                const RowSides s = row_sides(a, x, y, z);
                const uint32_t out = row_exits(i) & s.at & 15u;  // the layer beyond the outlet has the node's sides of x and y
                if (!(out & s.shut))
                    st(a.fdst + MFC_IDX(i * P + k + zs + row_shift(s, i, out), F::Q * P), outlet_value<3, FORMS>(i, a.rho_out, u0, u1, u2));
            } else {
                const int rx = x + F::c(i, 0), ry = y + F::c(i, 1);
                if (rx >= 0 && rx < g.nx && ry >= 0 && ry < g.ny)
                    st(a.fdst + MFC_IDX(i * P + k + zs, F::Q * P), outlet_value<3, FORMS>(i, a.rho_out, u0, u1, u2));
            }
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

// One plain step of pair q (numbered along the rows) of plane z.  PERIODIC: whether any axis may be periodic
// (without, the code for images is left out: its registers cost FP16 flow and transport alone 2%).
template <typename ST, bool FLOW, bool ADE, int SINK, int FORM, bool PERIODIC>
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
    const bool periodic = PERIODIC && (a.bc[0] == BC_PERIODIC || a.bc[1] == BC_PERIODIC || a.bc[2] == BC_PERIODIC);
    const bool ends = valid && a.bc[2] == BC_INOUT && (z == 0 || z == g.nz - 1);
    const bool images = valid && periodic && (x == 0 || x + 2 >= g.nx || y == 0 || y == g.ny - 1 || z == 0 || z == g.nz - 1);
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
            // FP32 flow alone, one node after the other: written out twice, more spills (flow step of 97x71x83 19.4
            // against 18.5 us); the other kernels are faster written out (FP16 256x128x128 95.1 against 96.6 us)
            constexpr int NODES = sizeof(ST) == 4 && !ADE ? 1 : 2;
#pragma unroll NODES
            for (int n = 0; n < 2; ++n)
                if (n ? o1 : o0)
                    row_flow_ends<ST, UU, !READER, PERIODIC>(a, x + n, y, z, k + n, n ? L.y : L.x, [&](int i) { return n ? d[i].y : d[i].x; },
                                                             n ? u[0].y : u[0].x, n ? u[1].y : u[1].x, n ? u[2].y : u[2].x);
        }
        if (images) {
            if (o0) row_images<F::Q>(a, a.fdst, row_sides(a, x, y, z), k, [&](int i) { return d[i].x; });
            if (o1) row_images<F::Q>(a, a.fdst, row_sides(a, x + 1, y, z), k + 1, [&](int i) { return d[i].y; });
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
        if (images) {
            if (o0) row_images<7>(a, a.gdst, row_sides(a, x, y, z), k, [&](int i) { return e[i].x; });
            if (o1) row_images<7>(a, a.gdst, row_sides(a, x + 1, y, z), k + 1, [&](int i) { return e[i].y; });
        }
    }
}

// One plain step of a lattice: grid (pairs of a plane / block, nz); the outlet plane first, whose ghost work is
// longest.
template <typename ST, bool FLOW, bool ADE, int SINK, int FORM, bool PERIODIC>
__global__ void __launch_bounds__(ROW_BLOCK, RowOccupancy<ST, FLOW && ADE>::blocks)
    lbm_row_kernel(const StepArgs<3, ST> a, const RowPairs rp)
{
    const int z = rp.back ? (int)(gridDim.y - 1 - blockIdx.y) : blockIdx.y == 0 ? (int)gridDim.y - 1 : (int)blockIdx.y - 1;
    const int b = (int)(rp.back ? gridDim.x - 1 - blockIdx.x : blockIdx.x);
    // warps beyond the plane's last pair leave (2x2x20000 in FP32, a pair in two lanes: 73.5 -> 34.2 us per step)
    if (b * ROW_BLOCK + (int)(threadIdx.x & ~31u) >= rp.n * a.geo.ny) return;
    row_step<ST, FLOW, ADE, SINK, FORM, PERIODIC>(a, rp, b * ROW_BLOCK + (int)threadIdx.x, z);
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
    bool periodic = false;
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
            periodic = sa.bc[0] == BC_PERIODIC || sa.bc[1] == BC_PERIODIC || sa.bc[2] == BC_PERIODIC;
        }
        if (periodic) row_step<ST, true, true, SINK_RUNTIME, SCALAR_FORM, true>(sa, rp, tile.x0 + (int)threadIdx.x, tile.z);
        else row_step<ST, true, true, SINK_RUNTIME, SCALAR_FORM, false>(sa, rp, tile.x0 + (int)threadIdx.x, tile.z);
    }
}

}  // namespace mfc
