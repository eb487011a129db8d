// Launchers of the step, batch-step and ghost-fill kernels for one dimension (MFC_DIM), one
// storage type (MFC_ST: float, __half, or double for the FP64 instantiation) and one transport
// velocity set (MFC_AQ, default D2Q5 / D3Q7), included
// by one translation unit per combination so that the instantiations compile in parallel.  The
// batch launchers exist for the default transport sets only (MFC_BATCH_FN defined).
#include <string.h>

#include "lbm_pair.cuh"
#include "lbm_march.cuh"
#include "lbm_row.cuh"
#include "lbm_sweep.cuh"
#include "mfc_internal.h"

#ifndef MFC_DIM
#error "MFC_DIM must be defined"
#endif

namespace mfc {

namespace {

using ST = MFC_ST;
constexpr int D = MFC_DIM;
#ifdef MFC_AQ
constexpr int AQ = MFC_AQ;
#else
constexpr int AQ = default_aq<D>();
#endif
using Args = StepArgs<D, ST, AQ>;

template <bool FLOW, bool ADE, int SINK>
cudaError_t launch_sink(const Args &a, const StepHost &h, cudaStream_t s)
{
    const dim3 grid((unsigned)h.grid, (unsigned)h.geo.ny, (unsigned)h.geo.nz);
    switch (h.mode) {
    case MODE_PLAIN:
        // one plain step: 32-bit element offsets where the arrays allow them, and the kernel of one_step_kernel
        if constexpr (D == 3 && !std::is_same<ST, double>::value) {
            if (h.kernel == MFC_KERNEL_ROW) {
                constexpr int FORM = FLOW && ADE && std::is_same<ST, __half>::value ? PAIR_FORM : SCALAR_FORM;
                const RowPairs rp = row_pairs(h.geo.nx, h.back);
                const dim3 pairs((unsigned)(((long long)rp.n * h.geo.ny + ROW_BLOCK - 1) / ROW_BLOCK), (unsigned)h.geo.nz);
                const bool periodic = h.bc[0] == BC_PERIODIC || h.bc[1] == BC_PERIODIC || h.bc[2] == BC_PERIODIC;
                if (periodic) lbm_row_kernel<ST, FLOW, ADE, SINK, FORM, true><<<pairs, ROW_BLOCK, 0, s>>>(a, rp);
                else lbm_row_kernel<ST, FLOW, ADE, SINK, FORM, false><<<pairs, ROW_BLOCK, 0, s>>>(a, rp);
                break;
            }
        } else if constexpr (D == 2 && FLOW && ADE && AQ == default_aq<D>() && PairedStep<D, ST>::value) {
            if (h.kernel == MFC_KERNEL_PAIR) {
                const dim3 pairs((unsigned)h.grid, (unsigned)((h.geo.ny + 1) / 2));
                lbm_pair_kernel<ST, SINK><<<pairs, h.block, 0, s>>>(a);
                break;
            }
        } else if (h.idx32) {
            lbm_step_kernel<D, ST, FLOW, ADE, MODE_PLAIN, AQ, SINK, true><<<grid, h.block, 0, s>>>(a);
            break;
        }
        lbm_step_kernel<D, ST, FLOW, ADE, MODE_PLAIN, AQ, SINK><<<grid, h.block, 0, s>>>(a);
        break;
    case MODE_SWEEP:
        if constexpr (D == 2 && !std::is_same<ST, double>::value) {
            // the rounding of the plain step it stands for
            constexpr int FORM = FLOW && ADE && AQ == default_aq<D>() && PairedStep<D, ST>::value ? PAIR_FORM : SCALAR_FORM;
            const dim3 tiles((unsigned)h.sweep.ntx, (unsigned)h.sweep.strips);
            if (h.sweep.tile) {
                const int warps = h.sweep.rows + 2 * h.sweep.steps;
                constexpr int row = 2 * TileExchange<FLOW, ADE, AQ>::row * (int)sizeof(float2);
                auto kernel = lbm_tile_kernel<ST, FLOW, ADE, AQ, SINK, FORM>;
                const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                           TILE_WARPS * row);
                if (e != cudaSuccess) return e;
                kernel<<<tiles, 32 * warps, warps * row, s>>>(a, h.sweep);
                break;
            }
            constexpr int most = SweepSteps<AQ, FLOW && ADE>::value;
            if (h.sweep.steps == most) lbm_sweep_kernel<ST, FLOW, ADE, AQ, SINK, FORM, most><<<tiles, 32, 0, s>>>(a, h.sweep);
            else lbm_sweep_kernel<ST, FLOW, ADE, AQ, SINK, FORM, 2><<<tiles, 32, 0, s>>>(a, h.sweep);
            break;
        }
        if constexpr (D == 3 && std::is_same<ST, float>::value && FLOW && ADE) {
            static_assert(!ReaderBoundaries<3, float>::step, "step 1 reads the ghost cells of the writer form");
            auto kernel = lbm_march_kernel<SINK>;
            const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, MarchExchange::bytes);
            if (e != cudaSuccess) return e;
            const dim3 columns((unsigned)h.sweep.ntx, (unsigned)((h.geo.ny + MARCH_ROWS - 3) / (MARCH_ROWS - 2)),
                               (unsigned)h.sweep.strips);
            kernel<<<columns, MARCH_ROWS * 32, MarchExchange::bytes, s>>>(a, h.sweep);
            break;
        }
        return cudaErrorInvalidValue;
    case MODE_WRITE: lbm_step_kernel<D, ST, FLOW, ADE, MODE_WRITE, AQ, SINK><<<grid, h.block, 0, s>>>(a); break;
    default: lbm_step_kernel<D, ST, FLOW, ADE, MODE_CHECK, AQ, SINK><<<grid, h.block, 0, s>>>(a); break;
    }
    return cudaGetLastError();
}

// Steps with transport take the kernels of the lattice's consumption law; flow-only steps have
// no consumption.
template <bool FLOW, bool ADE>
cudaError_t launch_mode(const Args &a, const StepHost &h, cudaStream_t s)
{
    if constexpr (ADE) {
        if (h.k_half > 0.0) return launch_sink<FLOW, ADE, SINK_MONOD>(a, h, s);
    }
    return launch_sink<FLOW, ADE, SINK_LINEAR>(a, h, s);
}

Args make_args(const StepHost &h)
{
    Args a;
    a.geo = h.geo;
    for (int i = 0; i < 3; ++i) a.bc[i] = h.bc[i];
    a.fsrc = static_cast<const ST *>(h.fsrc);
    a.fdst = static_cast<ST *>(h.fdst);
    a.gsrc = static_cast<const ST *>(h.gsrc);
    a.gdst = static_cast<ST *>(h.gdst);
    a.link = static_cast<const typename Links<D, AQ>::T *>(h.link);
    using R = typename Args::R;
    a.fld_rho = static_cast<R *>(h.fld_rho);
    a.fld_u = static_cast<R *>(h.fld_u);
    a.fld_c = static_cast<R *>(h.fld_c);
    a.partials = h.partials;
    a.omega = (R)h.omega; a.omega_c = (R)h.omega_c; a.k_sink = (R)h.k_sink; a.u_scale = (R)h.u_scale;
    a.rho_out = (R)h.rho_out; a.c_ref = (R)h.c_ref; a.ade_dirichlet = h.ade_dirichlet;
    a.cut[0] = h.cut[0];
    a.cut[1] = h.cut[1];
    a.bounds_err = h.bounds_err;
    a.k_half = (R)h.k_half;
    for (int i = 0; i < Args::QF; ++i) a.bb_in[i] = (R)h.bb_in[i];
    for (int i = 0; i < Args::QA; ++i) {
        a.gin_dev[i] = (R)h.gin_dev[i];
        a.gout_dev[i] = (R)h.gout_dev[i];
    }
    return a;
}

}  // namespace

cudaError_t MFC_STEP_FN(StepHost &h, cudaStream_t s)
{
    const Args a = make_args(h);
    h.nblocks = h.grid * h.geo.ny * h.geo.nz;
    switch (h.kind) {
    case KIND_COUPLED: return launch_mode<true, true>(a, h, s);
    case KIND_FLOW: return launch_mode<true, false>(a, h, s);
    default: return launch_mode<false, true>(a, h, s);
    }
}

#ifdef MFC_BATCH_FN
size_t MFC_ARGS_FN(const StepHost &h, void *out)
{
    const Args a = make_args(h);
    if (out) memcpy(out, &a, sizeof a);
    return sizeof a;
}

// Plain steps of the instances in the sweep table: several at once in 2-D, one in 3-D.
template <typename S> cudaError_t launch_batch_sweep(const BatchArgs<2, S> &b, const BatchHost &h, cudaStream_t s)
{
    auto kernel = lbm_batch_tile_kernel<S>;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, BatchSweep<S>::exchange);
    if (e != cudaSuccess) return e;
    kernel<<<h.grid, 32 * (BatchSweep<S>::rows + 2 * h.steps), BatchSweep<S>::exchange, s>>>(b, h.steps);
    return cudaGetLastError();
}
template <typename S> cudaError_t launch_batch_sweep(const BatchArgs<3, S> &b, const BatchHost &h, cudaStream_t s)
{
    lbm_batch_row_kernel<S><<<h.grid, ROW_BLOCK, 0, s>>>(b);
    return cudaGetLastError();
}

// One plain step of 2-D instances by row segments (3-D ones all take the row kernel).
template <typename S> cudaError_t launch_batch_plain(const BatchArgs<2, S> &b, const BatchHost &h, cudaStream_t s)
{
    lbm_batch_kernel<2, S, true, true, MODE_PLAIN><<<h.grid, h.block, 0, s>>>(b);
    return cudaGetLastError();
}
template <typename S> cudaError_t launch_batch_plain(const BatchArgs<3, S> &, const BatchHost &, cudaStream_t)
{
    return cudaErrorInvalidValue;
}

// Coupled steps only: a batch advances flow and transport of every instance together.
cudaError_t MFC_BATCH_FN(const BatchHost &h, cudaStream_t s)
{
    BatchArgs<D, ST> b;
    b.inst = static_cast<const StepArgs<D, ST> *>(h.inst);
    b.tiles = h.tiles;
    b.ntiles = h.ntiles;
    b.partials = h.partials;
    b.parity = h.parity;
    switch (h.mode) {
    case MODE_SWEEP:
        return launch_batch_sweep(b, h, s);
    case MODE_PLAIN: return launch_batch_plain(b, h, s);
    default: lbm_batch_kernel<D, ST, true, true, MODE_CHECK><<<h.grid, h.block, 0, s>>>(b); break;
    }
    return cudaGetLastError();
}

// Resident blocks per SM of the check step of batches at `block` threads (2-D plain steps have the same).
int MFC_OCC_FN(int block)
{
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, lbm_batch_kernel<D, ST, true, true, MODE_CHECK>, block, 0) !=
        cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return n > 0 ? n : 1;
}
#endif

cudaError_t MFC_FILL_FN(const StepHost &h, cudaStream_t s)
{
    const Args a = make_args(h);
    const long long N = (long long)h.geo.nx * h.geo.ny * h.geo.nz;
    const long long b = (N + 255) / 256;
    fill_ghosts_kernel<D, ST, AQ><<<(int)(b < 65535 ? b : 65535), 256, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace mfc
