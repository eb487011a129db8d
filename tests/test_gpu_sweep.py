"""Several plain steps per launch against the same steps one launch each: the kernels that carry a
lattice through several steps compute, bit for bit, what the one-step kernels compute, so every
comparison is exact.  Sizes sit at the edges of the column tiles and row strips."""
import numpy as np
import pytest

import mfc_inputs as mi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_1802_07525_gb300 as p
    from paper_1802_07525_gb300 import build
    build.build()
    return p


def _classes(shape, seed):
    if min(shape) < 10:
        return mi.mark_sink_layer(shape, mi.bernoulli_block(shape, 0.1, seed))
    return mi.mark_sink_layer(shape, mi.overlapping_balls(shape, 3, 0.8, seed))


def _pair(P, shape, **kw):
    out = []
    for _ in range(2):
        g = P.Lattice(shape, **kw)
        g.set_geometry(_classes(shape, 3))
        g.step_coupled(3)  # away from rest
        out.append(g)
    return out


def _same(P, a, b):
    for which in (P.MFC_POP_FLOW, P.MFC_POP_ADE):
        assert np.array_equal(a.read_populations(which), b.read_populations(which))
    for x, y in zip(a.read_fields()[:3], b.read_fields()[:3]):
        assert np.array_equal(x, y)


def _check(P, shape, n, **kw):
    a, b = _pair(P, shape, **kw)
    a.step_coupled_plain(n)
    for _ in range(n):
        b.step_coupled_plain(1)
    _same(P, a, b)
    # newly blocked nodes, then on from there
    assert a.biofilm_grow(1, 1, 0.5, -1.0) == b.biofilm_grow(1, 1, 0.5, -1.0)
    a.step_coupled(6)
    for _ in range(5):
        b.step_coupled_plain(1)
    b.step_coupled(1)
    _same(P, a, b)
    a.close()
    b.close()


SHAPES_2D = [(1, 1), (5, 2), (59, 7), (60, 24), (61, 25), (64, 33), (119, 5), (120, 40), (121, 3), (300, 70), (1000, 12)]


@pytest.mark.parametrize("shape", SHAPES_2D, ids=str)
@pytest.mark.parametrize("prec", ["MFC_FP32", "MFC_FP16_DEV"])
def test_2d_sweeps_compute_what_single_steps_compute(P, shape, prec):
    _check(P, shape, 7, precision=getattr(P, prec), tau=0.8, tau_c=0.7, u_in=0.01, k_sink=1e-3)


@pytest.mark.parametrize("ade_q", [0, 9])
@pytest.mark.parametrize("k_half", [0.0, 0.05])
@pytest.mark.parametrize("outlet", [0, 1])
@pytest.mark.parametrize("prec", ["MFC_FP32", "MFC_FP16_DEV"])
def test_2d_sweeps_options(P, ade_q, k_half, outlet, prec):
    _check(P, (131, 37), 10, precision=getattr(P, prec), ade_q=ade_q, tau=0.8, tau_c=0.7, u_in=0.01,
           k_sink=1e-3, k_half=k_half, ade_outlet=outlet, c_out=0.3, u_scale=1.25)


@pytest.mark.parametrize("shape", [(62, 9), (250, 31)], ids=str)
@pytest.mark.parametrize("ade_q", [0, 9])
def test_2d_sweeps_one_lattice_at_a_time(P, shape, ade_q):
    """Flow alone and transport alone have no plain entry point: a call's steps but the last are plain, the
    last stores its fields in another kernel.  Against single (stored) steps the difference is that
    kernel's rounding: within 2e-6 after 9 steps on values of order one (a few FP32 ulp per step)."""
    a, b = _pair(P, shape, ade_q=ade_q, tau=0.8, tau_c=0.7, u_in=0.01, k_sink=1e-3)
    a.step_flow(9)
    a.step_ade(9)
    for _ in range(9):
        b.step_flow(1)
    for _ in range(9):
        b.step_ade(1)
    for which in (P.MFC_POP_FLOW, P.MFC_POP_ADE):
        assert np.abs(a.read_populations(which) - b.read_populations(which)).max() < 2e-6
    a.close()
    b.close()


def test_2d_closed_box(P):
    _check(P, (90, 41), 9, bc=(P.MFC_BC_WALL, P.MFC_BC_WALL), tau=0.8, tau_c=0.7, k_sink=1e-3)


W, PE, IO = 0, 1, 2  # boundary kinds


@pytest.mark.parametrize("shape", [(1, 1, 2), (5, 4, 3), (31, 9, 8), (33, 16, 17), (64, 3, 5), (65, 10, 31)], ids=str)
@pytest.mark.parametrize("bc", [(W, W, IO), (PE, PE, IO), (W, PE, PE), (W, W, W)], ids=str)
@pytest.mark.parametrize("prec", ["MFC_FP32", "MFC_FP16_DEV"])
def test_3d_plain_steps_against_one_node_steps(P, shape, bc, prec):
    """The two-node plain steps against stored-field steps, which run one node per thread with 64-bit
    offsets: their multiply-adds may be contracted differently, so 8 steps agree to 2e-6 in FP32 (a few ulp
    per step on values of order one) and to two FP16 spacings per step in FP16 storage."""
    kw = dict(precision=getattr(P, prec), bc=bc, tau=0.7, tau_c=0.6, u_in=0.005, k_sink=5e-4, k_half=0.05)
    a, b = _pair(P, shape, **kw)
    a.step_coupled_plain(8)
    for _ in range(8):
        b.step_coupled(1)
    for which in (P.MFC_POP_FLOW, P.MFC_POP_ADE):
        x, y = a.read_populations(which), b.read_populations(which)
        tol = 2e-6 if prec == "MFC_FP32" else 8 * 2 * 2.0 ** -12
        assert np.abs(x - y).max() < tol
    a.close()
    b.close()


@pytest.mark.parametrize("shape,prec", [((97, 71, 83), "MFC_FP32"), ((130, 90, 91), "MFC_FP16_DEV")], ids=str)
def test_3d_planes_in_alternating_order(P, shape, prec):
    """Steps that read and write more than the L2 holds take their planes upwards and downwards in turn, a
    batch its chunks; a single lattice and a batch of it alone round differently by a few FP32 ulp (FP16:
    storage spacings) per step, so fields agree to 2e-6 (FP16: 5e-3, ten spacings at one)."""
    kw = dict(tau=0.7, tau_c=0.6, u_in=0.005, k_sink=5e-4)
    cls = _classes(shape, 3)
    a, b = (P.Lattice(shape, precision=getattr(P, prec), **kw) for _ in range(2))
    for g in (a, b):
        g.set_geometry(cls)
    a.step_coupled_plain(9)
    for _ in range(9):
        b.step_coupled_plain(1)
    _same(P, a, b)
    a.close()
    a = P.Lattice(shape, precision=getattr(P, prec), **kw)
    a.set_geometry(cls)
    a.step_coupled(10)
    batch = P.Batch(check_every=10, precision=getattr(P, prec))
    ticket = batch.submit(shape, cls, tol_flow=0.0, tol_ade=0.0, max_steps=10, **kw)
    batch.run()
    got = batch.poll(ticket)
    batch.close()
    tol = 2e-6 if prec == "MFC_FP32" else 5e-3
    for x, y in zip((got["u"], got["c"]), a.read_fields()[1:3]):
        assert np.abs(x - y).max() < tol
    a.close()
    b.close()


@pytest.mark.parametrize("shape", [(60, 114, 64), (119, 119, 120), (120, 113, 67)], ids=str)
@pytest.mark.parametrize("bc,k_half,outlet", [((W, W, IO), 0.0, 0), ((W, W, IO), 0.05, 1), ((W, W, W), 0.0, 0)], ids=str)
def test_3d_two_steps_per_launch(P, shape, bc, k_half, outlet):
    """Lattices whose coupled steps go two at a time, against one step per launch: exact."""
    _check(P, shape, 5, bc=bc, tau=0.7, tau_c=0.6, u_in=0.005, k_sink=5e-4, k_half=k_half, ade_outlet=outlet,
           c_out=0.3, u_scale=1.25)
