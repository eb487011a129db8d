"""The strips of large 2-D lattices (several plain steps per launch from a million nodes on): bit for bit
against single steps, with odd and ragged sizes, and with blocked, biofilm and consuming nodes on the first
and last columns, where a strip forms the inlet and outlet values itself."""
import numpy as np
import pytest

import mfc_inputs as mi

pytestmark = pytest.mark.gpu

KW = dict(tau=0.8, tau_c=0.7, u_in=0.01, k_sink=1e-3, c_out=0.3, u_scale=1.25)


@pytest.fixture(scope="module")
def P():
    import paper_1802_07525_gb300 as p
    from paper_1802_07525_gb300 import build
    build.build()
    return p


def _classes(shape, seed):
    nx, ny = shape
    c = mi.mark_sink_layer(shape, mi.bernoulli_block(shape, 0.03, seed)).reshape(ny, nx)
    rng = np.random.default_rng(seed)
    for x in (0, 1, nx - 2, nx - 1):
        c[:, x] = rng.choice([0, 0, 0, 3, 4, 5], ny)
    return c.reshape(-1)


def _pair(P, shape, **kw):
    assert np.prod(shape) > 1000000
    out = []
    for _ in range(2):
        g = P.Lattice(shape, **dict(KW, **kw))
        g.set_geometry(_classes(shape, 3))
        g.step_coupled(3)  # away from rest
        out.append(g)
    return out


def _same(P, a, b):
    for which in (P.MFC_POP_FLOW, P.MFC_POP_ADE):
        assert np.array_equal(a.read_populations(which), b.read_populations(which))


@pytest.mark.parametrize("shape,prec,ade_q,k_half,outlet", [
    ((1203, 853), "MFC_FP32", 0, 0.0, 0), ((1203, 853), "MFC_FP32", 0, 0.05, 1), ((2049, 509), "MFC_FP32", 0, 0.05, 0),
    ((1203, 853), "MFC_FP16_DEV", 0, 0.0, 0), ((509, 2011), "MFC_FP16_DEV", 0, 0.05, 1),
    ((1021, 1013), "MFC_FP32", 9, 0.0, 0), ((2049, 509), "MFC_FP32", 9, 0.05, 1),
    ((1203, 853), "MFC_FP16_DEV", 9, 0.0, 1), ((17, 65535), "MFC_FP32", 0, 0.0, 0), ((90001, 12), "MFC_FP32", 0, 0.0, 0),
], ids=str)
def test_strips_compute_what_single_steps_compute(P, shape, prec, ade_q, k_half, outlet):
    a, b = _pair(P, shape, precision=getattr(P, prec), ade_q=ade_q, k_half=k_half, ade_outlet=outlet)
    for n in (2, 3, 5):  # the lengths' remainders
        a.step_coupled_plain(n)
        for _ in range(n):
            b.step_coupled_plain(1)
        _same(P, a, b)
    # newly blocked nodes, then on from there, ending with a stored step
    assert a.biofilm_grow(1, 1, 0.5, -1.0) == b.biofilm_grow(1, 1, 0.5, -1.0)
    a.step_coupled(8)
    for _ in range(7):
        b.step_coupled_plain(1)
    b.step_coupled(1)
    _same(P, a, b)
    for x, y in zip(a.read_fields()[:3], b.read_fields()[:3]):
        assert np.array_equal(x, y)
    a.close()
    b.close()


def test_strips_closed_box(P):
    a, b = _pair(P, (1021, 1013), bc=(P.MFC_BC_WALL, P.MFC_BC_WALL))
    a.step_coupled_plain(5)
    for _ in range(5):
        b.step_coupled_plain(1)
    _same(P, a, b)
    a.close()
    b.close()


@pytest.mark.parametrize("prec,ade_q", [("MFC_FP32", 0), ("MFC_FP32", 9), ("MFC_FP16_DEV", 0), ("MFC_FP16_DEV", 9)])
def test_strips_of_flow_alone_and_transport_alone(P, prec, ade_q):
    """These have no plain entry point: a call's steps but the last are plain, the last is another kernel's,
    whose multiply-adds may be contracted differently.  Each step then differs by a rounding of the stored
    deviations: 16 units of 2^-24 of the largest of them per step in FP32 (a collision sums 9 and relaxes),
    and two spacings of the storage, 2^-11 each, in FP16."""
    shape, n = (1203, 853), 9
    a, b = _pair(P, shape, precision=getattr(P, prec), ade_q=ade_q)
    a.step_flow(n)
    a.step_ade(n)
    for _ in range(n):
        b.step_flow(1)
    for _ in range(n):
        b.step_ade(1)
    unit = 16 * 2.0 ** -24 if prec == "MFC_FP32" else 2 * 2.0 ** -11
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None]
    for which in (P.MFC_POP_FLOW, P.MFC_POP_ADE):
        x, y = a.read_populations(which), b.read_populations(which)
        open_ = y.any(axis=0)  # blocked nodes read as zero
        dev = np.abs(np.where(open_, y - w, 0.0) if which == P.MFC_POP_FLOW else y).max()
        assert dev > 1e-3
        assert np.abs(x - y).max() <= n * unit * dev
    a.close()
    b.close()
