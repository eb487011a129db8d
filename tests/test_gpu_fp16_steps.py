"""FP16 plain steps of 3-D lattices and FP16 batches against other kernels, with tolerances scaled to what is
stored.  Populations are stored as deviations (flow: f - w, of the order of the velocity; transport: g), and a
store keeps them to half a spacing of at most 2^-10 of their largest.  Two kernels that round a collision
differently may store neighbouring values: two spacings of the largest deviation per step, 2 x 2^-10 of it.
Every case also asserts that the signal is many times its tolerance, so that a state left at rest fails."""
import numpy as np
import pytest

import mfc_inputs as mi

pytestmark = pytest.mark.gpu

W, PE, IO = 0, 1, 2  # boundary kinds
KW = dict(tau=0.7, tau_c=0.6, u_in=0.005, k_sink=5e-4, k_half=0.05)
STEP = 2 * 2.0 ** -10
WF = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)[:, None]


@pytest.fixture(scope="module")
def P():
    import paper_1802_07525_gb300 as p
    from paper_1802_07525_gb300 import build
    build.build()
    return p


def _classes(shape):
    if min(shape) < 10:
        return mi.mark_sink_layer(shape, mi.bernoulli_block(shape, 0.1, 3))
    return mi.mark_sink_layer(shape, mi.overlapping_balls(shape, 3, 0.8, 3))


def _start(P, shape, **kw):
    """A lattice away from rest: with walls and periodic axes alone nothing moves by itself, so the flow starts
    from a velocity wave and the transport from a concentration one."""
    g = P.Lattice(shape, precision=P.MFC_FP16_DEV, **dict(KW, **kw))
    g.set_geometry(_classes(shape))
    n = int(np.prod(shape))
    x = np.arange(n)
    u = 0.01 * np.sin(2 * np.pi * (x % shape[0]) / shape[0] + 0.3 * (x // shape[0]))
    c = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
                  (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1),
                  (0, 1, -1), (0, -1, 1)])
    g.write_populations(P.MFC_POP_FLOW, WF * (1 + 3 * c.sum(1)[:, None] * u))
    wa = np.array([1 / 4] + [1 / 8] * 6)[:, None]
    g.write_populations(P.MFC_POP_ADE, wa * (0.5 + 0.4 * np.cos(0.7 * x)))
    return g


@pytest.mark.parametrize("shape", [(5, 4, 3), (31, 9, 8), (33, 16, 17), (64, 3, 5), (65, 10, 31)], ids=str)
@pytest.mark.parametrize("bc", [(W, W, IO), (PE, PE, IO), (W, PE, PE), (W, W, W)], ids=str)
def test_3d_fp16_plain_steps_against_one_node_steps(P, shape, bc):
    a, b = (_start(P, shape, bc=bc) for _ in range(2))
    assert a.plain_plan(8)["kernel"] == "row"
    n = 8
    a.step_coupled_plain(n)
    for _ in range(n):
        b.step_coupled(1)
    for which in (P.MFC_POP_FLOW, P.MFC_POP_ADE):
        x, y = a.read_populations(which), b.read_populations(which)
        open_ = y.any(axis=0)
        dev = np.where(open_, y - (WF if which == P.MFC_POP_FLOW else 0.0), 0.0)
        tol = n * STEP * np.abs(dev).max()
        assert np.abs(dev).max() > 1e-4
        assert np.abs(dev[1:]).max() > 10 * tol  # the moving populations: at rest they would be zero
        assert np.abs(x - y).max() <= tol
    a.close()
    b.close()


@pytest.mark.parametrize("shape", [(66, 40, 37), (130, 90, 91)], ids=str)
def test_3d_fp16_batch_against_single_steps(P, shape):
    """u sums the ten populations with a component along an axis, C all seven."""
    kw = dict(KW, u_in=0.05)
    cls = _classes(shape)
    n = 10
    with P.Lattice(shape, precision=P.MFC_FP16_DEV, **kw) as a:
        a.set_geometry(cls)
        for _ in range(n):
            a.step_coupled(1)
        u, c = a.read_fields()[1:3]
        f, g = a.read_populations(P.MFC_POP_FLOW), a.read_populations(P.MFC_POP_ADE)
    b = P.Batch(check_every=n, precision=P.MFC_FP16_DEV)
    ticket = b.submit(shape, cls, tol_flow=0.0, tol_ade=0.0, max_steps=n, **kw)
    b.run()
    got = b.poll(ticket)
    b.close()
    fdev = np.abs(np.where(f.any(axis=0), f - WF, 0.0)).max()
    tol_u, tol_c = 10 * n * STEP * fdev, 7 * n * STEP * np.abs(g).max()
    # the inlet's populations have come ten nodes by now: the field there is many times the tolerance
    assert np.abs(u).max() > 5 * tol_u and np.abs(c).max() > 2 * tol_c
    assert np.abs(got["u"] - u).max() <= tol_u
    assert np.abs(got["c"] - c).max() <= tol_c
