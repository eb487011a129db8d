"""Batches whose blocks hold one plain step: every instance alone and in a mix of walls, periodic axes and
dimensions gives the same bits, and the fields of a single lattice to FP32 rounding."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

W, PE, IO = 0, 1, 2  # boundary kinds
REQUESTS = [((90, 41), (IO, W)), ((64, 32), (IO, PE)), ((33, 70), (W, W)), ((20, 18, 15), (W, W, IO)), ((12, 9, 10), (PE, PE, IO))]


@pytest.fixture(scope="module")
def P():
    import paper_1802_07525_gb300 as p
    from paper_1802_07525_gb300 import build
    build.build()
    return p


def _classes(shape):
    rng = np.random.default_rng(5)
    return rng.choice([0] * 20 + [3, 4, 5], int(np.prod(shape))).astype(np.uint8)


def _kw(shape):
    return dict(tau=0.8, tau_c=0.7, u_in=0.01, k_sink=1e-3) if len(shape) == 2 else dict(tau=0.7, tau_c=0.6, u_in=0.005, k_sink=5e-4)


def _run(P, requests, prec, **kw):
    b = P.Batch(precision=prec, **kw)
    t = [b.submit(s, _classes(s), bc=bc, tol_flow=0.0, tol_ade=0.0, max_steps=12, **_kw(s)) for s, bc in requests]
    b.run()
    out = [b.poll(x) for x in t]
    b.close()
    return out


@pytest.mark.parametrize("prec", ["MFC_FP32", "MFC_FP16_DEV"])
@pytest.mark.parametrize("every", [2, 4])
def test_short_blocks(P, prec, every):
    prec = getattr(P, prec)
    mix = _run(P, REQUESTS, prec, check_every=every, block=64)
    for (shape, bc), got in zip(REQUESTS, mix):
        alone = _run(P, [(shape, bc)], prec, check_every=every, block=64)[0]
        for k in ("rho", "u", "c"):
            assert np.array_equal(got[k], alone[k])
        assert got["steps_flow"] == 12 and got["current"] == alone["current"]
        with P.Lattice(shape, bc=bc, precision=prec, **_kw(shape)) as g:
            g.set_geometry(_classes(shape))
            g.solve_steady(mode=P.MFC_CONCURRENT, tol_flow=0.0, tol_ade=0.0, max_steps=12, check_every=every)
            rho, u, c, _ = g.read_fields()
        # a single lattice's kernels may contract other multiply-adds: 16 units of 2^-24 per step of the
        # largest velocity and concentration in FP32 (rho - 1 is of the order of the velocity's square and
        # sum), two FP16 spacings per step and population summed over the set otherwise
        unit = 12 * 16 * 2.0 ** -24 if prec == P.MFC_FP32 else 12 * 19 * 2 * 2.0 ** -11
        scale = max(np.abs(u).max(), 1e-3)
        assert np.abs(got["u"] - u).max() <= unit * scale
        assert np.abs(got["c"] - c).max() <= unit * max(np.abs(c).max(), 1e-3)


@pytest.mark.parametrize("prec", ["MFC_FP32", "MFC_FP16_DEV"])
def test_tuned_block_gives_the_results_of_the_given_one(P, prec):
    """Tuning runs check steps, which store fields: the first check must still compare with the state at rest."""
    prec = getattr(P, prec)
    tuned = P.Batch(precision=prec, check_every=4)
    t = [tuned.submit(s, _classes(s), bc=bc, tol_flow=0.0, tol_ade=0.0, max_steps=4, **_kw(s)) for s, bc in REQUESTS]
    tuned.run()
    block = tuned.stats()["block"]
    got = [tuned.poll(x) for x in t]
    tuned.close()
    assert block in (64, 128, 256)
    want = P.Batch(precision=prec, check_every=4, block=block)
    t = [want.submit(s, _classes(s), bc=bc, tol_flow=0.0, tol_ade=0.0, max_steps=4, **_kw(s)) for s, bc in REQUESTS]
    want.run()
    for a, x in zip(got, t):
        b = want.poll(x)
        for k in ("rho", "u", "c"):
            assert np.array_equal(a[k], b[k])
        for k in ("res_flow", "res_ade", "mass", "current", "steps_flow"):
            assert a[k] == b[k], k
    want.close()
