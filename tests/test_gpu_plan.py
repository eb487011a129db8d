"""Which kernel a lattice's plain steps take (mfc_plain_plan): the kernels that the comparisons of the other
tests are about are the ones that run, and the benchmark reports the kernel and steps that the library chose."""
import pytest

pytestmark = pytest.mark.gpu

W, PE, IO = 0, 1, 2  # boundary kinds


@pytest.fixture(scope="module")
def P():
    import paper_1802_07525_gb300 as p
    from paper_1802_07525_gb300 import build
    build.build()
    return p


@pytest.mark.parametrize("shape,kw,kernel", [
    ((131, 37), {}, "tile"), ((1024, 512), {}, "tile"), ((1000, 1000), {}, "tile"),
    ((1203, 853), {}, "strip"), ((1203, 853), dict(precision=1), "strip"), ((1021, 1013), dict(ade_q=9), "strip"),
    ((1021, 1013), dict(bc=(W, W)), "strip"),
    ((131, 37), dict(bc=(IO, PE)), "node"), ((131, 37), dict(bc=(IO, PE), precision=1), "pair"),
    ((131, 37), dict(precision=2), "node"), ((40, 12), dict(cut=(0, 1)), "node"),
    # the lattices whose two steps per launch are tested against one
    ((60, 114, 64), {}, "march"), ((119, 119, 120), {}, "march"), ((120, 113, 67), {}, "march"),
    ((119, 119, 120), dict(bc=(W, W, W)), "march"), ((119, 119, 120), dict(precision=1), "row"),
    ((119, 119, 120), dict(bc=(PE, W, IO)), "row"), ((65, 10, 31), {}, "row"), ((13, 11, 17), dict(precision=2), "node"),
    ((10, 8, 24), dict(cut=(1, 0)), "row"),
], ids=str)
def test_kernel_of_plain_steps(P, shape, kw, kernel):
    with P.Lattice(shape, **kw) as g:
        many = kernel in ("tile", "strip", "march")
        plan = g.plain_plan(400)
        assert plan["kernel"] == kernel
        assert plan["launches"] == (-(-400 // plan["steps"]) if many else 400)
        assert (plan["steps"] > 1) == many
        one = g.plain_plan(1)
        assert one["launches"] == one["steps"] == 1 and one["kernel"] in ("node", "pair", "row")
        g.set_launch(block=128, offsets32=0)
        assert g.plain_plan(400) == {"kernel": "node", "steps": 1, "launches": 400}


@pytest.mark.parametrize("shape,kw", [((1024, 512), {}), ((128, 64), {}), ((1203, 853), dict(ade_q=9)),
                                      ((60, 114, 64), {}), ((64, 40, 48), dict(precision=1))], ids=str)
def test_benchmark_reports_the_plan(P, shape, kw):
    import bench
    with P.Lattice(shape, **kw) as g:
        name, steps = bench.plain_kernel(g, 2 if kw.get("precision") == 1 else 4, kw.get("ade_q", 0))
        plan = g.plain_plan(400)
        assert steps == plan["steps"]
        assert {"tile": "tile", "strip": "sweep", "march": "march", "row": "row"}[plan["kernel"]] in name
        # a block of n steps: n - 1 plain steps, the check step, one or two kernels for its sums
        n = bench.block_launches(g, 100, 128)
        assert n - g.plain_plan(99)["launches"] in (2, 3)


def test_plan_refuses_bad_arguments(P):
    with P.Lattice((16, 16)) as g:
        for kind, n in ((3, 10), (-1, 10), (0, 0)):
            with pytest.raises(P.MfcError) as e:
                g.plain_plan(n, kind)
            assert e.value.status == P.MFC_ERR_ARG


@pytest.mark.parametrize("ade_q,kind,steps", [(0, 0, 2), (0, 1, 2), (0, 2, 2), (9, 0, 2), (9, 1, 3), (9, 2, 3)])
def test_steps_of_strips(P, ade_q, kind, steps):
    """Three steps where the registers hold them: D2Q9 flow alone and transport alone, not coupled (which spills)."""
    with P.Lattice((1203, 853), ade_q=ade_q) as g:
        assert g.plain_plan(400, kind)["kernel"] == "strip" and g.plain_plan(400, kind)["steps"] == steps
        assert [g.plain_plan(n, kind)["launches"] for n in (1, 2, 3, 4, 5)] == ([1, 1, 2, 2, 3] if steps == 2 else [1, 1, 1, 2, 2])
