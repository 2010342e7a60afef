"""Workspace of FP64 plans: without a cap no more than a fifth of the free memory, in as
many waves as that takes, with the results of one wave."""
import pytest

from synth.water import make_water

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g
    g.build()
    import paper_2004_10811_gb300 as p
    return p


@pytest.mark.parametrize("kT", [0.0, 0.2])
def test_uncapped_plan_leaves_room(pkg, kT):
    import torch
    m = make_water(343, 6, 8.0, (2, -1.0, -0.3), (4, 0.3, 1.0), seed=31)
    K = torch.from_numpy(m.vals).cuda()
    with pkg.Plan.from_bsr(m, prec="fp64", kT=kT, workspace_cap_bytes=40 << 30) as plan:
        want = plan.sign(K, 0.0)
        s = plan.stats()
        assert s["waves"] == 1
        need = s["workspace_bytes"]
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    hog = torch.empty(free - 2 * need, dtype=torch.uint8, device="cuda")
    try:
        free, _ = torch.cuda.mem_get_info()
        with pkg.Plan.from_bsr(m, prec="fp64", kT=kT) as plan:
            got = plan.sign(K, 0.0)
            s = plan.stats()
            left, _ = torch.cuda.mem_get_info()
    finally:
        del hog
        torch.cuda.empty_cache()
    assert s["workspace_bytes"] <= 0.2 * free and s["waves"] > 1
    assert left >= 0.75 * free
    # at T > 0 a wave's submatrices share one scale and degree
    assert torch.equal(got, want) if kT == 0.0 else float((got - want).abs().max()) <= 1e-12
