"""Two correction rounds of the mixed path: the second one's sliced products are planned
launches of the tensor-core GEMM (csrc/mixed.cu, slice_plan) at either tile width."""
import numpy as np
import pytest

import oracle
from synth.water import make_water

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g
    g.build()
    import paper_2004_10811_gb300 as p
    return p


@pytest.mark.parametrize("width", [128, 256])
def test_width(pkg, width):
    """The bound of test_gpu_mixed.py's two rounds."""
    import torch
    m = make_water(40, 23, 6.0, (4, -1.0, -0.3), (19, 0.3, 1.5), seed=79)
    want = oracle.density_matrix(m, 0.0, workers=4)
    K = torch.from_numpy(m.vals).cuda()
    with pkg.Plan.from_bsr(m, prec="mixed", refine_rounds=2, tile_n_hp=width) as plan:
        D = plan.sign(K, 0.0, out=torch.full_like(K, float("nan"))).cpu().numpy()
        s = plan.stats()
    assert s["refine_rounds"] == 2 and s["refine_fallback"] == 0
    assert np.all(np.isfinite(D)) and np.max(np.abs(D - want)) <= 1e-10


def test_autotune(pkg):
    import torch
    m = make_water(40, 23, 6.0, (4, -1.0, -0.3), (19, 0.3, 1.5), seed=79)
    K = torch.from_numpy(m.vals).cuda()
    with pkg.Plan.from_bsr(m, prec="mixed", refine_rounds=2) as plan:
        assert all(w in (128, 256) for w in plan.autotune(K, 0.0).values())


def test_two_rounds_above_2048_one_slice_product_per_accumulator(pkg):
    """A second round slices S and a six times each, which the one-pass kernel has no
    shared memory for: the planned launches run, above 2048 with one product to an
    accumulator.  Two rounds meet 1e-10 at ~900 dims (test_gpu_mixed.py); the errors of a
    product grow with its terms."""
    import torch
    m = make_water(256, 23, 9.0, (4, -1.0, -0.3), (19, 0.3, 1.5), seed=106)
    want = oracle.density_matrix(m, 0.0, columns=range(0, 2))
    K = torch.from_numpy(m.vals).cuda()
    for width in (128, 256):
        with pkg.Plan.from_bsr(m, prec="mixed", columns=(0, 2), refine_rounds=2, tile_n_hp=width) as plan:
            D = plan.sign(K, 0.0, out=torch.full_like(K, float("nan"))).cpu().numpy()
            s = plan.stats()
        assert s["n_min"] > 2048 and s["refine_rounds"] == 2 and s["refine_fallback"] == 0
        vp = m.val_ptr
        idx = np.concatenate([np.arange(vp[p], vp[p + 1]) for p in range(m.nnzb) if m.col_idx[p] < 2])
        assert np.all(np.isfinite(D[idx])) and np.max(np.abs(D[idx] - want[idx])) <= 1e-9
