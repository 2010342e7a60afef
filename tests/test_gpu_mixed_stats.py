"""What the mixed path's statistics and tuner report."""
import numpy as np
import pytest

from synth.water import make_water

from test_gpu_rns import one_submatrix

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g
    g.build()
    import paper_2004_10811_gb300 as p
    return p


@pytest.mark.parametrize("asked,kept", [(0, 128), (256, 256)])
def test_one_round_has_no_sliced_width_to_tune(pkg, asked, kept):
    """The first round's sliced products have one width, so that a timing of two could
    only pick by noise: the plan's choice stands, in every one of six runs."""
    import torch
    m = make_water(24, 6, 4.5, (2, -1.0, -0.3), (4, 0.3, 1.0), seed=12)
    K = torch.from_numpy(m.vals).cuda()
    for _ in range(6):
        with pkg.Plan.from_bsr(m, prec="mixed", tile_n_hp=asked) as plan:
            assert plan.autotune(K, 0.0)["sliced"] == kept == plan.options.tile_n_hp
