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


@pytest.mark.parametrize("width", [128, 256])
@pytest.mark.parametrize("n", [60, 192, 250, 320, 570])
def test_executed_work_counts_the_columns_that_tiles_form(pkg, n, width):
    """kernel_exec by its definition, tile by tile: 128 rows x the columns inside the
    matrix (and, of a 256-wide tile, not those of a left half below the diagonal) x ld x
    2 flops, three MMAs per split product; the first round's 16 and 21 slice products
    run whole 128 x 128 tiles."""
    import torch
    m, _a, _st = one_submatrix(n, 500 + n)
    K = torch.from_numpy(m.vals).cuda()
    with pkg.Plan.from_bsr(m, prec="mixed", columns=(0, 1), tile_n_ns=width, tile_n_corr=width, timing=True) as plan:
        plan.sign(K, 0.0)
        s = plan.stats()
    assert s["refine_fallback"] == 0
    ld = (n + 63) // 64 * 64
    t = -(-ld // 128)

    def columns(a, b, sym):
        lo, hi = b * width, min(ld, (b + 1) * width)
        return max(0, hi - (max(lo, a * 128) if sym else lo))

    cols = {sym: sum(columns(a, b, sym) for a in range(t) for b in range(-(-ld // width))) for sym in (True, False)}
    flops = {sym: 2.0 * 128 * ld * c for sym, c in cols.items()}
    assert s["kernel_exec"][0] == pytest.approx(2 * s["iters_max"] * 3 * flops[True], rel=1e-12)
    assert s["kernel_exec"][4] == pytest.approx((16 * t * (t + 1) / 2 + 21 * t * t) * 2.0 * 128 * 128 * ld, rel=1e-12)
    # two symmetric products and a full one, and a full one per CG step
    cg = (s["kernel_exec"][1] - 3 * (2 * flops[True] + flops[False])) / (3 * flops[False])
    assert cg == pytest.approx(round(cg), abs=1e-9) and 1 <= cg <= s["refine_cg_iters"]
