"""The one-pass exact sliced products (csrc/slice_gemm.cu) and the tensor-core GEMM's
narrow last tiles through the mixed path, at the sizes where they can go wrong: tile
edges (64, 128, 256), ragged last tiles, and sums beyond one exact chunk (1056 terms).

Bound: the mixed path's contract against the oracle, max |dD| <= 1e-7; a slice product
left out or doubled leaves the FP16 iterate's error (1e-6 and more) in place."""
import numpy as np
import pytest

from test_gpu_rns import one_submatrix

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g
    g.build()
    import paper_2004_10811_gb300 as p
    return p


@pytest.mark.parametrize("width", [128, 256])
@pytest.mark.parametrize("n", [1, 63, 64, 65, 128, 129, 191, 256, 257, 320, 449, 1056, 1057, 1100])
def test_mixed_one_submatrix(pkg, n, width):
    import torch
    m, a, st = one_submatrix(n, 300 + n)
    w, q = np.linalg.eigh(a)
    want = (q * (w < 0)) @ q.T
    K = torch.from_numpy(m.vals).cuda()
    with pkg.Plan.from_bsr(m, prec="mixed", columns=(0, 1), tile_n_ns=width, tile_n_corr=width) as plan:
        got = plan.sign(K, 0.0, out=torch.zeros_like(K)).cpu().numpy()
        assert plan.stats()["refine_fallback"] == 0
    wide = np.concatenate([want[st[i]:st[i + 1], st[j]:st[j + 1]].ravel()
                           for i in range(len(m.block_sizes)) for j in range(len(m.block_sizes))])
    keep = got != 0
    assert np.max(np.abs(got - wide)[keep], initial=0.0) <= 1e-7
