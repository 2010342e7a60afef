"""The allocation-free dense evaluation (csrc/noalloc.cu, one cooperative launch over
8 x 8 blocks): block edges, one CTA to more blocks than SMs, and its exits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sm():
    import __graft_entry__ as g
    g.build()
    from paper_2004_10811_gb300 import submat
    return submat


def levels(n, seed, mu=0.0):
    """A matrix with a gap of 0.25 at mu, and its D."""
    rng = np.random.default_rng(seed)
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    w = rng.uniform(0.25, 1.4, n)
    w[: n // 3] *= -1
    a = (q * (w + mu)) @ q.T
    return 0.5 * (a + a.T), (q * (w < 0)) @ q.T


# 17 and 18 rows of blocks: 153 and 171 blocks, about one for each of 152 SMs
@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 15, 16, 17, 63, 64, 65, 127, 129, 136, 137, 144, 300, 505, 511, 512])
def test_dims(sm, n):
    """A product entry is off by n 2^-53, Newton-Schulz runs ~25, an error E moves sign(a)
    by E / gap."""
    import torch
    a, want = levels(n, n, 0.1)
    K = torch.from_numpy(a).cuda()
    d, iters = sm.dense_sign_noalloc(K, 0.1, out=torch.full_like(K, float("nan")))
    d = d.cpu().numpy()
    assert np.all(np.isfinite(d)) and 0 < iters < 60
    assert np.max(np.abs(d - want)) <= n * 25 * 2.0 ** -53 * n ** 0.5 / 0.25 + 1e-15


def test_output_in_place_of_the_input(sm):
    import torch
    a, want = levels(77, 5)
    K = torch.from_numpy(a).cuda()
    sm.dense_sign_noalloc(K, 0.0, out=K)
    assert np.max(np.abs(K.cpu().numpy() - want)) <= 1e-12


@pytest.mark.parametrize("n", [1, 9, 200])
def test_exits(sm, n):
    """K = mu I (nothing to iterate), a NaN or Inf in K, and a level exactly at mu, each
    followed by an ordinary call on the same scratch."""
    import torch
    a, want = levels(n, 40 + n)

    def ordinary():
        d, _ = sm.dense_sign_noalloc(torch.from_numpy(a).cuda(), 0.0)
        assert np.max(np.abs(d.cpu().numpy() - want)) <= 1e-12

    d, iters = sm.dense_sign_noalloc(0.3 * torch.eye(n, dtype=torch.float64, device="cuda"), 0.3)
    assert iters == 0 and torch.equal(d, 0.5 * torch.eye(n, dtype=torch.float64, device="cuda"))
    ordinary()
    for bad in (float("nan"), float("inf")):
        K = torch.from_numpy(a.copy()).cuda()
        K[n - 1, n // 2] = bad
        with pytest.raises(sm.SubmatError) as e:
            sm.dense_sign_noalloc(K, 0.0)
        assert e.value.name == "NONFINITE"
        ordinary()
    K = torch.diag(torch.linspace(0.0, 1.0, n, dtype=torch.float64, device="cuda"))
    if n > 1:  # level 0 at mu = 0 stays 0
        with pytest.raises(sm.SubmatError) as e:
            sm.dense_sign_noalloc(K, 0.0)
        assert e.value.name == "NOT_CONVERGED"
        ordinary()
