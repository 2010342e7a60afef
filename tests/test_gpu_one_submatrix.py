"""Every stored entry of one block column of D, on every path: the output starts as NaN,
so an entry that no kernel writes shows, and the entries looked at come from the pattern
(block column 0, or the last: other extracted rows of the same submatrix)."""
import numpy as np
import pytest

from synth.water import BSRMatrix
from test_gpu_rns import one_submatrix

pytestmark = pytest.mark.gpu

# tile edges (64, 128, 256), ragged last tiles, and sums beyond one exact chunk (1024, 1056)
DIMS = [1, 2, 63, 64, 65, 127, 128, 129, 191, 256, 257, 320, 449, 1025, 1057]


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g
    g.build()
    import paper_2004_10811_gb300 as p
    return p


def column_error(pkg, m, st, want, last, **kw):
    """Largest error over block column 0 (or the last); every other entry stays NaN."""
    import torch
    k = len(m.block_sizes)
    j = k - 1 if last else 0
    K = torch.from_numpy(m.vals).cuda()
    with pkg.Plan.from_bsr(m, columns=(j, j + 1), **kw) as plan:
        D = plan.sign(K, 0.0, out=torch.full_like(K, float("nan"))).cpu().numpy()
        stats = plan.stats()
    vp, mine = m.val_ptr, np.zeros(len(D), bool)
    err = 0.0
    for i in range(k):
        p = i * k + j  # block (i, j) of the full pattern
        mine[vp[p]:vp[p + 1]] = True
        e = D[vp[p]:vp[p + 1]] - want[st[i]:st[i + 1], st[j]:st[j + 1]].ravel()
        err = max(err, float(np.max(np.abs(e)))) if np.all(np.isfinite(e)) else np.inf
    assert np.all(np.isnan(D[~mine]))
    return err, stats


def exact_sign(a):
    w, q = np.linalg.eigh(a)
    return (q * (w < 0)) @ q.T


@pytest.mark.parametrize("last", [False, True])
@pytest.mark.parametrize("n", DIMS)
def test_fp64(pkg, n, last):
    """n 25 3e-16 / gap as in test_gpu_rns.py (the grid is finer now)."""
    m, a, st = one_submatrix(n, 40 + n)
    err, stats = column_error(pkg, m, st, exact_sign(a), last, prec="fp64")
    assert err <= n * 25 * 3e-16 / 0.2 + 1e-15


@pytest.mark.parametrize("width", [128, 256])
@pytest.mark.parametrize("last", [False, True])
@pytest.mark.parametrize("n", DIMS)
def test_mixed(pkg, n, last, width):
    """The mixed path's contract."""
    m, a, st = one_submatrix(n, 300 + n)
    err, stats = column_error(pkg, m, st, exact_sign(a), last, prec="mixed", tile_n_ns=width, tile_n_corr=width)
    assert stats["refine_fallback"] == 0 and err <= 1e-7


@pytest.mark.parametrize("last", [False, True])
@pytest.mark.parametrize("n,kT", [(1, 0.1), (63, 0.004), (64, 0.01), (65, 1.0), (127, 0.05), (129, 0.02), (200, 0.004),
                                  (320, 0.05), (1025, 0.1)])
def test_fermi(pkg, n, kT, last):
    """test_gpu_rns.py's bound; kT 0.004 has Clenshaw terms above 1."""
    m, a, st = one_submatrix(n, 70 + n)
    w, q = np.linalg.eigh(a)
    err, stats = column_error(pkg, m, st, (q / (1.0 + np.exp(w / kT))) @ q.T, last, prec="fp64", kT=kT)
    G = (stats["poly_degree"] + 16) // 16
    assert err <= 2e-13 + n * 3e-16 * (256 / (4 * kT) + G * G)


@pytest.mark.parametrize("kT", [1.0, 0.2, 0.05, 0.02, 0.008, 0.004, 0.0015])
def test_fermi_levels(pkg, kT):
    """Uncoupled levels: D is the series itself, from the coefficients that the GPU sums
    (256 to 16384 nodes over this list).  A sum of N terms of at most 1 is off by about
    sqrt(N) 2^-53 of their total, so a coefficient by 2 sqrt(N) 2^-53 and the series by
    N / 4 of them at most."""
    import torch
    rng = np.random.default_rng(3)
    x = np.concatenate([rng.uniform(-1, 1, 400), [1.0, -1.0, 1e-3, -1e-3, 0.0]])
    k = len(x)
    m = BSRMatrix(np.ones(k, np.int32), np.arange(k + 1, dtype=np.int64), np.arange(k, dtype=np.int32), x)
    K = torch.from_numpy(x).cuda()
    with pkg.Plan.from_bsr(m, prec="fp64", kT=kT) as plan:
        D = plan.sign(K, 0.0, out=torch.full_like(K, float("nan"))).cpu().numpy()
        deg = plan.stats()["poly_degree"]
    N = 256
    while N // 2 <= deg:
        N *= 2
    want = 1.0 / (1.0 + np.exp(x / kT))
    assert np.max(np.abs(D - want)) <= 2e-13 + 2 * N ** 0.5 * 2.0 ** -53 * N / 4


@pytest.mark.parametrize("kT", [0.0, 0.5])
def test_fp64_many_chunks(pkg, kT):
    """3300 dims: four exact chunks of each of 19 moduli, more phases (76) than the guard
    sums of k_rns_gemm take without being folded.  A = Q w Q^T with Q known to n 2^-53;
    bounds as above."""
    import torch
    n = 3300
    g = torch.Generator(device="cuda").manual_seed(5)
    q, _ = torch.linalg.qr(torch.randn(n, n, generator=g, device="cuda", dtype=torch.float64))
    w = 0.2 + 0.8 * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    w[: n // 2] *= -1.0
    a = (q * w) @ q.T
    a = 0.5 * (a + a.T)
    want = (q * (torch.sigmoid(-w / kT) if kT else (w < 0).double())) @ q.T
    with pkg.Plan(np.array([n], np.int32), np.array([0, 1], np.int64), np.array([0], np.int32), prec="fp64", kT=kT,
                  timing=True) as plan:
        D = plan.sign(a.flatten().contiguous(), 0.0).reshape(n, n)
        s = plan.stats()
    assert s["kernel_launches"][7] > 0 == s["kernel_launches"][2]
    err = float((D - want).abs().max())
    assert err <= n * 25 * 3e-16 / 0.2 if not kT else 2e-13 + n * 3e-16 * (256 / (4 * kT) + 16)
    assert err <= 1e-12
