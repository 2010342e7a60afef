"""The FP64 path's residue products (csrc/rns.cu) against the oracle and against
the SIMT GEMM, which the same plan runs when its workspace is too small for them.

Bound: a product entry is off by at most 14 * 128 * 2^-65 * 2.02 < 1.1e-16 from the
rounded weights and sqrt(n) 2^-55 from each operand's rounding (unit row norms), so
a product's spectral error is below n * 3e-16; Newton-Schulz takes about 25
products, and an error E moves sign(a) by at most |E| / gap."""
import numpy as np
import pytest

import oracle
from synth import random_symmetric_bsr, small_case
from synth.water import BSRMatrix, make_water

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g
    g.build()
    import paper_2004_10811_gb300 as p
    return p


def one_submatrix(n, seed, gap=0.2):
    """A full-cover pattern of blocks up to 60: every submatrix is the whole matrix."""
    rng = np.random.default_rng(seed)
    bs = []
    while sum(bs) < n:
        bs.append(int(min(rng.integers(1, 61), n - sum(bs))))
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    w = gap + (1 - gap) * rng.random(n)
    w[: (n + 1) // 2] *= -1
    a = (q * w) @ q.T
    a = 0.5 * (a + a.T)
    k = len(bs)
    st = np.concatenate([[0], np.cumsum(bs)])
    vals = np.concatenate([a[st[i]:st[i + 1], st[j]:st[j + 1]].ravel() for i in range(k) for j in range(k)])
    return BSRMatrix(np.array(bs, np.int32), np.arange(k + 1, dtype=np.int64) * k,
                     np.tile(np.arange(k, dtype=np.int32), k), vals), a, st


def sign(pkg, m, mu, allow=False, **kw):
    import torch
    K = torch.from_numpy(m.vals).cuda()
    with pkg.Plan.from_bsr(m, prec="fp64", **kw) as plan:
        D = plan.sign(K, mu, out=torch.zeros_like(K), allow_not_converged=allow).cpu().numpy()
        return D, plan.stats()


# tile edges (64, 128), ragged last tiles, and K beyond one exact accumulation (1024)
@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 127, 128, 129, 191, 320, 449, 1024, 1025, 1100])
def test_one_submatrix(pkg, n):
    m, a, st = one_submatrix(n, 40 + n)
    w, q = np.linalg.eigh(a)
    want = (q * (w < 0)) @ q.T
    # block columns 0 and the last: the same submatrix, other extracted rows
    got, stats = sign(pkg, m, 0.0, columns=(0, 1))
    wide = np.concatenate([want[st[i]:st[i + 1], st[j]:st[j + 1]].ravel()
                           for i in range(len(m.block_sizes)) for j in range(len(m.block_sizes))])
    keep = got != 0
    assert np.max(np.abs(got - wide)[keep]) <= n * 25 * 3e-16 / 0.2 + 1e-15
    assert stats["workspace_bytes"] >= 72 * ((n + 63) // 64 * 64) ** 2


FORMS = {
    "uneven": (lambda: random_symmetric_bsr([5, 7, 3, 9, 2, 8, 6, 4, 7, 5, 3, 6], density=0.35, seed=24, scale=0.5), 0.15, {}),
    "elementwise": (lambda: random_symmetric_bsr([1] * 70, density=0.2, seed=25, scale=0.5), -0.1, {}),
    "water": (lambda: make_water(96, 5, 6.5, (2, -1.0, -0.3), (3, 0.3, 1.2), seed=77), 0.05, {}),
    "bound scale": (lambda: make_water(96, 5, 6.5, (2, -1.0, -0.3), (3, 0.3, 1.2), seed=77), 0.05, {"beta_mode": 1}),
    "symmetrized": (lambda: small_case(n_mol=24, block=3, r_c=5.0, seed=8), 0.0, {"symmetrize": True}),
    "columns": (lambda: small_case(n_mol=24, block=3, r_c=5.0, seed=8), 0.0, {"columns": (5, 17)}),
    "grouped": (lambda: small_case(n_mol=24, block=3, r_c=5.0, seed=8), 0.0, {"groups": np.arange(24) // 3}),
    "step cap": (lambda: small_case(n_mol=24, block=4, r_c=5.0, seed=9), 0.0, {"max_iter": 3}),
}


@pytest.mark.parametrize("form", FORMS)
def test_matches_simt_path(pkg, form):
    make, mu, kw = FORMS[form]
    m = make()
    got, s1 = sign(pkg, m, mu, allow="max_iter" in kw, **kw)
    ld = (s1["n_max"] + 63) // 64 * 64
    simt, s2 = sign(pkg, m, mu, allow="max_iter" in kw, workspace_cap_bytes=30 * ld * ld, **kw)
    assert s2["workspace_bytes"] <= 30 * ld * ld < s1["workspace_bytes"]
    assert s1["not_converged"] == s2["not_converged"] and s1["scale_reduced"] == s2["scale_reduced"]
    # gaps here are 0.01 (uneven, random) or more
    gap = 0.25 if "uneven" not in form and form != "elementwise" else _gap(m, mu)
    assert np.max(np.abs(got - simt)) <= 2 * s1["n_max"] * 25 * 3e-16 / gap


def _gap(m, mu):
    return min(float(np.min(np.abs(lam))) for lam, _q in oracle.decompose_all(m, mu))


def test_exact_zero_eigenvalue(pkg):
    """An eigenvalue exactly at mu stays 0: NOT_CONVERGED, the others settled."""
    m = BSRMatrix(np.array([3], np.int32), np.array([0, 1]), np.array([0], np.int32),
                  np.diag([-0.5, 0.25, 1.0]).ravel())
    got, s = sign(pkg, m, 0.25, allow=True)
    assert s["not_converged"] == 1
    assert np.max(np.abs(got.reshape(3, 3) - np.diag([1.0, 0.5, 0.0]))) <= 1e-14


def fermi(pkg, m, mu, kT, **kw):
    import torch
    K = torch.from_numpy(m.vals).cuda()
    with pkg.Plan.from_bsr(m, prec="fp64", kT=kT, **kw) as plan:
        D = plan.sign(K, mu, out=torch.zeros_like(K)).cpu().numpy()
        return D, plan.stats()


# tile edges, K beyond 1024, one Clenshaw block (kT 1) to many (kT 0.004: terms above 1)
@pytest.mark.parametrize("n,kT", [(1, 0.1), (64, 0.01), (65, 1.0), (127, 0.05), (129, 0.02), (320, 0.05), (1025, 0.1)])
def test_fermi_one_submatrix(pkg, n, kT):
    m, a, st = one_submatrix(n, 70 + n)
    w, q = np.linalg.eigh(a)
    want = (q / (1.0 + np.exp(w / kT))) @ q.T
    got, s = fermi(pkg, m, 0.0, kT, columns=(0, 1))
    wide = np.concatenate([want[st[i]:st[i + 1], st[j]:st[j + 1]].ravel()
                           for i in range(len(m.block_sizes)) for j in range(len(m.block_sizes))])
    keep = got != 0
    # truncation, and per product n * 3e-16 through 16 baby steps (T_16: 256) and the
    # giant steps, whose errors grow with the derivative of f (at most 1 / (4 kT))
    G = (s["poly_degree"] + 16) // 16
    assert np.max(np.abs(got - wide)[keep]) <= 2e-13 + n * 3e-16 * (256 / (4 * kT) + G * G)
    assert s["workspace_bytes"] >= 152 * ((n + 63) // 64 * 64) ** 2


@pytest.mark.parametrize("form", [f for f in FORMS if f != "step cap"])
@pytest.mark.parametrize("kT", [0.05, 0.4])
def test_fermi_matches_simt_path(pkg, form, kT):
    make, mu, kw = FORMS[form]
    m = make()
    got, s1 = fermi(pkg, m, mu, kT, **kw)
    ld = (s1["n_max"] + 63) // 64 * 64
    simt, s2 = fermi(pkg, m, mu, kT, workspace_cap_bytes=100 * ld * ld, **kw)
    assert s2["workspace_bytes"] <= 100 * ld * ld < s1["workspace_bytes"]
    G = (s1["poly_degree"] + 16) // 16
    assert np.max(np.abs(got - simt)) <= 4e-13 + 2 * s1["n_max"] * 3e-16 * (256 / (4 * kT) + G * G)
    assert abs(s1["dn_dmu"] - s2["dn_dmu"]) <= 1e-10 * m.n / kT
