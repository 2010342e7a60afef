"""Small entries of D on the FP64 path.  D decays with distance, so its far blocks are
orders of magnitude below one; FP64 chains of multiply-adds keep their relative
accuracy, and the residue products (csrc/rns.cu) have to as well: by their 2^-73 grid
where a submatrix's extracted columns couple to its rows by 2^-18 or more, and by
leaving the submatrix to the chains below that.

References are Newton-Schulz runs in numpy's long double (64 or 113 bits of mantissa).

Bound on a coupling block's relative error (Frobenius, clusters of m functions): a
chain's product entry is off by (2m) 2^-53 (|A| |B|)_ij, || |A| |B| ||_F of the block is
at most 2 sqrt(m) times its own norm, Newton-Schulz runs 25 products, and an error E
moves sign(a) by |E| / gap."""
import numpy as np
import pytest

from synth.water import BSRMatrix, bsr_to_dense, make_water

pytestmark = pytest.mark.gpu

M, GAP = 12, 0.3
BOUND = 25 * 2 * M * 2.0 ** -53 * 2 * np.sqrt(M) / GAP
SIMT, RESIDUES = 2, 7  # kernel classes


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g
    g.build()
    import paper_2004_10811_gb300 as p
    return p


def cluster(rng):
    q, _ = np.linalg.qr(rng.standard_normal((M, M)))
    w = GAP + (1 - GAP) * rng.random(M)
    w[: M // 3] *= -1
    a = (q * w) @ q.T
    return 0.5 * (a + a.T)


def pairs(eps, seed=3):
    """Pairs of gapped clusters, pair i coupled by eps[i]; every pair is a submatrix."""
    rng = np.random.default_rng(seed)
    vals, cols = [], []
    for i, e in enumerate(eps):
        c = e * rng.standard_normal((M, M))
        vals += [cluster(rng), c, c.T, cluster(rng)]
        cols += [2 * i, 2 * i + 1] * 2
    k = 2 * len(eps)
    return BSRMatrix(np.full(k, M, np.int32), np.arange(k + 1, dtype=np.int64) * 2, np.array(cols, np.int32),
                     np.concatenate([v.ravel() for v in vals]))


def dense(m, i):
    v = m.vals.reshape(-1, 2, 2, M, M)[i]
    return v.transpose(0, 2, 1, 3).reshape(2 * M, 2 * M)


def sign_long(a):
    """sign(a) of a symmetric matrix in long double."""
    x = a.astype(np.longdouble) / np.linalg.norm(a, 2)
    for _ in range(60):
        y = x @ x
        x = (3 * x - x @ y) / 2
        if np.max(np.abs(y - np.eye(len(a)))) < 1e-9:
            break
    y = x @ x
    return (3 * x - x @ y) / 2


def run(pkg, m, kT=0.0, **kw):
    import torch
    K = torch.from_numpy(m.vals).cuda()
    with pkg.Plan.from_bsr(m, prec="fp64", kT=kT, timing=True, **kw) as plan:
        D = plan.sign(K, 0.0, out=torch.full_like(K, float("nan"))).cpu().numpy()
        return D, plan.stats()


def off_block_error(D, want):
    """Relative error of the two coupling blocks of pair 0."""
    got = D.reshape(-1, M, M)
    e = max(np.linalg.norm((got[1] - want[:M, M:]).astype(float)), np.linalg.norm((got[2] - want[M:, :M]).astype(float)))
    return e / np.linalg.norm(want[:M, M:].astype(float))


@pytest.mark.parametrize("eps", [0.1, 1e-2, 1e-3, 1e-4, 1e-5, 1e-6, 1e-8, 1e-10, 1e-13, 1e-16, 1e-25, 1e-100])
def test_weak_coupling(pkg, eps):
    m = pairs([eps])
    want = -0.5 * sign_long(dense(m, 0))
    for kw in ({}, {"groups": np.zeros(2, int)}, {"beta_mode": 1}):
        D, s = run(pkg, m, **kw)
        assert off_block_error(D, want) <= BOUND
        chains = s["kernel_launches"][SIMT] > 0
        assert chains or eps > 1e-7
        assert not chains or eps < 1e-3


@pytest.mark.parametrize("eps", [1e-2, 1e-4, 1e-8, 1e-12, 1e-25])
def test_weak_coupling_inside_a_block(pkg, eps):
    """The same pair of clusters as one block of 24 functions."""
    m = pairs([eps])
    a = dense(m, 0)
    one = BSRMatrix(np.array([2 * M], np.int32), np.array([0, 1]), np.array([0], np.int32), a.ravel().copy())
    D, s = run(pkg, one)
    want = -0.5 * sign_long(a)[:M, M:]
    e = np.linalg.norm((D.reshape(2 * M, 2 * M)[:M, M:] - want).astype(float)) / np.linalg.norm(want.astype(float))
    assert e <= BOUND and (s["kernel_launches"][SIMT] > 0) == (eps < 1e-5)


@pytest.mark.parametrize("eps", [1e-2, 1e-4, 1e-6, 1e-10, 1e-16])
@pytest.mark.parametrize("kT", [0.05, 0.3])
def test_weak_coupling_fermi(pkg, eps, kT):
    """f(a)'s coupling block to first order in eps is q1 (L o (q1^T c q2)) q2^T with the
    divided differences L of f; the second order is eps^2 below, and the chains' bound
    has the series' products (16 baby steps, T_16's errors by 256 / (4 kT), and the giant
    steps) for Newton-Schulz's.  Beyond degree m the series' derivative is off by about
    m^2 times its truncation."""
    m = pairs([eps])
    a = dense(m, 0)
    w1, q1 = np.linalg.eigh(a[:M, :M])
    w2, q2 = np.linalg.eigh(a[M:, M:])
    f1, f2 = 1 / (1 + np.exp(w1 / kT)), 1 / (1 + np.exp(w2 / kT))
    L = (f1[:, None] - f2[None]) / (w1[:, None] - w2[None])
    want = q1 @ (L * (q1.T @ a[:M, M:] @ q2)) @ q2.T
    D, s = run(pkg, m, kT=kT)
    got = D.reshape(-1, M, M)[1]
    G = (s["poly_degree"] + 16) // 16
    bound = 2 * M * 2.0 ** -53 * 2 * np.sqrt(M) * (256 / (4 * kT) + G * G) + (10 * eps / kT) ** 2
    bound += 2 * s["poly_trunc"] * s["poly_degree"] ** 2 / np.min(np.abs(L))
    assert np.linalg.norm(got - want) / np.linalg.norm(want) <= bound
    assert (s["kernel_launches"][SIMT] > 0) == (eps < 1e-5)


def test_routes_in_one_wave(pkg):
    """Submatrices of the chains among others: theirs are the chains' results to the bit,
    the others' those of a wave of their own."""
    eps = [0.05, 1e-9, 0.05, 0.0, 1e-30]
    m = pairs(eps)
    D, s = run(pkg, m)
    simt, s2 = run(pkg, m, workspace_cap_bytes=30 * 64 * 64)
    assert s2["kernel_launches"][RESIDUES] == 0 < s["kernel_launches"][RESIDUES] and s["kernel_launches"][SIMT] > 0
    per = 4 * M * M
    strong, _ = run(pkg, pairs([0.05, 0.0, 0.05, 0.0, 0.0]))
    for i, e in enumerate(eps):
        mine = D[i * per:(i + 1) * per]
        if 0 < e < 1e-5:
            assert np.array_equal(mine, simt[i * per:(i + 1) * per])
        elif e > 0:
            assert np.array_equal(mine, strong[i * per:(i + 1) * per])
        else:
            assert np.all(mine.reshape(4, M, M)[1:3] == 0.0)


def test_routes_in_one_wave_fermi(pkg):
    eps = [0.05, 1e-9, 0.05, 0.0]
    m = pairs(eps)
    D, s = run(pkg, m, kT=0.1)
    simt, s2 = run(pkg, m, kT=0.1, workspace_cap_bytes=110 * 64 * 64)
    assert s2["kernel_launches"][RESIDUES] == 0 < s["kernel_launches"][RESIDUES] and s["kernel_launches"][SIMT] > 0
    err = np.abs(D - simt).reshape(-1, 4, M, M).max(axis=(2, 3))
    assert np.max(err) <= 1e-12 and np.max(err[1, 1:3]) <= 1e-12 * 1e-9 * 100


def test_tiny_level(pkg):
    """A decoupled level far below the grid keeps its sign."""
    m = BSRMatrix(np.array([1, 1], np.int32), np.array([0, 2, 4]), np.array([0, 1, 0, 1], np.int32),
                  np.array([1.0, 0.0, 0.0, -1e-22]))
    D, s = run(pkg, m, max_iter=200)
    assert s["not_converged"] == 0
    assert np.max(np.abs(D - [0.0, 0.0, 0.0, 1.0])) <= 1e-14


@pytest.mark.parametrize("block", [6, 3])
def test_water_blocks(pkg, block):
    """Liquid water: no submatrix needs the chains, and over the blocks of D the largest
    relative error is no larger than theirs."""
    lo, hi = ((2, -1.0, -0.3), (4, 0.3, 1.0)) if block == 6 else ((1, -1.0, -0.3), (2, 0.3, 1.0))
    m = make_water(64, block, 5.0, lo, hi, seed=11)
    D, s = run(pkg, m)
    ld = (s["n_max"] + 63) // 64 * 64
    simt, _ = run(pkg, m, workspace_cap_bytes=30 * ld * ld)
    assert s["kernel_launches"][SIMT] == 0
    a = bsr_to_dense(m)
    worst = [0.0, 0.0]
    for j in (0, 17, 40):
        rows = m.col_idx[m.row_ptr[j]:m.row_ptr[j + 1]]
        idx = (rows[:, None] * block + np.arange(block)).ravel()
        sub = sign_long(a[np.ix_(idx, idx)])
        at = int(np.flatnonzero(rows == j)[0]) * block
        for t, i in enumerate(rows):
            want = (np.eye(block) * (i == j) - sub[t * block:(t + 1) * block, at:at + block]) / 2
            p = int(m.row_ptr[i] + np.flatnonzero(m.col_idx[m.row_ptr[i]:m.row_ptr[i + 1]] == j)[0])
            for k, got in enumerate((D, simt)):
                e = got[p * block * block:(p + 1) * block * block].reshape(block, block) - want
                worst[k] = max(worst[k], float(np.linalg.norm(e.astype(float)) / np.linalg.norm(want.astype(float))))
    assert worst[0] <= worst[1], worst



@pytest.mark.parametrize("beta_mode", [0, 1])
def test_residual_sums(pkg, beta_mode):
    """||X_0^2 - I||_F / sqrt(n), summed as FP64 sums it: a product entry is off by 2^-73
    and the rounding of X_0, n^(1/2) 2^-53, against a residual of order 1."""
    import torch
    m = make_water(40, 6, 5.0, (2, -1.0, -0.3), (4, 0.3, 1.0), seed=21)
    K = torch.from_numpy(m.vals).cuda()
    with pkg.Plan.from_bsr(m, prec="fp64", max_iter=1, beta_mode=beta_mode) as plan:
        plan.sign(K, 0.0, allow_not_converged=True)
        sub = plan.sub_stats()
    iters, resid, beta = sub["iters"], sub["resid"], sub["beta"]
    a = bsr_to_dense(m)
    for j in (0, 13, 39):
        rows = m.col_idx[m.row_ptr[j]:m.row_ptr[j + 1]]
        idx = (rows[:, None] * 6 + np.arange(6)).ravel()
        x = a[np.ix_(idx, idx)] / beta[j]
        want = np.linalg.norm(x @ x - np.eye(len(idx))) / np.sqrt(len(idx))
        assert iters[j] == 1 and abs(resid[j] / want - 1) <= len(idx) ** 0.5 * 2.0 ** -50


@pytest.mark.parametrize("beta_mode", [0, 1])
def test_values_beyond_fp32(pkg, beta_mode):
    """Entries beyond FP32's range saturate the spectral bound, so the iteration diverges:
    it says so after one step, and the mu search ends there, instead of running to the
    step cap on numbers that the grid cannot hold."""
    import torch
    m = make_water(20, 4, 4.0, (1, -1.0, -0.3), (3, 0.3, 1.2), seed=2)
    K = torch.from_numpy(m.vals * 1e100).cuda()
    with pkg.Plan.from_bsr(m, prec="fp64", beta_mode=beta_mode) as plan:
        plan.sign(K, 0.0, allow_not_converged=True)
        s = plan.stats()
        assert s["not_converged"] == 20 and s["iters_max"] <= 2
        with pytest.raises(pkg.SubmatError) as e:
            plan.mu_search(K, 20.0, mu0=0.0, tol=1e-9)
        assert e.value.name == "NOT_CONVERGED" and "diverged" in str(e.value)


@pytest.mark.parametrize("kT", [0.05, 0.3])
def test_fermi_moduli_in_two_parts(pkg, kT):
    """A workspace that holds 162 to 198 bytes for each entry of the largest submatrix:
    the residue sets hold half of the moduli at a time, with the same bits as a result
    (one block column a plan, so that the scale is the submatrix's own)."""
    import torch
    m = make_water(40, 6, 5.0, (2, -1.0, -0.3), (4, 0.3, 1.0), seed=21)
    K = torch.from_numpy(m.vals).cuda()
    ld = (6 * int(np.diff(m.row_ptr).max()) + 63) // 64 * 64
    for j in (3, 30):
        kw = dict(prec="fp64", kT=kT, columns=(j, j + 1), timing=True)
        got = []
        for cap in (0, 163 * ld * ld):
            with pkg.Plan.from_bsr(m, workspace_cap_bytes=cap, **kw) as plan:
                got.append(plan.sign(K, 0.0, out=torch.zeros_like(K)))
                s = plan.stats()
            assert s["kernel_launches"][RESIDUES] > 0 == s["kernel_launches"][SIMT]
        # 9 baby products and the giant steps, each in two launches
        assert s["kernel_launches"][RESIDUES] == 2 * s["iters_max"]
        assert torch.equal(got[0], got[1]) and float(got[0].abs().max()) > 0.1
