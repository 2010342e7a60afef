"""The work that programs have this library do, as cases to time: D builds of
block-sparse Kohn-Sham matrices at the three precisions, forward plus backward,
the finite-temperature mu search, grouped submatrices and the allocation-free
dense call, from one small matrix to batches of thousands of submatrices.

Systems are the seeded water-like boxes of the tests and the benchmark: molecules
on a jittered lattice at liquid density, a block stored within a distance cutoff,
off-diagonal entries N(0, 1) 0.05 exp(-r / 2 A), diagonal blocks with occupied
levels in [-1, -gap] and virtual ones in [gap, 1] (1.5 for 23 functions).  The geometry (and with it the
pattern) belongs to the case, as in an SCF loop; the values belong to the seed.
"""
import math

import numpy as np
import torch

import paper_2004_10811_gb300 as submat
from paper_2004_10811_gb300 import grouping
from paper_2004_10811_gb300.submat import dense_sign_noalloc

RHO = 0.03343     # molecules per cubic Angstrom, liquid water
CAP = 48 << 30    # device workspace granted to a plan: larger batches run in waves


def case(name, call, prec="mixed", mols=32, blocks="6", rc=6.0, gap=0.3, mu=0.0, kT=0.0, adjoint=0, symmetrize=False,
         slab=False):
    c = {"call": call, "prec": prec, "mols": mols, "blocks": blocks, "rc": rc, "gap": gap, "mu": mu, "kT": kT,
         "adjoint": adjoint, "symmetrize": symmetrize, "slab": slab}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one molecule cluster's dense matrix inside a host code that owns the device memory: the smallest call
        case("dense_191", "dense", "fp64", mols=191),
        # the smallest workload: 32 molecules, one D build of an SCF step, bound by launches and latency
        case("mixed_water32", "sign", mols=32, rc=6.0),
        # liquid next to vapour: the ragged mix of small and middle submatrices of a slab
        case("mixed_slab", "sign", mols=4096, rc=8.1, slab=True),
        # the benchmark's recipe (6 functions, 9 A, narrow gap) at the size of one rank's share, in waves
        case("mixed_b6_rc9", "sign", mols=4096, rc=9.0, gap=0.15),
        # the benchmark's second recipe: 23 functions, submatrices above 1024
        case("mixed_b23_rc8", "sign", mols=216, blocks="23", rc=8.0),
        # pairs of molecules found by k-means share a submatrix
        case("mixed_pairs", "pairs", mols=1000, rc=9.0, gap=0.15),
        # the default precision: a reference-quality D build
        case("fp64_b6", "sign", "fp64", mols=216, rc=8.0),
        # single precision D build, no correction
        case("fp32_b23", "sign", "fp32", mols=125, blocks="23", rc=7.0),
        # finite temperature at the default precision, one block per atom (13 + 5 + 5 functions)
        case("fermi_fp64_atoms", "sign", "fp64", mols=240, blocks="13,5,5", rc=6.5, kT=0.05),
        # canonical ensemble at finite temperature: the Newton search for mu
        case("fermi_mu_fp32", "mu", "fp32", mols=216, rc=8.0, kT=0.05, mu=0.1),
        # D and the gradient of a loss on it, default adjoint
        case("grad_b6", "grad", mols=216, rc=8.0),
        # the same with the tensor-core adjoint on larger blocks
        case("grad_tc_b23", "grad", mols=64, blocks="23", rc=6.0, adjoint=1),
    ]


# -- geometry and pattern ------------------------------------------------------
def _lattice(rng, n, lengths):
    """n sites of a jittered simple lattice filling a box, in lattice order."""
    h = (float(np.prod(lengths)) / n) ** (1.0 / 3.0)
    m = np.maximum(1, np.ceil(lengths / h - 1e-9)).astype(np.int64)
    site = np.sort(rng.permutation(int(np.prod(m)))[:n])
    xyz = np.stack([site // (m[1] * m[2]), site // m[2] % m[1], site % m[2]], 1) + 0.5
    return np.mod((xyz + rng.uniform(-0.2, 0.2, (n, 3))) * (lengths / m), lengths)


def _geometry(c):
    """Positions (a site per block), the periodic box and the block sizes.  A
    slab holds 15/16 of its molecules as a liquid layer, the rest as vapour."""
    n = int(c["mols"])
    sizes = [int(b) for b in c["blocks"].split(",")]
    rng = np.random.Generator(np.random.PCG64(7919 + n))
    if c["slab"]:
        few = n // 16
        side = 40.0 * (n / 4096.0) ** (1.0 / 3.0)
        liquid, vapour = (np.array([side, side, k / rho / side ** 2]) for k, rho in ((n - few, RHO), (few, 0.2 * RHO)))
        xyz = np.concatenate([_lattice(rng, n - few, liquid), _lattice(rng, few, vapour) + [0, 0, liquid[2]]])
        box = liquid + [0, 0, vapour[2]]
    else:
        box = np.full(3, (n / RHO) ** (1.0 / 3.0))
        xyz = _lattice(rng, n, box)
    return xyz, box, np.array([sizes[i % len(sizes)] for i in range(n)], dtype=np.int64)


def _pattern(c, device):
    xyz, box, bs = _geometry(c)
    x, side = torch.from_numpy(xyz).to(device), torch.from_numpy(box).to(device)
    rows, cols, dist = [], [], []
    for i in range(0, len(xyz), 1024):
        d = x[i:i + 1024, None] - x[None]
        r = (d - side * torch.round(d / side)).square().sum(-1).sqrt()
        a, b = torch.nonzero(r < c["rc"], as_tuple=True)
        rows.append(a + i), cols.append(b), dist.append(r[a, b])
    rows, cols, dist = torch.cat(rows), torch.cat(cols), torch.cat(dist)
    return xyz, box, bs, rows, cols, dist


def _maps(bs, rows, cols):
    """Per value: block, row and column function; the value's transpose; block starts."""
    dev = rows.device
    n = len(bs)
    b = torch.from_numpy(bs).to(dev)
    area = b[rows] * b[cols]
    ptr = torch.cat([torch.zeros(1, dtype=torch.int64, device=dev), area.cumsum(0)])
    p = torch.repeat_interleave(torch.arange(len(rows), device=dev), area)
    e = torch.arange(len(p), device=dev) - ptr[p]
    r, q = e // b[cols[p]], e % b[cols[p]]
    key = rows * n + cols
    tp = torch.searchsorted(key, cols * n + rows)
    start = torch.cat([torch.zeros(1, dtype=torch.int64, device=dev), b.cumsum(0)])
    return {"p": p, "fr": start[rows[p]] + r, "fc": start[cols[p]] + q, "t": ptr[tp[p]] + q * b[rows[p]] + r,
            "ptr": ptr, "start": start}


def _occupied(b):
    return b // 2 if b <= 6 else max(1, b // 5)


def _values(c, bs, rows, cols, dist, maps, seed):
    dev = rows.device
    g = torch.Generator(device=dev).manual_seed(int(seed))
    p = maps["p"]
    v = torch.randn(len(p), generator=g, device=dev, dtype=torch.float64)
    v *= (0.05 * torch.exp(-dist / 2.0))[p]
    v = torch.where((rows < cols)[p], v, v[maps["t"]])
    diag = torch.nonzero(rows == cols).flatten()
    for b in sorted(set(bs.tolist())):
        at = torch.from_numpy(np.flatnonzero(bs == b)).to(dev)
        lo = _occupied(b)
        u = torch.rand(len(at), b, generator=g, device=dev, dtype=torch.float64)
        ev = c["gap"] + ((1.5 if b == 23 else 1.0) - c["gap"]) * u
        ev[:, :lo] = -c["gap"] - (1.0 - c["gap"]) * u[:, :lo]
        q, _ = torch.linalg.qr(torch.randn(len(at), b, b, generator=g, device=dev, dtype=torch.float64))
        d = (q * ev[:, None]) @ q.transpose(1, 2)
        idx = maps["ptr"][diag[at]][:, None] + torch.arange(b * b, device=dev)
        v[idx] = (0.5 * (d + d.transpose(1, 2))).reshape(len(at), -1)
    return v.contiguous()


def _dense_matrix(n, seed, device):
    """A cluster's Hamiltonian: levels on both sides of a gap, mixed by a random rotation."""
    g = torch.Generator(device=device).manual_seed(int(seed))
    u = 0.3 + 0.7 * torch.rand(n, generator=g, device=device, dtype=torch.float64)
    u[: n // 3] *= -1.0
    q, _ = torch.linalg.qr(torch.randn(n, n, generator=g, device=device, dtype=torch.float64))
    a = (q * u) @ q.T
    return (0.5 * (a + a.T)).contiguous()


def _labels(c, xyz, box):
    k = max(1, len(xyz) // 2)
    return grouping.periodic_kmeans(xyz, box, k, seed=1).astype(np.int32)


# -- one case --------------------------------------------------------------------
def prepare(case, seed):
    c = case
    dev = torch.device("cuda")
    if c["call"] == "dense":
        return {"case": c, "K": _dense_matrix(c["mols"], seed, dev)}
    xyz, box, bs, rows, cols, dist = _pattern(c, dev)
    maps = _maps(bs, rows, cols)
    K = _values(c, bs, rows, cols, dist, maps, seed)
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(rows.cpu().numpy(), minlength=len(bs)))])
    kw = dict(prec=c["prec"], kT=c["kT"], adjoint_mode=c["adjoint"], symmetrize=c["symmetrize"],
              workspace_cap_bytes=CAP)
    if c["call"] == "pairs":
        kw["groups"] = _labels(c, xyz, box)
    plan = submat.Plan(bs, row_ptr, cols.cpu().numpy(), **kw)
    s = {"case": c, "K": K, "plan": plan}
    if c["call"] == "grad":
        s["fn"] = submat.make_autograd_sign(plan)
        s["K"] = K.requires_grad_()
        s["Dbar"] = _upstream(K, seed)
    if c["call"] == "mu":
        s["n_el"] = float(sum(_occupied(int(b)) for b in bs))
    return s


def _upstream(K, seed):
    g = torch.Generator(device=K.device).manual_seed(int(seed) + 77)
    return torch.randn(len(K), generator=g, device=K.device, dtype=torch.float64)


def run(state):
    c, K = state["case"], state["K"]
    if c["call"] == "dense":
        return {"D": dense_sign_noalloc(K, c["mu"])[0]}
    plan = state["plan"]
    if c["call"] == "grad":
        D = state["fn"](K, c["mu"])
        (Kbar,) = torch.autograd.grad(D, K, state["Dbar"])
        return {"D": D.detach(), "Kbar": Kbar}
    if c["call"] == "mu":
        mu, D, _ = plan.mu_search(K, state["n_el"], mu0=c["mu"], tol=1e-6)
        return {"D": D, "mu": mu}
    D = plan.sign(K, c["mu"])
    return {"D": D, "n_el": plan.trace(D)}


# -- what a pass cannot do without ---------------------------------------------------
def _dims(c):
    """Dimension of every submatrix, and the number of stored values."""
    xyz, box, bs, rows, cols, _ = _pattern(c, torch.device("cpu"))
    rows, cols = rows.numpy(), cols.numpy()
    vals = float((bs[rows] * bs[cols]).sum())
    if c["call"] != "pairs":
        return np.bincount(rows, weights=bs[cols], minlength=len(bs)), vals
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=len(bs)))])
    return grouping.group_dims(bs, row_ptr, cols, _labels(c, xyz, box))[0].astype(float), vals


def work(case):
    """Every value of K read and of D written once; flops: about ten Newton-Schulz
    steps of two symmetric products (n^3 flops each), at finite temperature a
    polynomial of degree ~32 / kT by 2 sqrt(degree / 2) of them; a gradient takes
    three times the products besides, a mu search about five evaluations."""
    c = case
    if c["call"] == "dense":
        n = float(c["mols"])
        return {"bytes": 16.0 * n * n, "flops": 20.0 * n ** 3}
    dims, vals = _dims(c)
    products = 2.0 * math.sqrt(16.0 / c["kT"]) if c["kT"] > 0 else 20.0
    flops = products * float((dims ** 3).sum())
    if c["call"] == "grad":
        return {"bytes": 32.0 * vals, "flops": 4.0 * flops}
    return {"bytes": 16.0 * vals, "flops": flops * (5.0 if c["call"] == "mu" else 1.0)}


# -- 64-bit reference: eigendecomposition of every submatrix -----------------------
def _f(x, kT):
    return torch.sigmoid(-x / kT) if kT > 0 else 0.5 - 0.5 * torch.sign(x)


def _eigh_seconds(dims):
    return float((3e-3 + 2.2e-10 * dims ** 3).sum())


def exact(case, seed):
    c = case
    dev = torch.device("cuda")
    if c["call"] == "dense":
        w, q = torch.linalg.eigh(_dense_matrix(c["mols"], seed, dev))
        return {"D": (q * _f(w - c["mu"], 0.0)) @ q.T}
    dims, _ = _dims(c)
    if _eigh_seconds(dims) > 14.0:
        return None
    xyz, box, bs, rows, cols, dist = _pattern(c, dev)
    maps = _maps(bs, rows, cols)
    K = _values(c, bs, rows, cols, dist, maps, seed)
    n = int(bs.sum())
    A = torch.zeros(n, n, device=dev, dtype=torch.float64)
    A[maps["fr"], maps["fc"]] = K
    start = maps["start"].cpu().numpy()
    hr, hc = rows.cpu().numpy(), cols.cpu().numpy()
    ptr = np.concatenate([[0], np.cumsum(np.bincount(hr, minlength=len(bs)))])
    nb = [hc[ptr[j]:ptr[j + 1]] for j in range(len(bs))]
    members = [[j] for j in range(len(bs))]
    if c["call"] == "pairs":
        lab = _labels(c, xyz, box)
        members = [np.flatnonzero(lab == k).tolist() for k in range(int(lab.max()) + 1)]
    eig = []
    for g in members:
        blocks = np.unique(np.concatenate([nb[j] for j in g]))
        idx = torch.from_numpy(np.concatenate([np.arange(start[i], start[i + 1]) for i in blocks])).to(dev)
        J = torch.from_numpy(np.concatenate([np.arange(start[j], start[j + 1]) for j in g])).to(dev)
        w, q = torch.linalg.eigh(A[idx][:, idx])
        eig.append((idx, J, torch.searchsorted(idx, J), w, q))
    mu = c["mu"]
    if c["call"] == "mu":
        want = float(sum(_occupied(int(b)) for b in bs))
        lo, hi = -3.0, 3.0
        wts = [(w, q[l].square().sum(0)) for _, _, l, w, q in eig]
        w_all, q_all = torch.cat([w for w, _ in wts]), torch.cat([u for _, u in wts])
        for _ in range(60):
            mu = 0.5 * (lo + hi)
            if float((q_all * _f(w_all - mu, c["kT"])).sum()) < want:
                lo = mu
            else:
                hi = mu
    Dd = torch.zeros_like(A)
    for idx, J, l, w, q in eig:
        Dd[idx[:, None], J[None]] = (q * _f(w - mu, c["kT"])) @ q[l].T
    D = Dd[maps["fr"], maps["fc"]]
    if c["symmetrize"]:
        D = 0.5 * (D + D[maps["t"]])
    if c["call"] == "mu":
        return {"D": D, "mu": mu}
    if c["call"] != "grad":
        return {"D": D, "n_el": float(Dd.diagonal().sum())}
    G = torch.zeros_like(A)
    G[maps["fr"], maps["fc"]] = _upstream(K, seed)
    out = torch.zeros_like(A)
    for idx, J, l, w, q in eig:
        x = w - mu
        f = _f(x, c["kT"])
        dx = x[:, None] - x[None]
        if c["kT"] > 0:
            near = dx.abs() < 1e-7
            d1 = -f * (1.0 - f) / c["kT"]
            L = torch.where(near, 0.5 * (d1[:, None] + d1[None]), (f[:, None] - f[None]) / dx.masked_fill(near, 1.0))
        else:
            same = f[:, None] == f[None]
            L = torch.where(same, torch.zeros_like(dx), (f[:, None] - f[None]) / dx.masked_fill(same, 1.0))
        inner = (q.T @ G[idx][:, J]) @ q[l]
        out[idx[:, None], idx[None]] += q @ (L * inner) @ q.T
    return {"D": D, "Kbar": out[maps["fr"], maps["fc"]]}


# -- more of the same ranges -----------------------------------------------------------
def draw(rng):
    """Another call of the ranges above: kind, precision, block sizes, cutoff, gap,
    temperature and system size; small next to large, within the largest's cost."""
    while True:
        call = rng.choice(("dense", "sign", "sign", "sign", "pairs", "grad", "mu"))
        if call == "dense":
            return case(None, "dense", "fp64", mols=int(round(math.exp(rng.uniform(math.log(24), math.log(512))))),
                        mu=round(rng.uniform(-0.1, 0.1), 3))
        c = case(None, call)
        c["mols"] = int(round(math.exp(rng.uniform(math.log(27), math.log(2500)))))
        c["blocks"] = rng.choice(("6", "6", "23", "13,5,5", "6,2,6,1", "9"))
        c["gap"] = rng.choice((0.15, 0.3)) if c["blocks"] == "6" else 0.3
        c["mu"] = round(rng.uniform(-0.02, 0.02), 3)
        c["slab"] = call == "sign" and c["mols"] >= 1000 and rng.random() < 0.25
        half = 20.0 * (c["mols"] / 4096.0) ** (1.0 / 3.0) if c["slab"] else 0.5 * (c["mols"] / RHO) ** (1.0 / 3.0)
        c["rc"] = round(min(rng.uniform(4.0, 9.0), 0.99 * half), 2)
        c["prec"] = "mixed" if call == "pairs" else rng.choice(("mixed", "fp64", "fp32"))
        if call == "mu" or (call != "pairs" and c["prec"] != "mixed" and rng.random() < 0.4):
            c["prec"] = rng.choice(("fp64", "fp32")) if c["prec"] == "mixed" else c["prec"]
            c["kT"] = rng.choice((0.05, 0.1))
        if call == "grad" and c["prec"] == "mixed":
            c["adjoint"] = rng.choice((0, 1))
        if call == "sign":
            c["symmetrize"] = rng.random() < 0.25
        if _seconds(c) <= 0.35:
            return c


def _seconds(c):
    """About what the call takes, from the rates in standard-count flops a second."""
    mean = float(np.mean([int(b) for b in c["blocks"].split(",")]))
    n = mean * max(1.0, RHO * 4.19 * c["rc"] ** 3) * (1.35 if c["call"] == "pairs" else 1.0)
    count = c["mols"] / (2.0 if c["call"] == "pairs" else 1.0)
    rate = {"fp64": 1.5e12, "fp32": 3e13, "mixed": 1e14}[c["prec"]]
    if c["call"] == "grad" and c["prec"] == "mixed":
        rate = 1e14 if c["adjoint"] else 2.5e13
    products = 45.0 if c["kT"] > 0 else 24.0
    scale = {"grad": 4.0, "mu": 7.0}.get(c["call"], 1.0)
    return 2e-3 + scale * products * 2.0 * count * n ** 3 / rate
