"""Performance cases: the work a user of this framework has it do, through its public entry points.

Kinds of case (``kind``):
  eri3c    Eri3cPlan(...).execute(out): one class of integral blocks written to device memory
  host     eri3c_host(...): the same from host shell tables into a page-locked host array
  dfj      DFJPlan(...).execute(D, c): gamma and J of one density (SCF Coulomb build)
  multi    DFJPlan(...).execute_multi(Ds, cs): several densities at once
  fit      MetricPlan.execute, cholesky, cholesky_solve: fitting metric, factor, solves
  grad     DFJEnergy.apply(R, ...) and backward(): energy and dE/dR at a new geometry
  batch    Batch(...).bind(...).execute(mode=2): several molecules' builds in one launch

Sizes follow the benchmark's sweep (every (la, lb <= 4 | lc <= 6) class, K_a = K_b in
{1, 3, 6}, up to 512 ket shells), its 64 x 32 small call, its cluster recipes (DF-J: 4s3p2d1f
orbitals, gradient and batch: 3s2p2d1f1g) and its eight-density build, at molecule sizes that
keep a pass below two seconds.

``exact`` evaluates the same outputs in 64 bits with torch alone: McMurchie-Davidson Hermite
integrals, the ket by Hobson's theorem, V and its factor by torch.linalg.
"""
import math

import numpy as np
import torch

import paper_2210_03192_gb300 as lx
from paper_2210_03192_gb300 import workloads as W

ORB = {"dfj": W.ORB_RECIPE_DFJ, "small": W.ORB_RECIPE_SMALL}
AUX = {"dfj": W.AUX_RECIPE_DFJ, "grad": W.AUX_RECIPE_GRAD, "batch": W.AUX_RECIPE_BATCH}


def listed():
    return [
        # the smallest call: (pp|d), 64 pairs x 32 ket shells; latency and launches decide
        dict(name="ppd_64x32", kind="eri3c", la=1, lb=1, lc=2, ka=1, kb=1, kc=1, npair=64, naux=32, pure=True,
             box=10.0, elo=0.1, ehi=100.0),
        # a low, deeply contracted class: valence p and s shells of a contracted basis
        dict(name="psf_k6", kind="eri3c", la=1, lb=0, lc=3, ka=6, kb=6, kc=1, npair=2047, naux=509, pure=True,
             box=20.0, elo=0.05, ehi=1e4),
        # mid angular momentum and contraction, odd pair count
        dict(name="ddf_k3", kind="eri3c", la=2, lb=2, lc=3, ka=3, kb=3, kc=1, npair=1023, naux=512, pure=True,
             box=20.0, elo=0.05, ehi=1e4),
        # uncontracted polarisation functions: the contracted stages decide
        dict(name="ffg_k1", kind="eri3c", la=3, lb=3, lc=4, ka=1, kb=1, kc=1, npair=1024, naux=512, pure=True,
             box=20.0, elo=0.05, ehi=1e4),
        # the sweep's dominant class (gg|i), K = 6, on an eighth of its pairs
        dict(name="ggi_k6", kind="eri3c", la=4, lb=4, lc=6, ka=6, kb=6, kc=1, npair=512, naux=512, pure=True,
             box=20.0, elo=0.05, ehi=1e4),
        # Cartesian bra, contracted ket, ragged sizes
        dict(name="dpd_cart", kind="eri3c", la=2, lb=1, lc=2, ka=3, kb=2, kc=2, npair=777, naux=301, pure=False,
             box=10.0, elo=0.1, ehi=100.0),
        # host arrays in, host blocks out: the whole call, planning and copies included
        dict(name="host_fdf_k3", kind="host", la=3, lb=2, lc=3, ka=3, kb=3, kc=1, npair=500, naux=300, pure=True,
             box=20.0, elo=0.05, ehi=1e4),
        # Coulomb build of one density, 32 atoms
        dict(name="dfj_32", kind="dfj", nx=4, ny=4, nz=2, orb="dfj", aux="dfj", contract=False),
        # response or open-shell builds: eight densities on 16 atoms
        dict(name="multi8_16", kind="multi", nx=4, ny=2, nz=2, orb="dfj", aux="dfj", nd=8),
        # fitting metric, its factor and a solve for three right-hand sides, 3,078 functions
        dict(name="fit_27", kind="fit", nx=3, ny=3, nz=3, nrhs=3),
        # energy and forces at a new geometry, 12 atoms with g functions
        dict(name="grad_12", kind="grad", nx=3, ny=2, nz=2, orb="small", aux="grad"),
        # three small molecules of uneven size in one launch
        dict(name="batch_3", kind="batch", n0=4, n1=7, n2=12),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eri3c"] * 5 + ["host", "dfj", "dfj", "multi", "fit", "grad", "batch"])
    if kind in ("eri3c", "host"):
        la, lb, lc = rng.randint(0, 4), rng.randint(0, 4), rng.randint(0, 6)
        ka, kb = rng.choice([1, 1, 2, 3, 6]), rng.choice([1, 1, 2, 3, 6])
        kc = rng.choice([1, 1, 1, 2])
        npair, naux = _log(rng, 16, 2048), _log(rng, 17, 512)
        c = dict(kind=kind, la=la, lb=lb, lc=lc, ka=ka, kb=kb, kc=kc, npair=npair, naux=naux,
                 pure=rng.random() < 0.8, box=20.0, elo=0.05, ehi=1e4)
        top = work(listed()[4])["flops"] * (1.0 if kind == "eri3c" else 0.25)
        while work(c)["flops"] > 0.6 * top or work(c)["bytes"] > 2.0e9:
            c["npair"] = max(1, c["npair"] * 2 // 3)
        return c
    dims = lambda hi: sorted((rng.randint(1, 4) for _ in range(3)), reverse=True)  # noqa: E731
    if kind in ("dfj", "multi", "grad"):
        most = {"dfj": 24, "multi": 12, "grad": 9}[kind]
        nx, ny, nz = dims(4)
        while nx * ny * nz > most or nx * ny * nz < 2:
            nx, ny, nz = dims(4)
        if kind == "dfj":
            return dict(kind=kind, nx=nx, ny=ny, nz=nz, orb=rng.choice(["dfj", "small"]),
                        aux=rng.choice(["dfj", "grad"]), contract=rng.random() < 0.5)
        if kind == "multi":
            return dict(kind=kind, nx=nx, ny=ny, nz=nz, orb="dfj", aux="dfj", nd=rng.randint(2, 8))
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, orb="small", aux=rng.choice(["dfj", "grad"]))
    if kind == "fit":
        return dict(kind=kind, nx=rng.randint(1, 3), ny=rng.randint(1, 3), nz=rng.randint(1, 2),
                    nrhs=rng.choice([1, 1, 2, 3, 5, 8]))
    return dict(kind=kind, n0=rng.randint(2, 6), n1=rng.randint(3, 8), n2=rng.randint(4, 11))


# ------------------------------------------------------------------ inputs


def _problem(c, seed):
    return W.class_problem(c["la"], c["lb"], c["lc"], c["npair"], c["naux"], c["ka"], c["kb"], c["kc"],
                           box=c["box"], exp_lo=c["elo"], exp_hi=c["ehi"], seed=seed)


def _nao(b):
    return int((2 * b.l.astype(np.int64) + 1).sum())


def _density(seed, nd, n):
    """nd densities C C^T, C an n x (n/5) standard normal matrix."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    C = torch.randn(nd, n, max(1, n // 5), dtype=torch.float64, device="cuda", generator=g)
    D = torch.bmm(C, C.transpose(1, 2))
    return 0.5 * (D + D.transpose(1, 2)).contiguous()


def _vector(seed, *shape):
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 7919)
    return torch.randn(*shape, dtype=torch.float64, device="cuda", generator=g)


def _cluster(c, seed):
    return W.cluster((c["nx"], c["ny"], c["nz"]), ORB[c["orb"]], AUX[c["aux"]], seed)


def _fit_aux(c, seed):
    """An even-tempered (as fitting sets in use are) 8s6p5d3f2g1h1i set (114 functions) per atom: per l a ladder of
    exponents of ratio 4, jittered by 10 %, each function scaled to a self-repulsion of
    order one; atoms 3.5 bohr apart."""
    rng = np.random.default_rng(seed)
    xyz = W.grid_atoms(rng, (c["nx"], c["ny"], c["nz"]), spacing=3.5, jitter=0.2)
    counts = {0: 8, 1: 6, 2: 5, 3: 3, 4: 2, 5: 1, 6: 1}
    ls, ks, cen, ex, co, at = [], [], [], [], [], []
    for i, R in enumerate(xyz):
        for l, n in counts.items():
            for j in range(n):
                z = 0.8 * 4.0 ** j * rng.uniform(0.9, 1.1)
                ls.append(l); ks.append(1); cen.append(R); at.append(i)
                ex.append([z]); co.append([z ** (0.5 * l + 1.25)])
    return W.make_basis(ls, ks, np.array(cen), np.concatenate(ex), np.concatenate(co), at)


def _molecules(c, seed):
    return [W.molecule(c[k], seed + 100 * i) for i, k in enumerate(("n0", "n1", "n2"))]


def _shape(c):
    f = (lambda l: 2 * l + 1) if c["pure"] else (lambda l: (l + 1) * (l + 2) // 2)
    return (c["npair"], c["naux"], f(c["la"]), f(c["lb"]), 2 * c["lc"] + 1)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "eri3c":
        p = _problem(case, seed)
        plan = lx.Eri3cPlan(p.orb, p.aux, p.pairs, p.auxs, bra_pure=case["pure"])
        return dict(kind=kind, plan=plan, out=torch.empty(plan.shape, dtype=torch.float64, device="cuda"))
    if kind == "host":
        p = _problem(case, seed)
        buf = torch.empty(_shape(case), dtype=torch.float64, pin_memory=True)
        return dict(kind=kind, p=p, pure=case["pure"], out=buf.numpy(), keep=buf)
    if kind in ("dfj", "multi"):
        cl = _cluster(case, seed)
        plan = lx.DFJPlan(cl.orb, cl.aux, 1e-12, contract=bool(case.get("contract", False)))
        nd = case.get("nd", 1)
        D, c = _density(seed, nd, plan.nao), _vector(seed, nd, plan.naux_ao)
        if kind == "multi":
            return dict(kind=kind, plan=plan, D=D, c=c)
        return dict(kind=kind, plan=plan, D=D[0], c=c[0], gamma=torch.empty_like(c[0]), J=torch.empty_like(D[0]))
    if kind == "fit":
        mp = lx.MetricPlan(_fit_aux(case, seed))
        b = _vector(seed, mp.naux_ao) if case["nrhs"] == 1 else _vector(seed, mp.naux_ao, case["nrhs"])
        V = torch.empty((mp.naux_ao, mp.naux_ao), dtype=torch.float64, device="cuda")
        return dict(kind=kind, plan=mp, b=b, V=V)
    if kind == "grad":
        cl = _cluster(case, seed)
        return dict(kind=kind, orb=cl.orb, aux=cl.aux, R=torch.tensor(cl.coords, dtype=torch.float64),
                    D=_density(seed, 1, _nao(cl.orb))[0], c=_vector(seed, _nao(cl.aux)))
    mols = _molecules(case, seed)
    Ds = [_density(seed + i, 1, _nao(m.orb))[0] for i, m in enumerate(mols)]
    cs = [_vector(seed + i, _nao(m.aux)) for i, m in enumerate(mols)]
    return dict(kind=kind, batch=lx.Batch([(m.orb, m.aux) for m in mols], 1e-12).bind(Ds, cs))


def run(s):
    kind = s["kind"]
    if kind == "eri3c":
        return s["plan"].execute(s["out"])
    if kind == "host":
        p = s["p"]
        return lx.eri3c_host(p.orb, p.aux, p.pairs, p.auxs, s["pure"], out=s["out"])
    if kind == "dfj":
        return list(s["plan"].execute(s["D"], s["c"], s["gamma"], s["J"]))
    if kind == "multi":
        return list(s["plan"].execute_multi(s["D"], s["c"]))
    if kind == "fit":
        V = s["plan"].execute(s["V"])
        L, info = lx.cholesky(V)
        return [L, info, lx.cholesky_solve(L, s["b"].clone())]
    if kind == "grad":
        R = s["R"].clone().requires_grad_(True)
        E = lx.DFJEnergy.apply(R, s["orb"], s["aux"], s["D"], s["c"])
        E.backward()
        return [E.detach(), R.grad]
    g, J = s["batch"].execute(mode=2)
    return [list(g), list(J)]


# ------------------------------------------------------------------ least work


def _herm(L):
    return (L + 1) * (L + 2) * (L + 3) // 6


def _table_bytes(b):
    return 12.0 * b.nshell + 24.0 * b.nshell + 16.0 * len(b.exps)


def _build_flops(orb, aux, nd, order):
    """Per primitive triple 40 flops (geometry, Boys function), two per Hermite integral
    of its angular momentum and two per use of one (gamma and J of each density)."""
    po = {}
    for l, k in zip(orb.l.tolist(), orb.k.tolist()):
        po[l, k] = po.get((l, k), 0) + 1
    pa = {}
    for l, k in zip(aux.l.tolist(), aux.k.tolist()):
        pa[l, k] = pa.get((l, k), 0) + 1
    keys, f = sorted(po), 0.0
    for i, x in enumerate(keys):
        for y in keys[:i + 1]:
            n = po[x] * (po[x] + 1) / 2 if x == y else po[x] * po[y]
            for (lc, kc), m in pa.items():
                Lab = x[0] + y[0] + order
                f += n * m * x[1] * y[1] * kc * (40 + 2 * _herm(Lab) + 4.0 * nd * _herm(Lab))
    return f


def work(case):
    kind = case["kind"]
    if kind in ("eri3c", "host"):
        sh = _shape(case)
        n, tri = float(np.prod(sh)), float(sh[0] * sh[1])
        k = case["ka"] * case["kb"] * case["kc"]
        prims = sh[0] * (case["ka"] + case["kb"]) + sh[1] * case["kc"]
        return dict(bytes=8.0 * n + 16.0 * prims + 36.0 * (2 * sh[0] + sh[1]) + 8.0 * sh[0] + 4.0 * sh[1],
                    flops=tri * k * (40 + 2 * _herm(case["la"] + case["lb"] + case["lc"])) + 2.0 * n)
    if kind in ("dfj", "multi", "grad"):
        cl = _cluster(case, 0)
        nd, n, na = case.get("nd", 1), _nao(cl.orb), _nao(cl.aux)
        out = 8.0 * (nd * (n * n + na) if kind != "grad" else 3 * cl.natom + 1)
        return dict(bytes=8.0 * nd * (n * n + na) + out + _table_bytes(cl.orb) + _table_bytes(cl.aux),
                    flops=_build_flops(cl.orb, cl.aux, nd, 1 if kind == "grad" else 0))
    if kind == "fit":
        b = _fit_aux(case, 0)
        n = _nao(b)
        f = sum((40 + 2 * _herm(int(x) + int(y))) for x in b.l[:26] for y in b.l[:26]) * (b.nshell / 26.0) ** 2 / 2
        return dict(bytes=8.0 * n * n + 16.0 * n * case["nrhs"] + _table_bytes(b),
                    flops=f + n ** 3 / 3.0 + 2.0 * n * n * case["nrhs"])
    by = fl = 0.0
    for m in _molecules(case, 0):
        n, na = _nao(m.orb), _nao(m.aux)
        by += 16.0 * (n * n + na) + _table_bytes(m.orb) + _table_bytes(m.aux)
        fl += _build_flops(m.orb, m.aux, 1, 0)
    return dict(bytes=by, flops=fl)


# ------------------------------------------------------------------ 64-bit reference


def _carts(l):
    return [(x, y, l - x - y) for x in range(l, -1, -1) for y in range(l - x, -1, -1)]


def _solid(l):
    """Real solid harmonics, Racah-normalised, m = -l..l, as rows over Cartesian monomials:
    r^(l-m) Legendre part times the real and imaginary parts of (x + i y)^m."""
    idx = {c: i for i, c in enumerate(_carts(l))}
    T = np.zeros((2 * l + 1, len(idx)))
    for m in range(l + 1):
        norm = math.sqrt((2.0 if m else 1.0) * math.factorial(l - m) / math.factorial(l + m))
        for k in range((l - m) // 2 + 1):
            pk = ((-1) ** k * math.comb(l, k) * math.comb(2 * l - 2 * k, l) * math.factorial(l - 2 * k)
                  / (2.0 ** l * math.factorial(l - 2 * k - m)))
            for i in range(k + 1):
                for j in range(k - i + 1):  # r^(2k) = sum k!/(i! j! q!) x^2i y^2j z^2q
                    q = k - i - j
                    mult = math.factorial(k) / (math.factorial(i) * math.factorial(j) * math.factorial(q))
                    for p in range(m + 1):  # (x + i y)^m
                        e = (m - p + 2 * i, p + 2 * j, l - m - 2 * k + 2 * q)
                        v = norm * pk * mult * math.comb(m, p) * (1, 1, -1, -1)[p % 4]
                        if p % 2 == 0:
                            T[l + m, idx[e]] += v
                        else:
                            T[l - m, idx[e]] += v
    return T


def _boys_values(T, M):
    """[F_0 .. F_M](T): series for T < 35, else erf and the upward relation."""
    small = T < 35.0
    t = torch.where(small, T, torch.ones_like(T))
    term = torch.full_like(t, 1.0 / (2 * M + 1))
    s = term.clone()
    for k in range(1, 140):
        term = term * (2.0 * t / (2 * M + 2 * k + 1))
        s = s + term
    e = torch.exp(-t)
    lo = [None] * (M + 1)
    lo[M] = s * e
    for m in range(M, 0, -1):
        lo[m - 1] = (2.0 * t * lo[m] + e) / (2 * m - 1)
    b = torch.where(small, torch.full_like(T, 36.0), T)
    hi = [0.5 * torch.sqrt(math.pi / b) * torch.erf(torch.sqrt(b))]
    eb = torch.exp(-b)
    for m in range(M):
        hi.append(((2 * m + 1) * hi[m] - eb) / (2.0 * b))
    return [torch.where(small, x, y) for x, y in zip(lo, hi)]


class _Boys(torch.autograd.Function):
    """All F_0..F_M stacked; dF_m/dT = -F_(m+1)."""

    @staticmethod
    def forward(ctx, T, M):
        F = torch.stack(_boys_values(T, M + 1))
        ctx.save_for_backward(F)
        return F[:M + 1].clone()

    @staticmethod
    def backward(ctx, g):
        F, = ctx.saved_tensors
        return -(g * F[1:]).sum(0), None


def _hermite(gam, P, zc, C, lc, Lab, every=True):
    """(Lambda_a|C) of unit Hermite Gaussians a, |a| <= Lab (only |a| = Lab when not every), of
    exponents gam at P [n] against solid-harmonic Gaussians zc at C [q]: [na, 2 lc + 1, n, q]."""
    L = Lab + lc
    g, z = gam[:, None], zc[None, :]
    R = [P[:, None, x] - C[None, :, x] for x in range(3)]
    rho = g * z / (g + z)
    pref = 2.0 * math.pi ** 2.5 / (g * z * torch.sqrt(g + z))
    F = _Boys.apply(rho * (R[0] ** 2 + R[1] ** 2 + R[2] ** 2), L)
    cur = {}
    for m in range(L, -1, -1):  # R_e^(m) for |e| <= L - m from R^(m+1)
        new = {(0, 0, 0): pref * (-2.0 * rho) ** m * F[m]}
        for n in range(1, L - m + 1):
            for e in _carts(n):
                i = max(range(3), key=lambda x: e[x])
                d = list(e); d[i] -= 1
                v = R[i] * cur[tuple(d)]
                if d[i]:
                    d2 = list(d); d2[i] -= 1
                    v = v + d[i] * cur[tuple(d2)]
                new[e] = v
        cur = new
    S = torch.tensor(_solid(lc), device=gam.device) * (-1.0) ** lc
    cc = _carts(lc)
    rows = []
    for n in range(0 if every else Lab, Lab + 1):
        for a in _carts(n):
            X = torch.stack([cur[a[0] + c[0], a[1] + c[1], a[2] + c[2]] for c in cc])
            rows.append(torch.tensordot(S, X, 1))
    return torch.stack(rows) / (2.0 * zc) ** lc


def _expansion(la, lb, A, B, za, zb, pure):
    """Hermite expansion of the product of two primitives [n]: E [n, nA*nB, na], gam, P."""
    g = za + zb
    P = (za[:, None] * A + zb[:, None] * B) / g[:, None]
    K = torch.exp(-za * zb / g * ((A - B) ** 2).sum(1))
    ax = []
    zero = torch.zeros_like(g)
    for x in range(3):
        pa, pb = P[:, x] - A[:, x], P[:, x] - B[:, x]
        E = {(0, 0): [torch.ones_like(g)]}
        up = lambda r, p: [(r[t - 1] / (2 * g) if t else zero) + (p * r[t] if t < len(r) else 0)  # noqa: E731
                           + ((t + 1) * r[t + 1] if t + 1 < len(r) else 0) for t in range(len(r) + 1)]
        for i in range(la + 1):
            if i:
                E[i, 0] = up(E[i - 1, 0], pa)
            for j in range(1, lb + 1):
                E[i, j] = up(E[i, j - 1], pb)
        ax.append(E)
    Lab = la + lb
    herm = [a for n in range(Lab + 1) for a in _carts(n)]
    rows = []
    for a in _carts(la):
        for b in _carts(lb):
            r = []
            for t in herm:
                if any(t[x] > a[x] + b[x] for x in range(3)):
                    r.append(zero)
                else:
                    r.append(ax[0][a[0], b[0]][t[0]] * ax[1][a[1], b[1]][t[1]] * ax[2][a[2], b[2]][t[2]] * K)
            rows.append(torch.stack(r, 1))
    E = torch.stack(rows, 1)
    if pure:
        T = torch.tensor(np.kron(_solid(la), _solid(lb)), device=g.device)
        E = torch.einsum("kr,nra->nka", T, E)
    return E, g, P


def _dev(x):
    return torch.as_tensor(np.ascontiguousarray(x), dtype=torch.float64, device="cuda")


def _exact_class(c, seed):
    p = _problem(c, seed)
    la, lb, lc = c["la"], c["lb"], c["lc"]
    ia, ib = p.pairs[:, 0].astype(np.int64), p.pairs[:, 1].astype(np.int64)
    ex, co, xyz = _dev(p.orb.exps), _dev(p.orb.coefs), _dev(p.orb.xyz)
    oa, ob = torch.as_tensor(p.orb.off[ia], device="cuda"), torch.as_tensor(p.orb.off[ib], device="cuda")
    A, B = xyz[torch.as_tensor(ia, device="cuda")], xyz[torch.as_tensor(ib, device="cuda")]
    aex, aco, axyz = _dev(p.aux.exps), _dev(p.aux.coefs), _dev(p.aux.xyz)
    oc = torch.as_tensor(p.aux.off, device="cuda")
    out = torch.zeros(_shape(c), dtype=torch.float64, device="cuda")
    per = 8.0 * c["naux"] * (2 * _herm(la + lb + lc) + 2 * _herm(la + lb) * (2 * lc + 1) + 4 * out[0, 0].numel() + 64)
    step = max(1, min(c["npair"], int(8e9 / per)))
    for p0 in range(0, c["npair"], step):
        s = slice(p0, p0 + step)
        for i in range(c["ka"]):
            for j in range(c["kb"]):
                E, g, P = _expansion(la, lb, A[s], B[s], ex[oa[s] + i], ex[ob[s] + j], c["pure"])
                E = E * (co[oa[s] + i] * co[ob[s] + j])[:, None, None]
                for k in range(c["kc"]):
                    H = _hermite(g, P, aex[oc + k], axyz, lc, la + lb) * aco[oc + k]
                    na, nC, n, q = H.shape
                    X = torch.bmm(E, H.permute(2, 0, 3, 1).reshape(n, na, q * nC))
                    out[s] += X.reshape(n, out.shape[2], out.shape[3], q, nC).permute(0, 3, 1, 2, 4)
    return out


def _shell_groups(b):
    off = np.concatenate([[0], np.cumsum(2 * b.l.astype(np.int64) + 1)])
    got = {}
    for s in range(b.nshell):
        got.setdefault((int(b.l[s]), int(b.k[s])), []).append(s)
    return off, {k: np.array(v) for k, v in got.items()}


def _exact_build(orb, aux, Ds, cs, Ro=None, Ra=None):
    """gamma [nd, naux] and J [nd, n, n] over all triples; with Ro, Ra (shell centres that need
    a gradient) only sum_d c_d gamma_d, back-propagated class by class."""
    nd, n = Ds.shape[0], Ds.shape[1]
    gamma = torch.zeros(nd, cs.shape[1], dtype=torch.float64, device="cuda")
    J = torch.zeros_like(Ds)
    total = 0.0
    ao, og = _shell_groups(orb)
    aq, ag = _shell_groups(aux)
    grad = Ro is not None
    oxyz, axyz = (Ro, Ra) if grad else (_dev(orb.xyz), _dev(aux.xyz))
    t = lambda v: torch.as_tensor(v, device="cuda")  # noqa: E731
    oex, oco, aex, aco = _dev(orb.exps), _dev(orb.coefs), _dev(aux.exps), _dev(aux.coefs)
    keys = sorted(og)
    for xi, (la, ka) in enumerate(keys):
        for lb, kb in keys[:xi + 1]:
            same = (la, ka) == (lb, kb)
            a, b = np.meshgrid(og[la, ka], og[lb, kb], indexing="ij")
            a, b = a.reshape(-1), b.reshape(-1)
            if same:
                keep = a >= b
                a, b = a[keep], b[keep]
            w = np.where(a == b, 1.0, 2.0)
            nA, nB = 2 * la + 1, 2 * lb + 1
            ra, rb = t(ao[a][:, None] + np.arange(nA)), t(ao[b][:, None] + np.arange(nB))
            nk = ka * kb
            pr = np.repeat(np.arange(len(a)), nk)
            pi, pj = np.tile(np.repeat(np.arange(ka), kb), len(a)), np.tile(np.tile(np.arange(kb), ka), len(a))
            big = len(pr)
            for (lc, kc), shells in ag.items():
                cols = t(aq[shells][:, None] + np.arange(2 * lc + 1))
                per = 8.0 * len(shells) * (3 * _herm(la + lb + lc) + 2 * _herm(la + lb) * (2 * lc + 1)) * (12 if grad else 1)
                step = max(1, min(big, int(10e9 / per)))
                for s0 in range(0, big, step):
                    q = pr[s0:s0 + step]
                    u, v = orb.off[a[q]] + pi[s0:s0 + step], orb.off[b[q]] + pj[s0:s0 + step]
                    E, g, P = _expansion(la, lb, oxyz[t(a[q])], oxyz[t(b[q])], oex[t(u)], oex[t(v)], True)
                    E = E * (oco[t(u)] * oco[t(v)] * t(w[q]))[:, None, None]
                    qt = t(q)
                    Dq = Ds[:, ra[qt][:, :, None], rb[qt][:, None, :]].reshape(nd, len(q), nA * nB)
                    Hd = torch.einsum("dnk,nka->dna", Dq, E)
                    for k in range(kc):
                        o = t(aux.off[shells] + k)
                        X = _hermite(g, P, aex[o], axyz[t(shells)], lc, la + lb) * aco[o]
                        gq = torch.einsum("dna,acnq->dqc", Hd, X)
                        if grad:
                            e = (gq * cs[:, cols]).sum()
                            e.backward()
                            total += float(e.detach())
                            if k + 1 < kc:
                                raise ValueError("gradient reference: one primitive per fitting shell")
                            continue
                        gamma[:, cols] += gq
                        y = torch.einsum("acnq,dqc->dna", X, cs[:, cols])
                        blk = torch.einsum("nka,dna->dnk", E, y)
                        for d in range(nd):
                            J[d].index_put_((ra[qt][:, :, None], rb[qt][:, None, :]),
                                            blk[d].reshape(len(q), nA, nB) * 0.5, accumulate=True)
    return total if grad else (gamma, J + J.transpose(1, 2))


def _exact_metric(b):
    off, groups = _shell_groups(b)
    V = torch.zeros(off[-1], off[-1], dtype=torch.float64, device="cuda")
    ex, co, xyz = _dev(b.exps), _dev(b.coefs), _dev(b.xyz)
    t = lambda v: torch.as_tensor(v, device="cuda")  # noqa: E731
    for (lp, _), sp in groups.items():
        S = torch.tensor(_solid(lp), device="cuda")
        rp = t(off[sp][:, None] + np.arange(2 * lp + 1))
        zp = ex[t(b.off[sp])]
        for (lq, _), sq in groups.items():
            rq = t(off[sq][:, None] + np.arange(2 * lq + 1))
            X = _hermite(zp, xyz[t(sp)], ex[t(b.off[sq])], xyz[t(sq)], lq, lp, every=False) * co[t(b.off[sq])]
            X = torch.einsum("ka,acnq->nkqc", S, X) * (co[t(b.off[sp])] / (2.0 * zp) ** lp)[:, None, None, None]
            V[rp[:, :, None, None], rq[None, None, :, :]] = X
    return V


def exact(case, seed):
    kind = case["kind"]
    if kind in ("eri3c", "host"):
        return _exact_class(case, seed)
    if kind in ("dfj", "multi"):
        cl = _cluster(case, seed)
        nd = case.get("nd", 1)
        Ds, cs = _density(seed, nd, _nao(cl.orb)), _vector(seed, nd, _nao(cl.aux))
        g, J = _exact_build(cl.orb, cl.aux, Ds, cs)
        return [g, J] if kind == "multi" else [g[0], J[0]]
    if kind == "fit":
        aux = _fit_aux(case, seed)
        V = _exact_metric(aux)
        L = torch.linalg.cholesky(0.5 * (V + V.T))
        n = V.shape[0]
        b = _vector(seed, n) if case["nrhs"] == 1 else _vector(seed, n, case["nrhs"])
        x = torch.cholesky_solve(b.reshape(n, -1), L).reshape(b.shape)
        return [L + torch.triu(V, 1), 0, x]
    if kind == "grad":
        cl = _cluster(case, seed)
        D, c = _density(seed, 1, _nao(cl.orb)), _vector(seed, _nao(cl.aux))[None]
        with torch.enable_grad():
            R = torch.tensor(cl.coords, dtype=torch.float64, device="cuda", requires_grad=True)
            Ro, Ra = R[_atoms(cl.orb)].detach().requires_grad_(True), R[_atoms(cl.aux)].detach().requires_grad_(True)
            E = _exact_build(cl.orb, cl.aux, D, c, Ro, Ra)
        G = torch.zeros_like(R).detach()
        G.index_add_(0, _atoms(cl.orb), Ro.grad)
        G.index_add_(0, _atoms(cl.aux), Ra.grad)
        return [torch.tensor(E, dtype=torch.float64), G.cpu()]
    gs, Js = [], []
    for i, m in enumerate(_molecules(case, seed)):
        g, J = _exact_build(m.orb, m.aux, _density(seed + i, 1, _nao(m.orb)), _vector(seed + i, _nao(m.aux))[None])
        gs.append(g[0])
        Js.append(J[0])
    return [gs, Js]


def _atoms(b):
    return torch.as_tensor(b.atom.astype(np.int64), device="cuda")
