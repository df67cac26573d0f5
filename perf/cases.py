"""Performance cases of the solver: what a user of the library runs, through its public calls.

A case is a dict of plain values; its ``kind`` names the call:

  entries   blocks of the Nystrom matrix by index lists (``wsbm_entries_raw``)
  proxy     proxy-circle blocks of one box (``wsbm_proxy_block``)
  matvec    matrix-free product A x or A^T x (``wsbm_matvec``)
  vjp       reverse mode of the matrix entries (``entries_vjp``)
  field     field off the curve from the densities (``field``)
  zgemm     complex GEMM of the factorizations (``wsbm_zgemm``)
  lu        dense LU with partial pivoting (``wsbm_lu_dense``)
  solve     solves with a factored curve (``Solver.solve``, ``Solver.farfield``)
  pipeline  curve in, refined densities and far field out (``Solver`` from create to far field)
  gradient  far field and its shape / refractive-index gradient (``autograd``)
  batch     many scatterers factored and solved together (``Batch``)

The curves are closed smooth curves r(t) = 1 + a cos(m t) + a small seeded Fourier part at 15
nodes per exterior wavelength unless stated.  ``exact`` evaluates the same quantities in plain
torch FP64, without the library.
"""
import math

import numpy as np
import torch

from paper_2607_00790_gb300 import autograd, binding

DEV = "cuda"


def listed():
    return [
        # one leaf block of the configured disk / star problems: the latency of a small request
        dict(name="entries_leaf", kind="entries", N=1024, nr=256, nc=256, spread=False, npw=15.0),
        # rows of a large system against scattered columns (sampling residuals, external compressors)
        dict(name="entries_rows", kind="entries", N=262144, nr=1999, nc=8192, spread=True, npw=15.0),
        # the proxy rows of a box a few levels above the leaves, as an external ID asks for them
        dict(name="proxy_rows", kind="proxy", N=65536, nidx=1500, P=712, side=0, precision=0, npw=15.0),
        # residual of the 16384-node star workload: one dense matrix-free product
        dict(name="matvec", kind="matvec", N=16384, nrhs=1, trans=False, npw=15.0),
        # the backward pair kernel of a gradient step
        dict(name="vjp", kind="vjp", N=6000, npw=15.0),
        # near-field picture: points inside and outside for the 8 incident angles of the star workload
        dict(name="field", kind="field", N=16384, nt=3001, nrhs=8, npw=15.0),
        # trailing update of a blocked factorization with 256-column panels
        dict(name="zgemm_update", kind="zgemm", m=5000, n=4000, k=256),
        # dense root system of the size the star workload leaves
        dict(name="lu_root", kind="lu", n=8200),
        # many incident angles on a curve that is factored once
        dict(name="solve_many", kind="solve", N=16384, nrhs=64, nang=360, tol=1e-10, npw=15.0),
        # the star workload end to end: create, factor, 8 plane waves, one refinement step, far field
        dict(name="star_pipeline", kind="pipeline", N=16384, nrhs=8, nang=360, leaf=128, nproxy=128,
             tol=1e-8, npw=15.0),
        # one step of a shape reconstruction: far field at 64 angles and its gradient
        dict(name="gradient_step", kind="gradient", N=4096, nang=64, leaf=64, nproxy=64, tol=1e-8, npw=15.0),
        # scatterers of uneven size in one batch, 16 plane waves each
        dict(name="batch", kind="batch", count=8, nmin=2048, nmax=6144, nrhs=16, tol=1e-10, npw=15.0),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["entries", "entries", "proxy", "matvec", "vjp", "field", "zgemm", "zgemm", "lu", "solve",
                       "pipeline", "gradient", "batch"])
    npw = math.exp(rng.uniform(math.log(12.0), math.log(120.0)))
    if kind == "entries":
        return dict(kind=kind, N=_logint(rng, 512, 262144), nr=_logint(rng, 17, 4096), nc=_logint(rng, 17, 4096),
                    spread=rng.random() < 0.5, npw=npw)
    if kind == "proxy":
        return dict(kind=kind, N=_logint(rng, 2048, 262144), nidx=_logint(rng, 64, 2048), P=8 * _logint(rng, 8, 128),
                    side=rng.randrange(2), precision=rng.choice([0, 0, 1, 2]), npw=npw)
    if kind == "matvec":
        return dict(kind=kind, N=_logint(rng, 300, 12000), nrhs=rng.randint(1, 4), trans=rng.random() < 0.5, npw=npw)
    if kind == "vjp":
        return dict(kind=kind, N=_logint(rng, 300, 10000), npw=npw)
    if kind == "field":
        return dict(kind=kind, N=_logint(rng, 500, 16384), nt=_logint(rng, 100, 4000), nrhs=rng.randint(1, 8), npw=npw)
    if kind == "zgemm":
        return dict(kind=kind, m=_logint(rng, 60, 6000), n=_logint(rng, 16, 6000), k=_logint(rng, 33, 1000))
    if kind == "lu":
        return dict(kind=kind, n=_logint(rng, 300, 8000))
    if kind == "solve":
        return dict(kind=kind, N=_logint(rng, 1024, 8192), nrhs=_logint(rng, 1, 128), nang=rng.randint(30, 360),
                    tol=1e-10, npw=npw)
    if kind == "pipeline":
        leaf = rng.choice([64, 128])
        return dict(kind=kind, N=_logint(rng, 1024, 12000), nrhs=rng.randint(1, 8), nang=rng.randint(30, 360),
                    leaf=leaf, nproxy=leaf, tol=rng.choice([1e-6, 1e-8, 1e-10]), npw=npw)
    if kind == "gradient":
        return dict(kind=kind, N=_logint(rng, 512, 6000), nang=rng.randint(8, 64), leaf=64, nproxy=64, tol=1e-8, npw=npw)
    nmin = _logint(rng, 512, 3000)
    return dict(kind="batch", count=rng.randint(2, 8), nmin=nmin, nmax=nmin + rng.randint(1, 4000),
                nrhs=rng.randint(1, 16), tol=1e-10, npw=npw)


# ------------------------------------------------------------------------------ inputs ----
NAMES = ("x", "y", "nx", "ny", "w", "kappa")
REFR = 1.5


def _polar(N, acoef, bcoef):
    """Nodes of r(t) = 1 + sum_j a_j cos jt + b_j sin jt at N equispaced t (rows: NAMES)."""
    t = 2.0 * np.pi * np.arange(N) / N
    r, r1, r2 = np.ones(N), np.zeros(N), np.zeros(N)
    for j, (a, b) in enumerate(zip(acoef, bcoef), start=1):
        c, s = np.cos(j * t), np.sin(j * t)
        r += a * c + b * s
        r1 += j * (b * c - a * s)
        r2 -= j * j * (a * c + b * s)
    c, s = np.cos(t), np.sin(t)
    xp, yp = r1 * c - r * s, r1 * s + r * c
    xpp, ypp = r2 * c - 2 * r1 * s - r * c, r2 * s + 2 * r1 * c - r * s
    sp = np.sqrt(xp * xp + yp * yp)
    return np.stack([r * c, r * s, yp / sp, -xp / sp, 2 * np.pi / N * sp, (xp * ypp - yp * xpp) / sp**3])


def _shape(rng, star=True):
    a, b = rng.normal(0.0, 0.004, 16), rng.normal(0.0, 0.004, 16)
    if star:
        a[int(rng.integers(3, 8)) - 1] += rng.uniform(0.1, 0.3)
    return a, b


def _curve(case, rng, N=None):
    """Node arrays (6 x N, numpy) and k0 of the case's curve."""
    c = _polar(N or case["N"], *_shape(rng))
    return c, _k0(c, case["npw"])


def _k0(c, npw):
    return float(2.0 * np.pi * c.shape[1] / (npw * c[4].sum()))


def _geom(c):
    return binding.make_geom(dict(zip(NAMES, c)), DEV)


def _randc(seed, *shape):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return torch.randn(*shape, dtype=torch.complex128, device=DEV, generator=g)


def _angles(n, off=0.0):
    return torch.arange(n, dtype=torch.float64, device=DEV) * (2.0 * math.pi / n) + off


def _index_lists(case, rng):
    N = case["N"]
    if case["spread"]:  # scattered unknowns of both kinds
        nr, nc = min(case["nr"], 2 * N), min(case["nc"], 2 * N)
        rows, cols = (np.sort(rng.choice(2 * N, k, replace=False)) for k in (nr, nc))
        return rows, cols
    out = []  # the unknowns (u then q) of two runs of neighbouring nodes
    start = int(rng.integers(0, N))
    for k in (case["nr"], case["nc"]):
        nodes = (start + np.arange(min((k + 1) // 2, N))) % N
        out.append(np.concatenate([nodes, N + nodes])[: min(k, 2 * N)])
    return out


def _lu_matrix(case, seed):
    """A second-kind system: 1/2 on the diagonal plus a dense part of comparable norm."""
    n = case["n"]
    A = _randc(seed, n, n) * (0.25 / math.sqrt(n))
    A.diagonal().add_(0.5)
    return A


def _proxy_box(case, rng):
    """Curve, k0, unknowns of one box of neighbouring nodes and its proxy circle."""
    c, k0 = _curve(case, rng)
    N = case["N"]
    nodes = (int(rng.integers(0, N)) + np.arange(min((case["nidx"] + 1) // 2, N // 8))) % N
    bx, by = c[0][nodes], c[1][nodes]
    cx, cy = 0.5 * (bx.min() + bx.max()), 0.5 * (by.min() + by.max())
    rho = 1.5 * float(np.sqrt((bx - cx) ** 2 + (by - cy) ** 2).max())
    return c, k0, np.concatenate([nodes, N + nodes]), (float(cx), float(cy), rho)


def _targets(case, c, rng):
    """Points at 0.5 .. 0.9 and 1.1 .. 2.5 of the curve's radius over random nodes' rays."""
    j = rng.integers(0, c.shape[1], case["nt"])
    f = np.where(rng.random(case["nt"]) < 0.4, rng.uniform(0.3, 0.9, case["nt"]), rng.uniform(1.1, 2.5, case["nt"]))
    return f * c[0][j], f * c[1][j]


def _batch_curves(case, rng):
    out = []
    for i in range(case["count"]):  # sizes spread over [nmin, nmax], the same for every seed
        N = case["nmin"] + int((case["nmax"] - case["nmin"]) * (0.618034 * (i + 1) % 1.0))
        c = _polar(N, *_shape(rng, star=rng.random() < 0.5))
        out.append((c, _k0(c, case["npw"]), float(rng.uniform(1.2, 2.0))))
    return out


def _t(v):
    return torch.as_tensor(v).to(DEV)


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    s = dict(case=case, kind=kind)
    if kind == "zgemm":
        m, n, k = case["m"], case["n"], case["k"]
        s.update(A=_randc(seed, m, k), B=_randc(seed + 1, k, n), C=_randc(seed + 2, m, n) * math.sqrt(k))
        return s
    if kind == "lu":
        s["A"] = _lu_matrix(case, seed)
        return s
    if kind == "batch":
        curves = _batch_curves(case, rng)
        s["geoms"] = [_geom(c) for c, _, _ in curves]
        s["params"] = [binding.make_params(k0, n, leaf=64, nproxy=64, id_tol=case["tol"]) for _, k0, n in curves]
        s["ang"] = _angles(case["nrhs"], 0.1)
        return s
    if kind == "gradient":
        a, b = _shape(rng)
        s.update(a=_t(a).requires_grad_(), b=_t(b).requires_grad_(),
                 n=torch.tensor(REFR, dtype=torch.float64, device=DEV, requires_grad=True),
                 k0=_k0(_polar(case["N"], a, b), case["npw"]), inc=_angles(1), obs=_angles(case["nang"]))
        s["target"] = 1.0 + _t(rng.random(case["nang"]))
        return s
    if kind == "proxy":
        c, k0, idx, s["circle"] = _proxy_box(case, rng)
        s["idx"] = _t(idx)
    else:
        c, k0 = _curve(case, rng)
    s["geom"], s["keep"] = _geom(c)
    s["params"] = binding.make_params(k0, REFR, leaf=case.get("leaf", 64), nproxy=case.get("nproxy", 64),
                                      id_tol=case.get("tol", 1e-8), precision=case.get("precision", 0))
    N = case["N"]
    if kind == "entries":
        s["rows"], s["cols"] = map(_t, _index_lists(case, rng))
    elif kind == "matvec":
        s["x"] = _randc(seed, case["nrhs"], 2 * N).T
    elif kind == "vjp":
        s["lam"], s["x"] = _randc(seed, 2 * N), _randc(seed + 1, 2 * N)
    elif kind == "field":
        tx, ty = _targets(case, c, rng)
        s.update(tx=_t(tx), ty=_t(ty), u=_randc(seed, case["nrhs"], N).T, q=_randc(seed + 1, case["nrhs"], N).T * k0)
    elif kind in ("solve", "pipeline"):
        s["inc"], s["obs"] = _angles(case["nrhs"], 0.2), _angles(case["nang"])
        if kind == "solve":
            s["solver"] = binding.Solver(s["geom"], s["params"], DEV)
            s["solver"].factor()
            s["rhs"] = s["solver"].rhs_planewave(s["inc"])
    return s


# --------------------------------------------------------------------------------- run ----
def run(s):
    kind = s["kind"]
    if kind == "entries":
        return binding.wsbm_entries_raw(s["geom"], s["params"], s["rows"], s["cols"])
    if kind == "proxy":
        return binding.wsbm_proxy_block(s["geom"], s["params"], s["case"]["side"], s["idx"], s["circle"], s["case"]["P"])
    if kind == "matvec":
        return binding.wsbm_matvec(s["geom"], s["params"], s["x"], trans=s["case"]["trans"])
    if kind == "vjp":
        return binding.entries_vjp(s["geom"], s["params"], s["lam"], s["x"])
    if kind == "field":
        return binding.field(s["geom"], s["params"], s["u"], s["q"], s["tx"], s["ty"])
    if kind == "zgemm":
        return binding.wsbm_zgemm(s["A"], s["B"], s["C"], alpha=-1.0, beta=1.0)
    if kind == "lu":
        return binding.wsbm_lu_dense(s["A"])
    if kind == "solve":
        u, q = s["solver"].solve(s["rhs"])
        return u, q, s["solver"].farfield(u, q, s["obs"])
    if kind == "pipeline":
        h = binding.Solver(s["geom"], s["params"], DEV)
        h.factor()
        rhs = h.rhs_planewave(s["inc"])
        u, q = h.solve(rhs)
        u, q, _ = h.refine(s["geom"], s["params"], rhs, u, q, iters=1)
        F = h.farfield(u, q, s["obs"])
        h.close()
        return u, q, F
    if kind == "gradient":
        case = s["case"]
        F = autograd.farfield(autograd.fourier_curve(s["a"], s["b"], case["N"]), s["n"], s["k0"], s["inc"], s["obs"],
                              leaf=case["leaf"], nproxy=case["nproxy"], tol=case["tol"], refine=2)
        loss = torch.sum((F[:, 0].abs() ** 2 - s["target"]) ** 2)
        return (F.detach(),) + torch.autograd.grad(loss, (s["a"], s["b"], s["n"]))
    b = binding.Batch([g for g, _ in s["geoms"]], s["params"], DEV)
    b.factor()
    handles = [b.solver(i) for i in range(len(s["geoms"]))]
    out = b.solve([h.rhs_planewave(s["ang"]) for h in handles])
    b.close()
    return [v for uq in out for v in uq]


def work(case):
    """Bytes and flops a pass cannot do without: an entry of the matrix is counted with the
    fewest operations that two Hankel evaluations and the block algebra take (about 300 per
    node pair for a 2x2 block), the dense algebra with its complex operation counts."""
    kind = case["kind"]
    if kind == "entries":
        n = min(case["nr"], 2 * case["N"]) * min(case["nc"], 2 * case["N"])
        return dict(bytes=16 * n, flops=75 * n)
    if kind == "proxy":
        n = 2 * case["P"] * 2 * min((case["nidx"] + 1) // 2, case["N"] // 8)
        return dict(bytes=16 * n, flops=75 * n)
    if kind == "zgemm":
        m, n, k = case["m"], case["n"], case["k"]
        return dict(bytes=16 * (m * k + k * n + 2 * m * n), flops=8 * m * n * k)
    if kind == "lu":
        return dict(bytes=32 * case["n"] ** 2, flops=8 * case["n"] ** 3 // 3)
    if kind == "batch":
        N = case["count"] * (case["nmin"] + case["nmax"]) // 2
        return dict(bytes=48 * N + 32 * N * case["nrhs"], flops=N * 128 * 300)
    N = case["N"]
    if kind == "matvec":
        return dict(bytes=48 * N + 64 * N * case["nrhs"], flops=N * N * (300 + 32 * case["nrhs"]))
    if kind == "vjp":
        return dict(bytes=48 * N * 2 + 64 * N, flops=N * N * 600)
    if kind == "field":
        return dict(bytes=48 * N + 32 * N * case["nrhs"] + 16 * case["nt"] * (1 + case["nrhs"]),
                    flops=N * case["nt"] * (150 + 16 * case["nrhs"]))
    if kind == "solve":
        return dict(bytes=64 * N * case["nrhs"] + 16 * case["nang"] * case["nrhs"],
                    flops=N * case["nrhs"] * (1024 + 20 * case["nang"]))
    if kind == "pipeline":  # two residuals of one refinement step and the near entries
        return dict(bytes=48 * N + 64 * N * case["nrhs"], flops=2 * N * N * (300 + 32 * case["nrhs"]))
    return dict(bytes=48 * N, flops=N * N * (6 * 332 + 600))  # gradient


# ------------------------------------------------------------------------------- exact ----
def _bessel_small(z, top=70):
    """J0, J1, Y0, Y1 for z < 25: Miller's downward recurrence normalized by J0 + 2 sum J_2k = 1,
    and Neumann's series of Y0 (and its derivative) in the J_n."""
    jp, j = torch.zeros_like(z), torch.full_like(z, 1e-290)  # J_{n+1}, J_n up to a factor
    norm, s0, s1 = torch.zeros_like(z), torch.zeros_like(z), torch.zeros_like(z)
    for n in range(top, 0, -1):
        jm = 2 * n / z * j - jp
        if n % 2 == 0:
            k, sg = n // 2, (-1 if n % 4 else 1)
            norm += 2 * j
            s0 += sg / k * j
            s1 += sg / (2 * k) * (jm - jp)
        jp, j = j, jm
    norm += j
    j0, j1, s0, s1 = j / norm, jp / norm, s0 / norm, s1 / norm
    L = torch.log(0.5 * z) + 0.57721566490153286061
    return j0, j1, 2 / math.pi * (L * j0 - 2 * s0), 2 / math.pi * (L * j1 - j0 / z + 2 * s1)


def _hankel_values(z):
    """H0, H1 (complex128) at z > 0: Bessel functions below 25, beyond it Hankel's expansion
    with the argument reduced by three parts of 2 pi whose products with the count are exact."""
    small = z < 25.0
    j0, j1, y0, y1 = _bessel_small(torch.where(small, z, torch.ones_like(z)))
    zl = torch.where(small, torch.full_like(z, 50.0), z)
    p1 = math.ldexp(math.floor(math.ldexp(2 * math.pi, 28)), -28)
    p2 = math.ldexp(math.floor(math.ldexp(2 * math.pi - p1, 56)), -56)
    p3 = 2 * math.pi - p1 - p2 + 2.4492935982947064e-16  # 2 pi in double + its residual
    cnt = torch.round(zl / (2 * math.pi))
    y = ((zl - cnt * p1) - cnt * p2) - cnt * p3
    cs, sn = torch.cos(y), torch.sin(y)
    rt = math.sqrt(0.5)
    amp = torch.sqrt(2.0 / (math.pi * zl))
    h = []
    for nu, near in ((0, torch.complex(j0, y0)), (1, torch.complex(j1, y1))):
        P, Q, term = torch.ones_like(zl), torch.zeros_like(zl), torch.ones_like(zl)
        for k in range(1, 24):
            term = term * (4.0 * nu * nu - (2 * k - 1) ** 2) / (k * 8.0 * zl)
            if k % 2:
                Q = Q + term * (1 if k % 4 == 1 else -1)
            else:
                P = P + term * (1 if k % 4 == 0 else -1)
        E, F = (cs + sn) * rt, (sn - cs) * rt  # e^{i(z - pi/4)}
        if nu == 1:
            E, F = F, -E
        h.append(torch.where(small, near, torch.complex(amp * (P * E - Q * F), amp * (P * F + Q * E))))
    return h


class _Hankel(torch.autograd.Function):
    @staticmethod
    def forward(ctx, z):
        h0, h1 = _hankel_values(z)
        ctx.save_for_backward(z, h0, h1)
        return h0, h1

    @staticmethod
    def backward(ctx, g0, g1):
        z, h0, h1 = ctx.saved_tensors
        return torch.real(g0.conj() * -h1 + g1.conj() * (h0 - h1 / z))


def _blocks(T, S, same, k0, k1, eps0, eps1):
    """The four entries of the 2x2 blocks of target nodes T (rows) and source nodes S (columns),
    6 x n tensors; `same`: where both are one node (the one-point corrected diagonal)."""
    xi, yi, nxi, nyi, wi, kap = (v[:, None] for v in T)
    xj, yj, nxj, nyj, wj, _ = (v[None, :] for v in S)
    dx, dy = xi - xj, yi - yj
    r = torch.sqrt(torch.where(same, torch.ones_like(dx), dx * dx + dy * dy))
    dnx, dny, nn = (dx * nxi + dy * nyi) / r, (dx * nxj + dy * nyj) / r, nxi * nxj + nyi * nyj
    z0, z1 = k0 * r, k1 * r
    a0, a1 = _Hankel.apply(z0)
    b0, b1 = _Hankel.apply(z1)
    af, bf = (h / z + 2j / (math.pi * z * z) for h, z in ((a1, z0), (b1, z1)))
    c = dnx * dny
    dN = 0.25j * ((k0 * k0 * a0 - k1 * k1 * b0) * c + (k0 * k0 * af - k1 * k1 * bf) * (nn - 2 * c))
    al = 1j / k0
    A11 = wj * 0.25j * k1 * b1 * dny
    A12 = -eps1 * wj * 0.25j * b0
    A21 = wj * (0.25j * k0 * a1 * dny + al * dN)
    A22 = wj * (-eps0 * 0.25j * a0 - al * (-0.25j) * (eps0 * k0 * a1 - eps1 * k1 * b1) * dnx)
    if bool(same.any()):
        w, g = wi, 0.57721566490153286061
        L0, L1 = torch.log(k0 * w / (4 * math.pi)), torch.log(k1 * w / (4 * math.pi))
        S0, S1 = (w * (0.25j - (g + L) / (2 * math.pi)) for L in (L0, L1))
        Dd = -w * kap / (4 * math.pi)
        f0, f1 = k0 * k0 * (L0 + g - 0.5), k1 * k1 * (L1 + g - 0.5)
        dNd = w * ((k0 * k0 - k1 * k1) * 0.125j - (f0 - f1) / (4 * math.pi))
        A11 = torch.where(same, Dd + 0.5 + 0j, A11)
        A12 = torch.where(same, -eps1 * S1, A12)
        A21 = torch.where(same, Dd - 0.5 + al * dNd, A21)
        A22 = torch.where(same, -eps0 * S0 - al * ((eps0 - eps1) * Dd + 0.5 * (eps0 + eps1)), A22)
    return A11, A12, A21, A22


def _phys(k0, n=REFR):
    return k0, n * k0, 1.0, n * n


def _chunks(N, cols):
    step = max(1, (8 << 20) // cols)
    return [(i, min(N, i + step)) for i in range(0, N, step)]


def _eye(i0, i1, N):
    return torch.arange(i0, i1, device=DEV)[:, None] == torch.arange(N, device=DEV)[None, :]


def _dense(g, ph):
    N = g.shape[1]
    A = torch.empty(2 * N, 2 * N, dtype=torch.complex128, device=DEV)
    for i0, i1 in _chunks(N, N):
        b = _blocks(g[:, i0:i1], g, _eye(i0, i1, N), *ph)
        A[i0:i1, :N], A[i0:i1, N:], A[N + i0:N + i1, :N], A[N + i0:N + i1, N:] = b
    return A


def _planewave(g, k0, ang):
    d = torch.stack([torch.cos(ang), torch.sin(ang)])
    u = torch.exp(1j * k0 * (g[0][:, None] * d[0] + g[1][:, None] * d[1]))
    dn = 1j * k0 * (g[2][:, None] * d[0] + g[3][:, None] * d[1]) * u
    return torch.cat([torch.zeros_like(u), -u - 1j / k0 * dn])


def _far(g, k0, u, q, ang, eps0=1.0):
    d = torch.stack([torch.cos(ang), torch.sin(ang)])
    ph = torch.exp(-1j * k0 * (d[0][:, None] * g[0] + d[1][:, None] * g[1]))
    dn = d[0][:, None] * g[2] + d[1][:, None] * g[3]
    c = complex(math.cos(math.pi / 4), math.sin(math.pi / 4)) / math.sqrt(8 * math.pi * k0)
    return c * ((-1j * k0 * dn * g[4] * ph) @ u - eps0 * (g[4] * ph) @ q)


def _bilinear(g, k1, eps1, k0, lam, x):
    """Re(lam^T A x) in row chunks, each as a function of (g, k1, eps1) for autograd."""
    N = g.shape[1]
    for i0, i1 in _chunks(N, 4 * N):
        A11, A12, A21, A22 = _blocks(g[:, i0:i1], g, _eye(i0, i1, N), k0, k1, 1.0, eps1)
        yield torch.real(lam[i0:i1] @ (A11 @ x[:N] + A12 @ x[N:]) + lam[N + i0:N + i1] @ (A21 @ x[:N] + A22 @ x[N:]))


def _leaf_vars(g, k1, eps1):
    one = lambda v: torch.tensor(v, dtype=torch.float64, device=DEV, requires_grad=True)  # noqa: E731
    return g.detach().clone().requires_grad_(), one(k1), one(eps1)


def _vjp(g, k0, lam, x, n=REFR):
    v = _leaf_vars(g, n * k0, n * n)
    tot = [torch.zeros_like(t) for t in v]
    for part in _bilinear(*v, k0, lam, x):
        for t, d in zip(tot, torch.autograd.grad(part, v)):
            t += d
    return tot[0], torch.stack(tot[1:])


def _torch_curve(a, b, N):
    t = torch.arange(N, dtype=torch.float64, device=DEV) * (2 * math.pi / N)
    j = torch.arange(1, a.numel() + 1, dtype=torch.float64, device=DEV)
    C, S = torch.cos(t[:, None] * j), torch.sin(t[:, None] * j)
    r, r1, r2 = 1 + C @ a + S @ b, C @ (j * b) - S @ (j * a), -(C @ (j * j * a)) - S @ (j * j * b)
    c, s = torch.cos(t), torch.sin(t)
    xp, yp = r1 * c - r * s, r1 * s + r * c
    xpp, ypp = r2 * c - 2 * r1 * s - r * c, r2 * s + 2 * r1 * c - r * s
    sp = torch.sqrt(xp * xp + yp * yp)
    return torch.stack([r * c, r * s, yp / sp, -xp / sp, 2 * math.pi / N * sp, (xp * ypp - yp * xpp) / sp**3])


def _exact_gradient(case, rng):
    a, b = _shape(rng)
    N, nang = case["N"], case["nang"]
    target = 1.0 + _t(rng.random(nang))
    k0 = _k0(_polar(N, a, b), case["npw"])
    a, b = _t(a).requires_grad_(), _t(b).requires_grad_()
    g = _torch_curve(a, b, N)
    gd = g.detach()
    inc, obs = _angles(1), _angles(nang)
    LU, piv = torch.linalg.lu_factor(_dense(gd, _phys(k0)))
    x = torch.linalg.lu_solve(LU, piv, _planewave(gd, k0, inc))
    xv = x.clone().requires_grad_()
    gv = gd.clone().requires_grad_()
    F = _far(gv, k0, xv[:N], xv[N:], obs)
    loss = torch.sum((F[:, 0].abs() ** 2 - target) ** 2)
    g_ff, g_x = torch.autograd.grad(loss, (gv, xv))
    lam = torch.linalg.lu_solve(LU, piv, g_x, adjoint=True).conj()  # A^T lam = conj(g_x)
    del LU
    gv2 = gd.clone().requires_grad_()
    (g_b,) = torch.autograd.grad(torch.real(torch.sum(lam * _planewave(gv2, k0, inc))), gv2)
    g_a, g_p = _vjp(gd, k0, lam[:, 0], x[:, 0])
    ga, gb = torch.autograd.grad(g, (a, b), g_ff + g_b - g_a)
    return F.detach(), ga, gb, -(g_p[0] * k0 + 2 * REFR * g_p[1])


def _exact_proxy(case, rng):
    c, k0, idx, (cx, cy, rho) = _proxy_box(case, rng)
    N, P = case["N"], case["P"]
    g, idx = _t(c), _t(idx)
    node, second = idx % N, (idx >= N)[:, None]
    X = g[:, node]
    th = torch.arange(P, dtype=torch.float64, device=DEV) * (2 * math.pi / P)
    pn = torch.stack([torch.cos(th), torch.sin(th)])
    dx, dy = X[0][:, None] - (cx + rho * pn[0]), X[1][:, None] - (cy + rho * pn[1])
    r = torch.sqrt(dx * dx + dy * dy)
    dnx = (dx * X[2][:, None] + dy * X[3][:, None]) / r
    parts = []
    for k, eps in ((REFR * k0, REFR * REFR), (k0, 1.0)):
        h0, h1 = _hankel_values(k * r)
        if case["side"] == 1:
            # the field of the box unknowns at p: d = p - x, so d.n_x / r = -dnx
            parts.append(torch.where(second, -0.25j * eps * X[4][:, None] * h0, -0.25j * k * X[4][:, None] * h1 * dnx))
            continue
        dnu = (dx * pn[0] + dy * pn[1]) / r
        nn, cc = X[2][:, None] * pn[0] + X[3][:, None] * pn[1], dnx * dnu
        phi = 0.25j * k * h1 * dnu + 0.25 * k * h0
        dphi = 0.25j * k * k * (h0 * cc + h1 / (k * r) * (nn - 2 * cc)) - 0.25 * k * k * h1 * dnx
        first = phi if not parts else torch.zeros_like(phi)
        parts.append(2 * math.pi * rho / P * torch.where(second, (phi if parts else 0) + (1 if parts else -1) * 1j / k0 * dphi, first))
    if case["side"] == 1:
        return torch.cat(parts, dim=1).T
    return torch.cat(parts, dim=1)


def _exact_lu(A):
    """Right-looking LU, 32 columns at a time; the pivot has the largest max(|Re|, |Im|)."""
    n = A.shape[0]
    piv = torch.empty(n, dtype=torch.int64)
    for j0 in range(0, n, 32):
        j1 = min(n, j0 + 32)
        for j in range(j0, j1):
            p = j + int(torch.maximum(A[j:, j].real.abs(), A[j:, j].imag.abs()).argmax())
            piv[j] = p
            if p != j:
                A[[j, p]] = A[[p, j]]
            A[j + 1:, j] /= A[j, j].clone()
            A[j + 1:, j + 1:j1] -= A[j + 1:, j, None] * A[None, j, j + 1:j1]
        if j1 < n:
            A[j0:j1, j1:] = torch.linalg.solve_triangular(A[j0:j1, j0:j1], A[j0:j1, j1:], upper=False, unitriangular=True)
            A[j1:, j1:] -= A[j1:, j0:j1] @ A[j0:j1, j1:]
    return A, piv.to(torch.int32)


def exact(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "zgemm":
        m, n, k = case["m"], case["n"], case["k"]
        return _randc(seed + 2, m, n) * math.sqrt(k) - _randc(seed, m, k) @ _randc(seed + 1, k, n)
    if kind == "lu":
        return _exact_lu(_lu_matrix(case, seed))
    if kind == "batch":
        if case["nmax"] > 2500:
            return None
        out = []
        for c, k0, n in _batch_curves(case, rng):
            g = _t(c)
            x = torch.linalg.solve(_dense(g, _phys(k0, n)), _planewave(g, k0, _angles(case["nrhs"], 0.1)))
            out += [x[: g.shape[1]], x[g.shape[1]:]]
        return out
    if kind == "gradient":
        return _exact_gradient(case, rng) if case["N"] <= 4096 else None
    if kind == "proxy":
        return _exact_proxy(case, rng) if case["precision"] == 0 else None
    c, k0 = _curve(case, rng)
    g, N = _t(c), case["N"]
    if kind == "entries":
        rows, cols = map(_t, _index_lists(case, rng))
        out = torch.empty(rows.numel(), cols.numel(), dtype=torch.complex128, device=DEV)
        for i0, i1 in _chunks(rows.numel(), cols.numel()):
            tn, sn = rows[i0:i1] % N, cols % N
            b = _blocks(g[:, tn], g[:, sn], tn[:, None] == sn[None, :], *_phys(k0))
            r2, c2 = (rows[i0:i1] >= N)[:, None], (cols >= N)[None, :]
            out[i0:i1] = torch.where(r2, torch.where(c2, b[3], b[2]), torch.where(c2, b[1], b[0]))
        return out
    if kind == "matvec":
        x = _randc(seed, case["nrhs"], 2 * N).T
        y = torch.zeros_like(x)
        for i0, i1 in _chunks(N, N):
            b = _blocks(g[:, i0:i1], g, _eye(i0, i1, N), *_phys(k0))
            if case["trans"]:
                y[:N] += b[0].T @ x[i0:i1] + b[2].T @ x[N + i0:N + i1]
                y[N:] += b[1].T @ x[i0:i1] + b[3].T @ x[N + i0:N + i1]
            else:
                y[i0:i1] = b[0] @ x[:N] + b[1] @ x[N:]
                y[N + i0:N + i1] = b[2] @ x[:N] + b[3] @ x[N:]
        return y
    if kind == "vjp":
        return _vjp(g, k0, _randc(seed, 2 * N), _randc(seed + 1, 2 * N))
    if kind == "field":
        tx, ty = map(_t, _targets(case, c, rng))
        u, q = _randc(seed, case["nrhs"], N).T, _randc(seed + 1, case["nrhs"], N).T * k0
        out, ins = torch.empty(case["nt"], case["nrhs"], dtype=torch.complex128, device=DEV), torch.empty(case["nt"], dtype=torch.bool, device=DEV)
        for i0, i1 in _chunks(case["nt"], N):
            dx, dy = tx[i0:i1, None] - g[0], ty[i0:i1, None] - g[1]
            r = torch.sqrt(dx * dx + dy * dy)
            dn = (dx * g[2] + dy * g[3]) / r
            inside = ((dn / r) @ g[4]) / (-2 * math.pi) > 0.5
            k = (k0 + inside.double() * (REFR - 1) * k0)[:, None]
            h0, h1 = _hankel_values(k * r)
            D, S = 0.25j * k * h1 * dn * g[4], 0.25j * h0 * g[4]
            eps = (1.0 + inside.double() * (REFR * REFR - 1))[:, None]
            v = D @ u - eps * (S @ q)
            out[i0:i1], ins[i0:i1] = torch.where(inside[:, None], -v, v), inside
        return out, ins
    if N > 4096:  # solve, pipeline: a dense solve
        return None
    inc, obs = _angles(case["nrhs"], 0.2), _angles(case["nang"])
    x = torch.linalg.solve(_dense(g, _phys(k0)), _planewave(g, k0, inc))
    return x[:N], x[N:], _far(g, k0, x[:N], x[N:], obs)
