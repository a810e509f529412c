"""What this library is timed on: its public entry points, over the sizes that its users bring.

Every case is one call (or the few calls that belong together) of a program
that keeps a `Surface` handle: the mat-vec A u in each arithmetic and
direction for callers with a Krylov loop of their own, the charge passes, and
whole solves with what is read from them.  Surfaces are smooth, randomly
displaced spheres of any number of elements (about four elements per square
Angstrom, as the Kirkwood and protein-like surfaces of the benchmark have),
charges lie in their inner 80 %, and the medium is water at 0.15 M unless a
case says otherwise.

The single-precision operators (FP32, TENSOR, TREE32) hand their result over
in FP64 tensors; the caller of a single-precision operator goes on in single
precision, so `run` returns those as float32.
"""
import math

import numpy as np
import torch

import paper_2312_10044_gb300 as bipb
from paper_2312_10044_gb300.torch_ops import BipbEnergy

EPS_IN, EPS_OUT, KAPPA = 1.0, 80.0, 0.1257
KCAL = 4.0 * math.pi * 332.0716
SINGLE = ("FP32", "TENSOR", "TREE32")


def listed():
    return [
        # A Born-size ion or a side chain: 1280 elements.  Launches and latency decide.
        dict(name="solve_small", kind="solve", n=1280, nc=12, precision="MIXED_DF64", precond=0, pts=0),
        # The benchmark's system: a 20480-element sphere with 50 charges, solved, with the
        # energy, the surface potential and the potential at points in the molecule read back.
        dict(name="solve_sphere", kind="solve", n=20480, nc=50, precision="MIXED_DF64", precond=0, pts=1000),
        # Many small molecules of uneven size in one handle (conformers, fragments).
        dict(name="solve_batch", kind="batch", surfaces=12, n_min=320, n_max=5120, nc=30, precond=1),
        # Forces on the charges through autograd: 16 charge sets, forward and backward.
        dict(name="forces_sets", kind="forces", n=5120, nc=200, sets=16, precision="MIXED_TENSOR", precond=1),
        # The FP32 mat-vec of a Krylov loop, at the benchmark's size ...
        dict(name="matvec_f32", kind="matvec", n=20480, vecs=1, precision="FP32", transpose=0, kappa=KAPPA),
        # ... and its transpose (adjoint solves) on a larger surface whose size no tile divides.
        dict(name="matvec_f32_t", kind="matvec", n=65537, vecs=1, precision="FP32", transpose=1, kappa=KAPPA),
        # The double-float mat-vec: the residual of every mixed solve.
        dict(name="matvec_df64", kind="matvec", n=20480, vecs=1, precision="DF64", transpose=0, kappa=KAPPA),
        # The FP64 mat-vec, transposed: reference solves and their adjoints.
        dict(name="matvec_f64_t", kind="matvec", n=7001, vecs=1, precision="FP64", transpose=1, kappa=KAPPA),
        # 64 right-hand sides of one surface at once: the tensor-core operator ...
        dict(name="sets_tensor", kind="matvec", n=40001, vecs=64, precision="TENSOR", transpose=0, kappa=KAPPA),
        # ... and the double-float residual of such a batch.
        dict(name="sets_df64", kind="matvec", n=20001, vecs=64, precision="DF64", transpose=0, kappa=KAPPA),
        # The far-field operator on a large molecule.
        dict(name="treecode", kind="matvec", n=120001, vecs=1, precision="TREE32", transpose=0, kappa=KAPPA),
        # Source term and solvation energy of 2000 charges (a protein), four charge sets.
        dict(name="charges", kind="charges", n=40961, nc=2000, sets=4),
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "batch", "forces", "charges"] + 8 * ["matvec"])
    if kind == "solve":
        return dict(kind=kind, n=_size(rng, 320, 20480), nc=_size(rng, 1, 300), precision="MIXED_DF64",
                    precond=rng.randint(0, 1), pts=rng.choice([0, _size(rng, 1, 3000)]))
    if kind == "batch":
        return dict(kind=kind, surfaces=rng.randint(2, 16), n_min=_size(rng, 200, 1500), n_max=_size(rng, 1500, 5200),
                    nc=_size(rng, 1, 100), precond=rng.randint(0, 1))
    if kind == "forces":
        sets = _size(rng, 1, 32)
        return dict(kind=kind, n=_size(rng, 640, 5200), nc=_size(rng, 2, 300), sets=sets,
                    precision="MIXED_TENSOR" if sets >= 8 else "MIXED_DF64", precond=rng.randint(0, 1))
    if kind == "charges":
        return dict(kind=kind, n=_size(rng, 1000, 41000), nc=_size(rng, 10, 2000), sets=_size(rng, 1, 4))
    precision = rng.choice(["FP32", "FP32", "DF64", "DF64", "FP64", "TENSOR", "SETS_DF64", "TREE32"])
    lo, hi, vecs = {"FP32": (1000, 66000, 1), "DF64": (1000, 21000, 1), "FP64": (500, 7100, 1),
                    "TENSOR": (2000, 41000, _size(rng, 4, 64)), "SETS_DF64": (1000, 20500, _size(rng, 4, 64)),
                    "TREE32": (20000, 121000, 1)}[precision]
    return dict(kind="matvec", n=_size(rng, lo, hi), vecs=vecs, precision=precision.replace("SETS_", ""),
                transpose=rng.randint(0, 1), kappa=rng.choice([KAPPA, KAPPA, 0.05, 0.4]))


# ------------------------------------------------------------------ inputs
def _surface(n, rng):
    """Centroids, normals and areas of n elements on a displaced sphere r = R f(direction),
    and a function of directions giving r."""
    radius = 20.0 * math.sqrt(n / 20480.0)
    k = np.arange(n)
    z = 1.0 - (2.0 * k + 1.0) / n
    ang = k * (math.pi * (3.0 - math.sqrt(5.0)))
    rho = np.sqrt(1.0 - z * z)
    d = np.stack([rho * np.cos(ang), rho * np.sin(ang), z], 1)
    q, _ = np.linalg.qr(rng.standard_normal((3, 3)))
    d = d @ q.T
    wave = rng.standard_normal((6, 3)) * rng.uniform(0.5, 3.0, (6, 1))
    phase = rng.uniform(0.0, 2.0 * math.pi, 6)
    amp = 0.04 * rng.uniform(0.5, 1.0, 6)

    def f(dirs):
        return 1.0 + np.sin(dirs @ wave.T + phase) @ amp

    r = f(d)
    g = (np.cos(d @ wave.T + phase) * amp) @ wave
    g -= np.sum(g * d, 1, keepdims=True) * d
    nrm = r[:, None] * d - g
    length = np.linalg.norm(nrm, axis=1)
    area = (radius * r) * (radius * length) * (4.0 * math.pi / n)
    return radius * r[:, None] * d, nrm / length[:, None], area, lambda dirs: radius * f(dirs)


def _charges(n, rng, radius_of):
    d = rng.standard_normal((n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    return (0.8 * radius_of(d) * rng.uniform(0.0, 1.0, n) ** (1.0 / 3.0))[:, None] * d, rng.uniform(-1.0, 1.0, n)


def _charge_sets(case, rng, radius_of):
    got = [_charges(case["nc"], rng, radius_of) for _ in range(case["sets"])]
    return np.stack([p for p, _ in got]), np.stack([q for _, q in got])


def _batch(case, rng):
    sizes = np.exp(np.linspace(math.log(case["n_min"]), math.log(case["n_max"]), case["surfaces"]))
    surfaces, charges = [], []
    for n in np.rint(sizes).astype(int):
        c, v, a, rf = _surface(int(n), rng)
        surfaces.append((c, v, a))
        charges.append(_charges(case["nc"], rng, rf))
    return surfaces, charges


def _inputs(case, seed):
    """The host arrays of a case (every kind but "batch")."""
    rng = np.random.default_rng([seed, 77])
    c, v, a, rf = _surface(case["n"], rng)
    x = dict(c=c, v=v, a=a)
    if case["kind"] == "solve":
        x["pos"], x["q"] = _charges(case["nc"], rng, rf)
        x["pts"] = _charges(case["pts"], rng, rf)[0] if case["pts"] else None
    elif case["kind"] in ("forces", "charges"):
        x["pos"], x["q"] = _charge_sets(case, rng, rf)
    return x


def _vectors(case, seed, k, n):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 13)
    return torch.randn((k, 2 * n) if k > 1 else (2 * n,), dtype=torch.float64, device="cuda", generator=g)


def _params(case, precision):
    # 1e-10, two refinement steps: energies, potentials and forces are read to nine digits
    return bipb.solve_params(EPS_IN, EPS_OUT, KAPPA, tol=1e-10, precision=getattr(bipb, precision),
                             precond=case["precond"])


def prepare(case, seed):
    case = dict(case)
    if case["kind"] == "batch":
        surfaces, charges = _batch(case, np.random.default_rng([seed, 77]))
        return dict(case=case, surface=bipb.BatchSurface(surfaces), charges=charges,
                    params=_params(case, "MIXED_DF64"))
    x = _inputs(case, seed)
    s = bipb.Surface(x["c"], x["v"], x["a"])
    state = dict(case=case, surface=s)
    if case["kind"] == "matvec":
        u = _vectors(case, seed, case["vecs"], case["n"])
        state |= dict(u=u, y=torch.empty_like(u), precision=getattr(bipb, case["precision"]),
                      med=bipb.medium(EPS_IN, EPS_OUT, case["kappa"]))
        if case["precision"] == "TREE32":
            s.treecode_stats()  # the tree is built once per surface
    elif case["kind"] == "charges":
        s.set_charges(x["pos"], x["q"])
        u = _vectors(case, seed, case["sets"], case["n"])
        dev = dict(dtype=torch.float64, device="cuda")
        state |= dict(u=u, b=torch.empty_like(u), med=bipb.medium(EPS_IN, EPS_OUT, KAPPA),
                      phi=torch.empty(case["sets"] * case["nc"], **dev), e=torch.empty(case["sets"], **dev))
    elif case["kind"] == "forces":
        state |= dict(pos=torch.tensor(x["pos"], device="cuda"), q=torch.tensor(x["q"], device="cuda"),
                      params=_params(case, case["precision"]))
    else:
        state |= dict(pos=x["pos"], q=x["q"], pts=x["pts"], params=_params(case, case["precision"]))
    return state


def run(state):
    case, s = state["case"], state["surface"]
    if case["kind"] == "matvec":
        y = s.matvec(state["u"], state["y"], precision=state["precision"], transpose=bool(case["transpose"]),
                     med=state["med"])
        return y.float() if case["precision"] in SINGLE else y
    if case["kind"] == "charges":
        s.source(state["b"], med=state["med"])
        s.reaction(state["u"], phi_reac=state["phi"], e_sol=state["e"], med=state["med"])
        return dict(b=state["b"], phi=state["phi"], e=state["e"])
    if case["kind"] == "forces":
        q, pos = state["q"].detach().requires_grad_(), state["pos"].detach().requires_grad_()
        e = BipbEnergy.apply(q, pos, s, state["params"])
        e.sum().backward()
        return dict(e=e.detach(), dq=q.grad, dpos=pos.grad)
    if case["kind"] == "batch":
        s.set_charges(state["charges"])
        s.solve(state["params"])
        phi, dphi = s.surface_potential()
        return dict(e=s.energy(), phi=np.concatenate(phi), dphi=np.concatenate(dphi))
    s.set_charges(state["pos"], state["q"])
    s.solve(state["params"])
    phi, dphi = s.surface_potential()
    out = dict(e=s.energy(), phi=phi, dphi=dphi)
    if state["pts"] is not None:
        out["inside"] = s.potential_at(state["pts"], inside=True)
    return out


# ------------------------------------------------------------------ work
#: conventional operations of one ordered pair of the mat-vec (two square roots and exponentials aside)
PAIR = 63


def _solve_work(n, steps):
    return dict(bytes=8.0 * (7 * n + 2 * n), flops=float(PAIR) * n * n * steps)


def work(case):
    kind = case["kind"]
    if kind == "matvec":
        n, k = case["n"], case["vecs"]
        # each kernel block once, then four multiply-adds for each right-hand side;
        # the far field evaluates about a quarter of the pairs, fewer on larger surfaces
        pairs = float(n) * (n - 1) if case["precision"] != "TREE32" else 20000.0 * n
        return dict(bytes=8.0 * (7 * n + 4 * n * k), flops=pairs * (PAIR + 8.0 * (k - 1)))
    if kind == "charges":
        n, m = case["n"], case["nc"] * case["sets"]
        return dict(bytes=8.0 * (7 * n + 4 * n * case["sets"] + 5 * m), flops=50.0 * n * m)
    if kind == "batch":
        sizes = np.exp(np.linspace(math.log(case["n_min"]), math.log(case["n_max"]), case["surfaces"]))
        steps = 12 if case["precond"] else 40
        return dict(bytes=8.0 * 9 * float(sizes.sum()), flops=float(PAIR) * float((sizes ** 2).sum()) * steps)
    if kind == "forces":
        n, k = case["n"], case["sets"]
        steps = 2 * (12 if case["precond"] else 40)
        return dict(bytes=8.0 * (7 * n + 8 * case["nc"] * k), flops=float(n) * n * steps * (PAIR + 8.0 * (k - 1)))
    return _solve_work(case["n"], 12 if case["precond"] else 40)


# ------------------------------------------------------------------ 64-bit answers in plain torch
def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _blocks(xt, nt, xs, ns, ds, kappa, first):
    """K1..K4 (times 4 pi ds_j) of targets (rows first ...) against all sources; the self pair is zero."""
    d = [xt[:, k, None] - xs[None, :, k] for k in range(3)]
    r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
    rows = torch.arange(xt.shape[0], device=xt.device)
    if first is not None:
        r2[rows, rows + first] = math.inf
    s = r2.rsqrt()
    r = torch.where(torch.isinf(r2), torch.zeros_like(r2), r2 * s)
    kr = kappa * r
    e = torch.exp(-kr)
    t = e * (1.0 + kr)
    w = e * (3.0 + 3.0 * kr + kr * kr)
    eps = EPS_OUT / EPS_IN
    cj = ns[:, 0] * d[0] + ns[:, 1] * d[1] + ns[:, 2] * d[2]
    s3 = s * s * s * ds
    k1 = -torch.expm1(-kr) * s * ds
    k2 = (eps * t - 1.0) * cj * s3
    if nt is None:
        return k1, k2, None, None
    ci = nt[:, 0, None] * d[0] + nt[:, 1, None] * d[1] + nt[:, 2, None] * d[2]
    k3 = (t / eps - 1.0) * ci * s3
    k4 = ((t - 1.0) * (nt @ ns.T) - (w - 3.0) * ci * cj * (s * s)) * s3
    return k1, k2, k3, k4


def _rows(n):
    return max(1, int(1.5e8 // n))


def _apply(x, u, kappa, transpose):
    """A u or A^T u for u (k, 2n), without keeping A."""
    xs, ns, ds = _t(x["c"]), _t(x["v"]), _t(x["a"])
    n = xs.shape[0]
    eps = EPS_OUT / EPS_IN
    phi, psi = u[:, :n], u[:, n:]
    y = torch.cat([0.5 * (1 + eps) * phi, 0.5 * (1 + 1 / eps) * psi], 1)
    for i in range(0, n, _rows(n)):
        j = min(n, i + _rows(n))
        k1, k2, k3, k4 = _blocks(xs[i:j], ns[i:j], xs, ns, ds, kappa, i)
        if transpose:
            y[:, :n] -= (phi[:, i:j] @ k2 + psi[:, i:j] @ k4) / (4 * math.pi)
            y[:, n:] -= (phi[:, i:j] @ k1 + psi[:, i:j] @ k3) / (4 * math.pi)
        else:
            y[:, i:j] -= (phi @ k2.T + psi @ k1.T) / (4 * math.pi)
            y[:, n + i:n + j] -= (phi @ k4.T + psi @ k3.T) / (4 * math.pi)
    return y


def _dense(x):
    xs, ns, ds = _t(x["c"]), _t(x["v"]), _t(x["a"])
    n = xs.shape[0]
    eps = EPS_OUT / EPS_IN
    a = torch.empty((2 * n, 2 * n), dtype=torch.float64, device="cuda")
    for i in range(0, n, _rows(n)):
        j = min(n, i + _rows(n))
        k1, k2, k3, k4 = _blocks(xs[i:j], ns[i:j], xs, ns, ds, KAPPA, i)
        a[i:j, :n], a[i:j, n:], a[n + i:n + j, :n], a[n + i:n + j, n:] = -k2, -k1, -k4, -k3
    a /= 4 * math.pi
    dg = a.diagonal()
    dg[:n] += 0.5 * (1 + eps)
    dg[n:] += 0.5 * (1 + 1 / eps)
    return a


def _krylov(a, b):
    """a u = b by GMRES without restarts, right-preconditioned by the diagonal, restarted on the true residual."""
    dg = a.diagonal().clone()
    u = torch.zeros_like(b)
    for _ in range(4):
        r = b - a @ u
        beta = float(r.norm())
        if beta <= 1e-15 * float(b.norm()):
            break
        basis, cols = [r / beta], []
        for k in range(30):
            w = a @ (basis[k] / dg)
            h = torch.zeros(k + 2, dtype=torch.float64, device="cuda")
            v = torch.stack(basis)
            for _ in range(2):
                p = v @ w
                h[:k + 1] += p
                w = w - p @ v
            h[k + 1] = w.norm()
            cols.append(h)
            if float(h[k + 1]) < 1e-14:
                break
            basis.append(w / h[k + 1])
        m = len(cols)
        hm = np.zeros((m + 1, m))
        for k, h in enumerate(cols):
            hm[:k + 2, k] = h.cpu().numpy()
        g = np.zeros(m + 1)
        g[0] = beta
        y = _t(np.linalg.lstsq(hm, g, rcond=None)[0])
        u = u + (y @ torch.stack(basis[:m])) / dg
    return u


def _source(x, pos, q):
    """b = [S1; S2] of one charge set; differentiable in pos and q."""
    xs, ns = _t(x["c"]), _t(x["v"])
    d = xs[:, None, :] - pos[None, :, :]
    r = d.norm(dim=2)
    s1 = (q / r).sum(1)
    s2 = -(q * (ns[:, None, :] * d).sum(2) / r ** 3).sum(1)
    return torch.cat([s1, s2]) / (4 * math.pi * EPS_IN)


def _reaction(x, pos, u):
    """phi_reac at pos from u = [phi; psi]; differentiable in pos."""
    xs, ns, ds = _t(x["c"]), _t(x["v"]), _t(x["a"])
    n = xs.shape[0]
    k1, k2, _, _ = _blocks(pos, None, xs, ns, ds, KAPPA, None)
    return (k1 @ u[n:] + k2 @ u[:n]) / (4 * math.pi)


def _solve_exact(x, pos, q):
    pos, q = _t(pos), _t(q)
    u = _krylov(_dense(x), _source(x, pos, q))
    n = x["c"].shape[0]
    e = 0.5 * KCAL * float(q @ _reaction(x, pos, u))
    return e, KCAL * u[:n], KCAL * u[n:], u


def exact(case, seed):
    if case["kind"] == "batch":
        surfaces, charges = _batch(case, np.random.default_rng([seed, 77]))
        got = [_solve_exact(dict(c=c, v=v, a=a), p, q) for (c, v, a), (p, q) in zip(surfaces, charges)]
        return dict(e=np.array([g[0] for g in got]), phi=torch.cat([g[1] for g in got]),
                    dphi=torch.cat([g[2] for g in got]))
    x = _inputs(case, seed)
    if case["kind"] == "matvec":
        u = _vectors(case, seed, case["vecs"], case["n"])
        return _apply(x, u.reshape(case["vecs"], -1), case["kappa"], bool(case["transpose"])).reshape(u.shape)
    if case["kind"] == "charges":
        u = _vectors(case, seed, case["sets"], case["n"]).reshape(case["sets"], -1)
        b, phi, e = [], [], []
        for k in range(case["sets"]):
            pos, q = _t(x["pos"][k]), _t(x["q"][k])
            b.append(_source(x, pos, q))
            phi.append(_reaction(x, pos, u[k]))
            e.append(0.5 * KCAL * float(q @ phi[-1]))
        shape = (case["sets"], -1) if case["sets"] > 1 else (-1,)
        return dict(b=torch.cat(b).reshape(shape), phi=torch.cat(phi), e=np.array(e))
    if case["kind"] == "forces":
        a = _dense(x)
        at = a.T.contiguous()
        es, dqs, dps = [], [], []
        for k in range(case["sets"]):
            pos, q = _t(x["pos"][k]).requires_grad_(), _t(x["q"][k]).requires_grad_()
            u = _krylov(a, _source(x, pos, q).detach())
            # c . u = sum_k q_k phi_reac(y_k): its row c is the gradient with respect to u
            ur = u.clone().requires_grad_()
            cu = q @ _reaction(x, pos, ur)
            c, = torch.autograd.grad(cu, ur, retain_graph=True)
            lam = _krylov(at, c)
            half = 0.5 * KCAL * (cu + lam @ _source(x, pos, q))
            gq, gp = torch.autograd.grad(half, (q, pos))
            es.append(0.5 * KCAL * float(cu.detach()))
            dqs.append(gq)
            dps.append(gp)
        return dict(e=np.array(es), dq=torch.stack(dqs), dpos=torch.stack(dps))
    e, phi, dphi, u = _solve_exact(x, x["pos"], x["q"])
    out = dict(e=np.array([e]), phi=phi[None], dphi=dphi[None])
    if x["pts"] is not None:
        p = _t(x["pts"])
        inv = (p[:, None, :] - _t(x["pos"])[None]).norm(dim=2).reciprocal()
        out["inside"] = (KCAL * (_reaction(x, p, u) + inv @ _t(x["q"]) / (4 * math.pi * EPS_IN)))[None]
    return out
