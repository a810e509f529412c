"""Surfaces with pairs of elements far closer than a mesh has them, against the FP64 oracle.

Centroids are accepted as long as their FP32 copies differ, so no operator may lose a
pair because its distance is near the rounding of FP32 coordinates.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def bipb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_10044_gb300.build import build

    build()
    import paper_2312_10044_gb300 as b

    b.load_library()
    return b


@pytest.fixture(scope="module")
def orc():
    import oracle

    return oracle


def _dev(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _paired_sphere(radius, gap, tangent, n_pairs=40, seed=3):
    """A sphere of 320 elements, n_pairs of which get a neighbour `gap` away, along the
    sphere or in any direction; the neighbours' elements come last."""
    p = synth.kirkwood_problem(level=2)
    f = radius / np.linalg.norm(p.centroids, axis=1).mean()
    c, a = p.centroids * f, p.areas * f * f
    nv = c / np.linalg.norm(c, axis=1, keepdims=True)
    rng = np.random.default_rng(seed)
    at = rng.choice(p.n, n_pairs, replace=False)
    d = rng.standard_normal((n_pairs, 3))
    if tangent:
        d -= np.sum(d * nv[at], axis=1, keepdims=True) * nv[at]
    d *= gap / np.linalg.norm(d, axis=1, keepdims=True)
    c2 = c[at] + d
    if tangent:  # back onto the sphere: n.d is gap^2 / (2 radius)
        c2 *= (np.linalg.norm(c[at], axis=1) / np.linalg.norm(c2, axis=1))[:, None]
    n2 = c2 / np.linalg.norm(c2, axis=1, keepdims=True) if tangent else nv[at]
    return np.concatenate([c, c2]), np.concatenate([nv, n2]), np.concatenate([a, a[at]])


@pytest.mark.parametrize("n_rhs", [4, 17])
@pytest.mark.parametrize("kappa", [0.0, 0.1257])
@pytest.mark.parametrize("radius,gap,tangent", [(20.0, 0.02, True), (20.0, 0.01, True), (20.0, 0.003, True),
                                                (20.0, 1e-5, False), (100.0, 1e-5, False)])
def test_multi_rhs_double_float_close_pairs(bipb, orc, radius, gap, tangent, kappa, n_rhs):
    """The row scales of the exact tensor-core pass hold for the largest value of each
    row: pairs 0.02 to 1e-5 A apart, a few FP32 spacings of their coordinates.

    Bound per row, with M the row's largest coefficient bound a (s + s^2 + s^3), s = 1/r:
    1 - e and 1 - t carry an absolute error of a few 2^-47, so each coefficient one of
    (1 + eps) M times that, and the digits one of 2^-46 of the row's largest; 2^-40 leaves
    a factor of about sixty for the few roundings.
    """
    c, nv, a = _paired_sphere(radius, gap, tangent)
    n, eps = len(a), 80.0
    U = np.random.default_rng(n_rhs).standard_normal((n_rhs, 2 * n))
    r = np.linalg.norm(c[:, None] - c[None], axis=2)
    np.fill_diagonal(r, np.inf)
    s = 1.0 / r
    M = s + s**2 + s**3
    with bipb.Surface(c, nv, a) as srf:
        for transpose in (False, True):
            Y = torch.full_like(_dev(U), float("nan"))
            srf.matvec(_dev(U), Y, precision=bipb.DF64, transpose=transpose, med=bipb.medium(1.0, eps, kappa))
            Y = Y.cpu().numpy()
            rows = a * M.max(axis=1) if transpose else (M * a).max(axis=1)
            for k in (0, n_rhs - 1):
                ref = (orc.matvec_t if transpose else orc.matvec)(c, nv, a, eps, kappa, U[k])
                tol = 2.0**-40 * (1.0 + eps) * np.tile(rows, 2) * np.abs(U[k]).sum() + 2.0**-40 * np.abs(ref).max()
                worst = np.max(np.abs(Y[k] - ref) / tol)
                assert worst < 1.0, (transpose, k, worst)


def _capped_matvec(c, nv, a, eps, kappa, u, transpose):
    """A u or A^T u with 1/r at most 1e6 (pair.cuh) in FP64, 1 - t of small kappa r from
    its series, and per row the bound 1e-12 sum |K u|, plus 2^-54 s^3 ds |phi| in the psi
    row (1 - t is a difference of numbers near 1) and (1 + eps) 2^-66 s^3 ds |u| (the
    coordinates' grid: 2^-72 of 32 A and more for a difference, twice that)."""
    n = len(a)
    d = c[:, None, :] - c[None, :, :]
    r2 = np.sum(d * d, axis=2)
    with np.errstate(divide="ignore"):
        s = np.minimum(1.0 / np.sqrt(r2), 1e6)
    np.fill_diagonal(s, 0.0)
    x = kappa * r2 * s
    e = np.exp(-x)
    omt = np.where(x < 1e-2, x * x * (0.5 - x * (1 / 3 - x * (1 / 8 - x * (1 / 30 - x / 144)))), -np.expm1(-x) - x * e)
    ci, cj = np.einsum("ik,ijk->ij", nv, d), np.einsum("jk,ijk->ij", nv, d)
    w = e * kappa * kappa - 3.0 * omt * s**2  # (w - 3) s^2
    k1 = -np.expm1(-x) * s
    k2 = ((eps - 1.0) - eps * omt) * cj * s**3
    k3 = ((1.0 / eps - 1.0) - omt / eps) * ci * s**3
    k4 = (-omt * (nv @ nv.T) - w * ci * cj) * s**3
    B = np.block([[k2, k1], [k4, k3]]) * np.tile(a, 2)[None, :] / (4.0 * np.pi)
    g = (1.0 + eps) * 2.0**-66 * s**3
    E = np.block([[g, g], [g + 2.0**-54 * s**3, g]]) * np.tile(a, 2)[None, :] / (4.0 * np.pi)
    if transpose:
        B, E = B.T, E.T
    diag = np.repeat([0.5 * (1.0 + eps), 0.5 * (1.0 + 1.0 / eps)], n)
    return diag * u - B @ u, 1e-12 * (np.abs(B) @ np.abs(u) + diag * np.abs(u)) + E @ np.abs(u)


def _mirrored_surface(gap, n_pairs):
    """Elements at x and -x in turn (their mean is the origin exactly): half an
    icosphere of 20 A and n_pairs pairs `gap` apart near the middle, where FP32 copies
    that close differ; without pairs, one point gap / 2 from the origin, which is a
    pair with its mirror image."""
    p = synth.kirkwood_problem(level=1)
    half = p.centroids[p.centroids[:, 0] > 0.0]
    rng = np.random.default_rng(2)
    near = 0.2 * rng.standard_normal((n_pairs, 3))
    d = rng.standard_normal((max(n_pairs, 1), 3))
    d *= gap / np.linalg.norm(d, axis=1, keepdims=True)
    pts = np.concatenate([half, near, near + d] if n_pairs else [half, 0.5 * d])
    c = np.stack([pts, -pts], axis=1).reshape(-1, 3)
    nv = rng.standard_normal(c.shape)
    for _ in range(2):
        nv /= np.linalg.norm(nv, axis=1, keepdims=True)
    return c, nv, rng.uniform(0.5, 1.5, len(c)), rng.standard_normal(2 * len(c))


def _check_fp64(bipb, c, nv, a, u, kappa):
    with bipb.Surface(c, nv, a) as srf:
        for transpose in (False, True):
            y = torch.full_like(_dev(u), float("nan"))
            srf.matvec(_dev(u), y, precision=bipb.FP64, transpose=transpose, med=bipb.medium(1.0, 80.0, kappa))
            ref, tol = _capped_matvec(c, nv, a, 80.0, kappa, u, transpose)
            worst = np.max(np.abs(y.cpu().numpy() - ref) / tol)
            assert worst < 1.0, (transpose, worst)


@pytest.mark.parametrize("gap", [1e-2, 1e-4, 2e-6])
@pytest.mark.parametrize("kappa", [0.0, 0.1257])
def test_fp64_symmetric_close_pairs(bipb, gap, kappa):
    """Differences of the coordinates whose leading parts cancel keep FP64's digits in
    the symmetric FP64 mat-vec: components below the leading grid (4e-6 A here)."""
    _check_fp64(bipb, *_mirrored_surface(gap, 40), kappa)


@pytest.mark.parametrize("gap,n_pairs", [(3e-7, 6), (9.9e-7, 6), (1e-20, 0)])
@pytest.mark.parametrize("kappa", [0.0, 0.1257])
def test_fp64_symmetric_pair_keeps_the_cap_of_the_inverse_distance(bipb, gap, n_pairs, kappa):
    """1/r is capped at 1e-6 A in the symmetric FP64 mat-vec as in the ordered one, and a
    pair whose squared distance leaves the FP32 range stays finite."""
    _check_fp64(bipb, *_mirrored_surface(gap, n_pairs), kappa)


@pytest.mark.parametrize("n_rhs", [1, 5])
@pytest.mark.parametrize("kappa", [1e-8, 1e-5])
@pytest.mark.parametrize("gap", [0.05, 1e-3])
def test_double_float_t_minus_one_of_close_elements(bipb, gap, kappa, n_rhs):
    """K4 of close elements is s^3 (1 - t) with 1 - t far below e's rounding: its error
    stays that of e, also where nothing else is as large (no dielectric contrast, hardly
    any screening).  Bound per row: e = 1 - kappa r is held to 2^-50 (kappa r below 2^-24
    lies in its trailing part, rounded at 2^-24 of that), 2^-49 s^3 ds |phi| in the psi row and
    2^-48 (s + s^2) ds |u| for K1 to K3 (A^T likewise), and 2^-44 of the row's terms."""
    c, nv, a = _paired_sphere(20.0, gap, False)
    n = len(a)
    U = np.random.default_rng(n_rhs).standard_normal((n_rhs, 2 * n))
    x0 = c - c.mean(axis=0)
    with np.errstate(divide="ignore"):
        s = 1.0 / np.linalg.norm(x0[:, None] - x0[None], axis=2)
    np.fill_diagonal(s, 0.0)
    with bipb.Surface(c, nv, a) as srf:
        for transpose in (False, True) if n_rhs == 1 else (False,):
            Y = torch.full_like(_dev(U), float("nan"))
            srf.matvec(_dev(U), Y, precision=bipb.DF64, transpose=transpose, med=bipb.medium(1.0, 1.0, kappa))
            Y = Y.cpu().numpy()
            w = (a[:, None] if transpose else a[None, :]) / (4.0 * np.pi)
            for k in (0, n_rhs - 1):
                phi, psi = np.abs(U[k, :n]), np.abs(U[k, n:])
                ref, tol = _capped_matvec(x0, nv, a, 1.0, kappa, U[k], transpose)
                e1 = 2.0**-48 * (((s + s**2) * w) @ (phi + psi))
                e4 = 2.0**-49 * ((s**3 * w) @ (psi if transpose else phi))
                tol = 2.0**-44 * 1e12 * tol + np.concatenate([e1 + e4, e1] if transpose else [e1, e1 + e4])
                worst = np.max(np.abs(Y[k] - ref) / tol)
                assert worst < 1.0, (transpose, k, worst)
