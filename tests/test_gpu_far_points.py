"""Charge passes whose points spread far beyond the surface, against the FP64 oracle.

The coordinates of a pass share a grid set by its farthest point; one point far out
must not cost the others their digits.  Bounds as in test_gpu_arithmetic.py: 1e-12 of the
largest value.
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


@pytest.mark.parametrize("far", [0.9 * 2.0**20, 1.1 * 2.0**20, 1e9, 1e13])
@pytest.mark.parametrize("kappa", [0.0, 0.1257])
def test_potential_beside_a_far_point(bipb, orc, far, kappa):
    """Potentials at points near the surface beside some `far` radii away (on both sides
    of the line where the grid is given up): those near as the oracle's, those far to 1e-10
    of their own size where nothing screens them."""
    p = synth.kirkwood_problem(level=2)
    rng = np.random.default_rng(1)
    d = rng.standard_normal((40, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    r = np.concatenate([np.full(30, 23.0), 20.0 * far * rng.uniform(0.5, 1.0, 9), [20.0 * far]])
    eps = p.eps_out / p.eps_in
    with bipb.Surface(p.centroids, p.normals, p.areas) as s:
        s.set_charges(p.charge_pos, p.q)
        s.solve(eps_in=p.eps_in, eps_out=p.eps_out, kappa=kappa, tol=1e-12, precision=bipb.FP64)
        phi, dphi = s.surface_potential()
        u = np.concatenate([np.ravel(phi), np.ravel(dphi)]) / orc.KCAL
        for inside, pts in ((True, d * np.where(r > 23.0, r, 12.0)[:, None]), (False, d * r[:, None])):
            got = np.ravel(s.potential_at(pts, inside=inside))
            q = np.asarray(p.q).reshape(-1)
            ref = orc.KCAL * np.ravel(orc.potential(p.centroids, p.normals, p.areas, eps, kappa, u, pts, inside,
                                                    p.charge_pos, q, p.eps_in))
            np.testing.assert_allclose(got[:30], ref[:30], rtol=0, atol=1e-12 * np.abs(ref).max())
            if not inside and kappa == 0.0:
                np.testing.assert_allclose(got[30:], ref[30:], rtol=1e-10)


@pytest.mark.parametrize("far", [0.9 * 2.0**20, 1.1 * 2.0**20, 1e9, 1e13])
def test_charge_passes_beside_a_far_charge(bipb, orc, far):
    """Source, reaction and gradient passes with one charge `far` radii out, set from the
    host and from the device: the other charges keep their digits."""
    p = synth.kirkwood_problem(level=2)
    eps = p.eps_out / p.eps_in
    pos, q = p.charge_pos.copy(), np.asarray(p.q).reshape(-1, p.nc)[0]
    pos[3] = [0.0, -far * 20.0, 0.3]
    u = np.random.default_rng(5).standard_normal(2 * p.n)
    b_ref = orc.source(p.centroids, p.normals, pos, q, p.eps_in)
    e_ref, pr_ref = orc.energy(p.centroids, p.normals, p.areas, eps, p.kappa, pos, q, u)
    med = bipb.medium(p.eps_in, p.eps_out, p.kappa)
    got = []
    with bipb.Surface(p.centroids, p.normals, p.areas) as s:
        for device in (False, True):
            s.set_charges_dev(_dev(pos), _dev(q)) if device else s.set_charges(pos, q)
            b, pr, e = _dev(np.zeros(2 * p.n)), _dev(np.zeros(p.nc)), _dev(np.zeros(1))
            s.source(b, med=med)
            s.reaction(_dev(u), pr, e, med=med)
            np.testing.assert_allclose(b.cpu().numpy(), b_ref, rtol=0, atol=1e-12 * np.abs(b_ref).max())
            np.testing.assert_allclose(pr.cpu().numpy(), pr_ref, rtol=0, atol=1e-12 * np.abs(pr_ref).max())
            np.testing.assert_allclose(pr[3].item(), pr_ref[3], rtol=1e-10)
            got.append(np.concatenate([b.cpu().numpy(), pr.cpu().numpy(), e.cpu().numpy()]))
        np.testing.assert_array_equal(got[0], got[1])
        # near charges again: the grid is back
        s.set_charges(p.charge_pos, p.q)
        s.source(b, med=med)
        ref = orc.source(p.centroids, p.normals, p.charge_pos, q, p.eps_in)
        np.testing.assert_allclose(b.cpu().numpy(), ref, rtol=0, atol=1e-12 * np.abs(ref).max())


@pytest.mark.parametrize("far", [1.1 * 2.0**20, 1e9])
def test_gradient_beside_a_far_charge(bipb, far):
    """Energy gradients of the near charges do not see a charge far out whose value is
    zero: as those without it, to 1e-9 of the largest."""
    p = synth.kirkwood_problem(level=2)
    pos, q = p.charge_pos.copy(), np.asarray(p.q).reshape(-1, p.nc)[0].copy()
    q[3] = 0.0
    got = []
    with bipb.Surface(p.centroids, p.normals, p.areas) as s:
        for y in (pos[3].copy(), np.array([0.0, -far * 20.0, 0.3])):
            pos[3] = y
            s.set_charges(pos, q)
            s.solve(eps_in=p.eps_in, eps_out=p.eps_out, kappa=p.kappa, tol=1e-12, precision=bipb.FP64)
            dq, dy = s.energy_grad(eps_in=p.eps_in, eps_out=p.eps_out, kappa=p.kappa, tol=1e-12, precision=bipb.FP64)
            keep = np.arange(p.nc) != 3
            got.append((np.ravel(s.energy())[0], np.ravel(dq)[keep], np.reshape(dy, (p.nc, 3))[keep]))
    for a, b in zip(*got):
        np.testing.assert_allclose(b, a, rtol=0, atol=1e-9 * np.abs(a).max())


@pytest.mark.parametrize("x", [4.0, 8.0, 16.0, 32.0, 60.0])
def test_exterior_potential_keeps_its_digits_where_it_is_screened(bipb, orc, x):
    """Potentials at points x Debye lengths out are of the order of e^{-x}: right
    relative to their own terms.  Bound: kappa r to a few 2^-48 of itself makes e^{-kappa r}
    wrong by x times that; over 1280 elements its random part averages out to less than
    x 2^-48, and 2e-14 for the other factors, both relative to the sum of the terms'
    magnitudes."""
    p = synth.kirkwood_problem(level=3)
    rng = np.random.default_rng(1)
    d = rng.standard_normal((200, 3))
    pts = d / np.linalg.norm(d, axis=1, keepdims=True) * (x / p.kappa)
    eps = p.eps_out / p.eps_in
    with bipb.Surface(p.centroids, p.normals, p.areas) as s:
        s.set_charges(p.charge_pos, p.q)
        s.solve(eps_in=p.eps_in, eps_out=p.eps_out, kappa=p.kappa, tol=1e-12, precision=bipb.FP64)
        phi, dphi = s.surface_potential()
        u = np.concatenate([np.ravel(phi), np.ravel(dphi)]) / orc.KCAL
        got = np.ravel(s.potential_at(pts, inside=False)) / orc.KCAL
    ref = np.ravel(orc.potential(p.centroids, p.normals, p.areas, eps, p.kappa, u, pts, False))
    r = np.linalg.norm(pts[:, None] - p.centroids[None], axis=2)
    e = np.exp(-p.kappa * r)
    size = ((e * (1.0 + p.kappa * r) / r**2) @ (p.areas * np.abs(u[:p.n])) + (e / r) @ (p.areas * np.abs(u[p.n:])) / eps) / (4.0 * np.pi)
    worst = np.max(np.abs(got - ref) / size)
    assert worst < x * 2.0**-48 + 2e-14, worst
