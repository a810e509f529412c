"""Edges of the kernels' arithmetic against the FP64 CPU oracle (through the C ABI).

Tolerances are those of tests/test_gpu_parity.py: 1e-12 of the largest output
for the double-float charge passes, 2e-12 for the double-float mat-vec.
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


@pytest.mark.parametrize("far", [1.0, 1.9, 37.0, 1e5])
def test_charge_pass_grid_follows_the_farthest_charge(bipb, orc, far):
    """The coordinate grid of the double-float charge passes covers the surface and
    the charges of its system: one charge `far` surface radii away, on either side
    of a power of two and far outside, set from the host and from the device."""
    p = synth.kirkwood_problem(level=3)
    eps = p.eps_out / p.eps_in
    pos = p.charge_pos.copy()
    pos[3] = [0.0, -far * 20.0, 0.3]
    u = np.random.default_rng(5).standard_normal(2 * p.n)
    b_ref = orc.source(p.centroids, p.normals, pos, p.q[0], p.eps_in)
    e_ref, pr_ref = orc.energy(p.centroids, p.normals, p.areas, eps, p.kappa, pos, p.q[0], u)
    med = bipb.medium(p.eps_in, p.eps_out, p.kappa)
    got = []
    with bipb.Surface(p.centroids, p.normals, p.areas) as s:
        for device in (False, True):
            s.set_charges_dev(_dev(pos), _dev(p.q)) if device else s.set_charges(pos, p.q)
            b = _dev(np.zeros(2 * p.n))
            pr, e = _dev(np.zeros(p.nc)), _dev(np.zeros(1))
            s.source(b, med=med)
            s.reaction(_dev(u), pr, e, med=med)
            np.testing.assert_allclose(b.cpu().numpy(), b_ref, rtol=0, atol=1e-12 * np.abs(b_ref).max())
            np.testing.assert_allclose(pr.cpu().numpy(), pr_ref, rtol=0, atol=1e-12 * np.abs(pr_ref).max())
            got.append((b.cpu().numpy(), pr.cpu().numpy()))
    np.testing.assert_array_equal(got[0][0], got[1][0])
    np.testing.assert_array_equal(got[0][1], got[1][1])


@pytest.mark.parametrize("scale", [1e-3, 1.0, 31.0, 1e4])
def test_double_float_matvec_grid_scales_with_the_surface(bipb, orc, scale):
    """The double-float mat-vec's coordinate grid is taken from the surface's own
    extent times kappa: small and large surfaces in one batch handle, both directions."""
    p = synth.kirkwood_problem(level=2)
    parts = [(p.centroids * f, p.normals, p.areas * f * f) for f in (1.0, scale)]
    kappa = 0.1257 / max(scale, 1.0)
    u = np.random.default_rng(7).standard_normal(4 * p.n)
    with bipb.BatchSurface(parts) as s:
        for transpose in (False, True):
            y = _dev(np.zeros_like(u))
            s.matvec(_dev(u), y, precision=bipb.DF64, transpose=transpose, med=bipb.medium(1.0, 80.0, kappa))
            y = y.cpu().numpy().reshape(2, -1)
            f = orc.matvec_t if transpose else orc.matvec
            for k, (c, n, a) in enumerate(parts):
                ref = f(c, n, a, 80.0, kappa, u.reshape(2, -1)[k])
                np.testing.assert_allclose(y[k], ref, rtol=0, atol=2e-12 * np.abs(ref).max(), err_msg=f"{transpose} {k}")


@pytest.mark.parametrize("n", [2, 3, 31, 33, 255, 257, 513, 1279, 1536, 1537, 4095, 4096])
@pytest.mark.parametrize("transpose", [False, True])
def test_fp32_symmetric_shapes_small_and_ragged(bipb, orc, n, transpose):
    """Every shape of the packed symmetric FP32 mat-vec (and the default's choice by
    size) on surfaces around its tiles of 256 and 512 targets, its chunks of 32 and 64
    sources and the line between shapes: the FP32 bounds of test_matvec_fp64_and_fp32."""
    p = synth.protein_like_problem(level=4, n_charges=3)
    keep = np.sort(np.random.default_rng(n).choice(p.n, n, replace=False))
    c, nv, a = p.centroids[keep], p.normals[keep], p.areas[keep]
    u = np.random.default_rng(3).standard_normal(2 * n)
    for kappa in (p.kappa, 0.0):
        ref = (orc.matvec_t if transpose else orc.matvec)(c, nv, a, 80.0, kappa, u)
        with bipb.Surface(c, nv, a) as s:
            for variant in (7, 8, 9):
                s.set_variant(variant)
                y = _dev(np.zeros_like(u))
                s.matvec(_dev(u), y, precision=bipb.FP32, transpose=transpose, med=bipb.medium(1.0, 80.0, kappa))
                y = y.cpu().numpy()
                assert np.linalg.norm(y - ref) < 3e-6 * np.linalg.norm(ref), (variant, kappa)
                assert np.abs(y - ref).max() < 2e-5 * np.abs(ref).max(), (variant, kappa)


@pytest.mark.parametrize("n,sets,precond", [(2, 1, 0), (37, 20, 1), (37, 21, 1), (2048, 1, 0), (2049, 1, 0), (2560, 1, 0), (2561, 2, 1)])
def test_krylov_step_as_cluster_and_as_kernels(bipb, orc, n, sets, precond):
    """The Arnoldi step as one cluster launch per system (small systems, up to 20 of
    them) and as three kernels, on both sides of the lines between them, with the
    fused FP32 mat-vec and (FP64) without: mixed and FP64 solves against the
    oracle's, 1e-7 and 1e-9 of the energy (test_kirkwood_solve's bounds or looser)."""
    p = synth.protein_like_problem(level=4, n_charges=3)
    keep = np.sort(np.random.default_rng(n).choice(p.n, n, replace=False))
    p.centroids, p.normals, p.areas = p.centroids[keep], p.normals[keep], p.areas[keep]
    q = np.random.default_rng(1).uniform(-1.0, 1.0, (sets, p.nc))
    p.q = q
    ref = [orc.solve(p, rhs=r, method="gmres", tol=1e-12).energy_kcal for r in range(min(sets, 2))]
    for prec, tol, rt in ((bipb.MIXED_DF64, 1e-9, 1e-7), (bipb.FP64, 1e-11, 1e-9)):
        if prec == bipb.FP64 and n > 2560:
            continue
        for restart in (10, 3):
            with bipb.Surface(p.centroids, p.normals, p.areas) as s:
                s.set_charges(p.charge_pos, q)
                info = s.solve(eps_in=p.eps_in, eps_out=p.eps_out, kappa=p.kappa, tol=tol, precision=prec,
                               precond=precond, restart=restart)
                assert all(i["converged"] for i in info)
                np.testing.assert_allclose(s.energy()[:2], ref, rtol=rt)


@pytest.mark.parametrize("n", [2, 63, 65, 515])
@pytest.mark.parametrize("kappa", [0.0, 9e-7, 1.1e-6, 0.1257, 2.5])
@pytest.mark.parametrize("transpose", [False, True])
def test_multi_rhs_double_float_scaling_rule(bipb, orc, n, kappa, transpose):
    """The multi-RHS double-float passes on both sides of the rule that scales their
    coordinates by kappa (1e-6), on surfaces around one tile of 64 targets and one
    step of 16 sources, on the CUDA cores (3 right-hand sides, forward) and as exact
    digits (17): the bound of test_multi_rhs_df64_matvec_matches_oracle."""
    p = synth.protein_like_problem(level=3, n_charges=3)
    keep = np.sort(np.random.default_rng(n).choice(p.n, n, replace=False))
    c, nv, a = p.centroids[keep], p.normals[keep], p.areas[keep]
    f = orc.matvec_t if transpose else orc.matvec
    for n_rhs in (3, 17):
        U = np.random.default_rng(n + n_rhs).standard_normal((n_rhs, 2 * n))
        with bipb.Surface(c, nv, a) as s:
            yd = torch.full_like(_dev(U), float("nan"))
            s.matvec(_dev(U), yd, precision=bipb.DF64, transpose=transpose, med=bipb.medium(1.0, 80.0, kappa))
            Y = yd.cpu().numpy()
        for r in (0, n_rhs - 1):
            ref = f(c, nv, a, 80.0, kappa, U[r])
            np.testing.assert_allclose(Y[r], ref, rtol=0, atol=2e-12 * np.abs(ref).max(), err_msg=f"{n_rhs} {r}")


@pytest.mark.parametrize("n,params", [(33, (0.8, 4, 32)), (257, (0.9, 4, 32)), (1280, (0.9, 8, 33)), (1111, (0.7, 6, 64))])
@pytest.mark.parametrize("kappa", [0.0, 9e-7, 1.1e-6, 0.4])
@pytest.mark.parametrize("transpose", [False, True])
def test_treecode_forms_and_ragged_leaves(bipb, orc, n, params, kappa, transpose):
    """The packed far-field pass in its three forms (both sides of the lines at kappa =
    0 and 1e-6), with odd leaves and proxy counts, several elements on a group of the
    upward pass and one leaf only: test_treecode_matvec_matches_oracle_treecode's bounds."""
    p = synth.protein_like_problem(level=3, n_charges=3)
    keep = np.sort(np.random.default_rng(n).choice(p.n, min(n, p.n), replace=False))
    c, nv, a = p.centroids[keep], p.normals[keep], p.areas[keep]
    u = np.random.default_rng(4).standard_normal(2 * len(keep))
    with bipb.Surface(c, nv, a) as s:
        s.treecode(*params)
        y = torch.full_like(_dev(u), float("nan"))
        s.matvec(_dev(u), y, precision=bipb.TREE32, transpose=transpose, med=bipb.medium(1.0, 80.0, kappa))
        y = y.cpu().numpy()
    ref = orc.treecode.matvec(c, nv, a, 80.0, kappa, u, *params, transpose=transpose)
    assert np.linalg.norm(y - ref) < 3e-6 * np.linalg.norm(ref)
    assert np.abs(y - ref).max() < 2e-5 * np.abs(ref).max()


@pytest.mark.parametrize("n", [2, 31, 33, 64, 65, 129, 1280])
@pytest.mark.parametrize("scale,kappa", [(1.0, 0.0), (1.0, 0.1257), (1e-3, 1.1e-6), (1e-3, 2.5), (1e3, 2.5), (1e3, 1.1e-6)])
def test_fp64_symmetric_pair_range(bipb, orc, n, scale, kappa):
    """The symmetric FP64 mat-vec, its radial factors in triple-float arithmetic, from
    kappa r = 1e-9 (t - 1 cancels) to 1e5 (e^{-kappa r} underflows), on surfaces around
    its blocks of 32 sources and tiles of 64 targets, both directions: the FP64 bound of
    test_matvec_fp64_and_fp32.  Without contrast and screening the kernels vanish exactly."""
    p = synth.protein_like_problem(level=3, n_charges=3)
    keep = np.sort(np.random.default_rng(n).choice(p.n, min(n, p.n), replace=False))
    c, nv, a = scale * p.centroids[keep], p.normals[keep], scale * scale * p.areas[keep]
    u = np.random.default_rng(9).standard_normal(2 * len(keep))
    with bipb.Surface(c, nv, a) as s:
        for transpose in (False, True):
            for eps in (80.0, 1.0):
                y = torch.full_like(_dev(u), float("nan"))
                s.matvec(_dev(u), y, precision=bipb.FP64, transpose=transpose, med=bipb.medium(1.0, eps, kappa))
                y = y.cpu().numpy()
                ref = (orc.matvec_t if transpose else orc.matvec)(c, nv, a, eps, kappa, u)
                np.testing.assert_allclose(y, ref, rtol=0, atol=1e-12 * np.abs(ref).max(), err_msg=f"{transpose} {eps}")
                if eps == 1.0 and kappa == 0.0:
                    np.testing.assert_array_equal(y, u)


@pytest.mark.parametrize("transpose", [False, True])
def test_tensor_right_hand_side_packing(bipb, orc, transpose):
    """The packing of right-hand sides by their bits: values over forty orders of
    magnitude within one right-hand side, subnormals, an infinity and a NaN, whose
    right-hand sides come out not finite while the others keep the FP32 bounds of
    test_tensor_core_matvec_matches_oracle; more sources than one pass of the maximum's
    cluster takes, an odd number."""
    p = synth.protein_like_problem(level=4, n_charges=3)
    n = 4099
    keep = np.sort(np.random.default_rng(n).choice(p.n, n, replace=False))
    c, nv, a = p.centroids[keep], p.normals[keep], p.areas[keep]
    rng = np.random.default_rng(6)
    U = rng.standard_normal((6, 2 * n))
    U[1] *= 10.0 ** rng.uniform(-40, 0, 2 * n)
    U[2, ::3] *= 1e-310
    U[3, 5] = np.inf
    U[4, n + 7] = np.nan
    med = bipb.medium(p.eps_in, p.eps_out, p.kappa)
    with bipb.Surface(c, nv, a) as s:
        yd = torch.zeros_like(_dev(U))
        s.matvec(_dev(U), yd, precision=bipb.TENSOR, transpose=transpose, med=med)
        Y = yd.cpu().numpy()
    f = orc.matvec_t if transpose else orc.matvec
    for r in (0, 1, 2, 5):
        ref = f(c, nv, a, p.eps_out / p.eps_in, p.kappa, U[r])
        assert np.linalg.norm(Y[r] - ref) < 3e-6 * np.linalg.norm(ref), r
        assert np.abs(Y[r] - ref).max() < 2e-5 * np.abs(ref).max(), r
    assert not np.isfinite(Y[3:5]).any()


@pytest.mark.parametrize("nc", [1, 31, 33, 257, 300])
def test_reaction_reduction_tiles(bipb, orc, nc):
    """The reduction of the reaction potentials over tiles of 32 charges, one block of
    the cluster each, and ranges of the splits (many for few charges): two charge sets
    of unequal size beside a tile's and the cluster's width, at 1e-12 as the charge passes."""
    p = synth.protein_like_problem(level=3, n_charges=nc, seed=2)
    u = np.random.default_rng(8).standard_normal(2 * p.n)
    eps = p.eps_out / p.eps_in
    q = np.asarray(p.q).reshape(-1, p.nc)[0]
    e_ref, pr_ref = orc.energy(p.centroids, p.normals, p.areas, eps, p.kappa, p.charge_pos, q, u)
    with bipb.Surface(p.centroids, p.normals, p.areas) as s:
        s.set_charges(p.charge_pos, np.stack([q, -2.0 * q]))
        pr, e = _dev(np.zeros((2, p.nc))), _dev(np.zeros(2))
        s.reaction(_dev(np.stack([u, u])), pr, e, med=bipb.medium(p.eps_in, p.eps_out, p.kappa))
        pr, e = pr.cpu().numpy(), e.cpu().numpy()
    for k, f in enumerate((1.0, -2.0)):
        np.testing.assert_allclose(pr[k], pr_ref, rtol=0, atol=1e-12 * np.abs(pr_ref).max())
        scale = 0.5 * orc.KCAL * np.abs(f * q).sum() * np.abs(pr_ref).max()
        assert abs(e[k] - orc.KCAL * f * e_ref) < 1e-12 * scale


@pytest.mark.parametrize("n", [5120, 5121])
@pytest.mark.parametrize("precision", ["FP64", "MIXED_TENSOR"])
def test_krylov_step_without_fused_matvec_at_its_line(bipb, orc, n, precision):
    """The Arnoldi step beside a mat-vec that is not fused into it (two Gram-Schmidt
    passes for FP64, one for the tensor-core operator), as one cluster launch up to 5120
    elements and as kernels above: energies against the oracle's solve, with the bounds
    of test_krylov_step_as_cluster_and_as_kernels."""
    p = synth.protein_like_problem(level=5, n_charges=3)
    keep = np.sort(np.random.default_rng(n).choice(p.n, n, replace=False))
    p.centroids, p.normals, p.areas = p.centroids[keep], p.normals[keep], p.areas[keep]
    ref = orc.solve(p, rhs=0, method="gmres", tol=1e-12).energy_kcal
    tol, rt = (1e-11, 1e-9) if precision == "FP64" else (1e-9, 1e-7)
    with bipb.Surface(p.centroids, p.normals, p.areas) as s:
        s.set_charges(p.charge_pos, p.q)
        info = s.solve(eps_in=p.eps_in, eps_out=p.eps_out, kappa=p.kappa, tol=tol, precision=getattr(bipb, precision),
                       precond=1)
        assert all(i["converged"] for i in info)
        np.testing.assert_allclose(s.energy()[0], ref, rtol=rt)
