"""Single-precision mat-vecs of values near the top of the FP32 range."""
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


def _dev(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("n", [2000, 4500])
@pytest.mark.parametrize("kappa", [0.0, 0.1257])
def test_symmetric_sums_above_the_fp32_range(bipb, n, kappa):
    """Partial sums are FP32, their total is not bound by its range: with potentials of
    one sign whose largest row sum is 1.2 times the range's end (its partials are all below
    it), the result is that of u times the factor, to FP32 rounding."""
    p = synth.protein_like_problem(level=4, n_charges=3)
    keep = np.sort(np.random.default_rng(n).choice(p.n, n, replace=False))
    c, nv, a = p.centroids[keep], p.normals[keep], p.areas[keep] * (p.n / n)
    u = np.concatenate([np.ones(n), np.zeros(n)])
    med = bipb.medium(1.0, 80.0, kappa)
    with bipb.Surface(c, nv, a) as s:
        y = torch.zeros_like(_dev(u))
        s.matvec(_dev(u), y, precision=bipb.FP32, med=med)
        y1 = y.cpu().numpy()
        # the phi rows' sums, in the units in which they are summed (times 1 / kappa where scaled)
        top = 4.0 * np.pi * np.abs(0.5 * 81.0 - y1[:n]).max() / (kappa if kappa else 1.0)
        f = 1.2 * 2.0**128 / top
        s.matvec(_dev(u * f), y, precision=bipb.FP32, med=med)
        y2 = y.cpu().numpy() / f
    np.testing.assert_allclose(y2, y1, rtol=0, atol=3e-6 * np.abs(y1).max())


@pytest.mark.parametrize("scale", [1.0, 1e25])
@pytest.mark.parametrize("kappa", [1e-6, 1.1e-6, 1e-4, 9.99e-4, 1.001e-3])
@pytest.mark.parametrize("transpose", [False, True])
def test_weak_screening_keeps_the_range(bipb, transpose, kappa, scale):
    """The far-field and the multi-RHS double-float passes with Debye lengths of 1000 to
    10^6 A, a contrast of 1000 and values up to 1e25, on both sides of the line of their
    scaled form (1e-3): the bounds of test_treecode_matvec_matches_oracle_treecode and
    test_multi_rhs_df64_matvec_matches_oracle."""
    import oracle as orc

    p = synth.protein_like_problem(level=3, n_charges=3)
    keep = np.sort(np.random.default_rng(3).choice(p.n, 515, replace=False))
    c, nv, a = p.centroids[keep], p.normals[keep], p.areas[keep]
    n, eps = len(a), 1000.0
    med = bipb.medium(1.0, eps, kappa)
    U = scale * np.random.default_rng(5).standard_normal((17, 2 * n))
    f = orc.matvec_t if transpose else orc.matvec
    with bipb.Surface(c, nv, a) as s:
        s.treecode(0.8, 4, 33)
        y = torch.full_like(_dev(U[0]), float("nan"))
        s.matvec(_dev(U[0]), y, precision=bipb.TREE32, transpose=transpose, med=med)
        y = y.cpu().numpy()
        ref = orc.treecode.matvec(c, nv, a, eps, kappa, U[0], 0.8, 4, 33, transpose=transpose)
        assert np.linalg.norm((y - ref) / scale) < 3e-6 * np.linalg.norm(ref / scale)
        assert np.abs(y - ref).max() < 2e-5 * np.abs(ref).max()
        for k in (4, 17):
            Y = torch.full_like(_dev(U[:k]), float("nan"))
            s.matvec(_dev(U[:k]), Y, precision=bipb.DF64, transpose=transpose, med=med)
            Y = Y.cpu().numpy()
            for r in (0, k - 1):
                ref = f(c, nv, a, eps, kappa, U[r])
                np.testing.assert_allclose(Y[r], ref, rtol=0, atol=2e-12 * np.abs(ref).max())
