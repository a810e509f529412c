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
