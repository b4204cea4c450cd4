"""FP64 products and solves of few slices: every width of the few-slice form
and the sizes around them, against the oracle's FP64 matrix."""
import numpy as np
import pytest
import torch

import oracle
from paper_2009_07226_gb300 import inputs

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def xct():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2009_07226_gb300 import xct as x
    return x


@pytest.mark.parametrize("S", [1, 2, 3, 4, 5, 8, 9, 16, 17, 31, 64 + 2, 64 + 9])
@pytest.mark.parametrize("n,m,nd,off", [(37, 23, 41, -0.4), (96, 70, 100, 0.25), (9, 7, 30, 0.5)])
def test_products_within_summation_bound(xct, n, m, nd, off, S):
    g = oracle.Geometry(n=n, m=m, nd=nd, cos_sin=inputs.angle_table(m), det_offset=off)
    a = oracle.siddon_csr(g)
    rng = np.random.default_rng(n + S)
    x, y = rng.uniform(-1, 1, size=(S, n * n)), rng.uniform(-1, 1, size=(S, m * nd))
    with xct.Plan(n, m, nd, "f32", cos_sin=g.table(), det_offset=off, keep_f64=True) as p:
        yo = torch.full((S, m, nd), float("nan"), dtype=torch.float64, device="cuda")
        xo = torch.full((S, n, n), float("nan"), dtype=torch.float64, device="cuda")
        p.project_f64(torch.tensor(x.reshape(S, n, n), device="cuda"), out=yo)
        p.backproject_f64(torch.tensor(y.reshape(S, m, nd), device="cuda"), out=xo)
        torch.cuda.synchronize()
    for got, mat, v in ((yo, a, x), (xo, oracle.transpose(a), y)):
        k = (int(np.diff(mat.rowptr).max()) + 1) * U
        bound = 2 * k / (1 - k) * oracle.project(
            oracle.CSR(mat.nrow, mat.ncol, mat.rowptr, mat.col, np.abs(mat.val)), np.abs(v))
        err = np.abs(got.cpu().numpy().reshape(S, -1) - oracle.project(mat, v))
        assert np.all(err <= bound + 1e-300)


@pytest.mark.parametrize("S", [2, 4, 8, 16, 17])
def test_solves_equal_their_slices(xct, S):
    """The norms that the product leaves: slices solved together as alone."""
    n, m, nd = 64, 90, 64
    g = torch.Generator(device="cuda").manual_seed(S)
    with xct.Plan(n, m, nd, "f32", cos_sin=inputs.angle_table(m), keep_f64=True) as p:
        b = p.project_f64(torch.rand((S, n, n), dtype=torch.float64, device="cuda", generator=g))
        x, log = p.cgls_f64(b, 3, resid=True)
        for s in range(S):
            x1, log1 = p.cgls_f64(b[s:s + 1].contiguous(), 3, resid=True)
            # 3 iterations, before rounding is amplified: the bar of the solve's test
            assert float((x[s] - x1[0]).norm() / x1.norm()) <= 1e-11
            assert torch.allclose(log[:, s], log1[:, 0], rtol=1e-11, atol=0)
