"""The tensor cores truncate inside sums of 16 columns: over positive data that
leaves products a little low, by no more than the header says, and their
error is no larger than that of the row-ordered products."""
import numpy as np
import pytest
import scipy.sparse as sp
import torch

from paper_2009_07226_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def xct():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2009_07226_gb300 import xct as x
    return x


@pytest.mark.parametrize("kind", ["f16", "bf16"])
@pytest.mark.parametrize("S", [3, 8, 16, 64])
def test_mean_error_of_positive_sums(xct, kind, S):
    n, m, nd = 192, 160, 192
    rng = np.random.default_rng(S)
    mats, outs, vecs = [], {}, []
    for k in (n * n, m * nd):       # values that 16 bits hold, maximum 1
        v = torch.tensor(rng.uniform(0.25, 1, size=(S, k)), dtype=torch.float32)
        v = v.to(torch.float16 if kind == "f16" else torch.bfloat16).float()
        v[:, 0] = 1.0
        vecs.append(v)
    for rows_only in (False, True):
        with xct.Plan(n, m, nd, kind, cos_sin=inputs.angle_table(m), rows_only=rows_only) as p:
            if not mats:
                for what, shape in ((xct.XCT_EXPORT_A_STORED, (m * nd, n * n)),
                                    (xct.XCT_EXPORT_AT_STORED, (n * n, m * nd))):
                    rp, col, val = xct.xct_plan_export(p.handle, what)
                    mats.append(sp.csr_matrix((val, col, rp), shape=shape))
            outs[rows_only] = [p.project(vecs[0].reshape(S, n, n).cuda()), p.backproject(vecs[1].reshape(S, m, nd).cuda())]
    for i, mat in enumerate(mats):
        want = (mat @ vecs[i].double().numpy().T).T
        far, rms = {}, {}
        for rows_only in (False, True):
            got = outs[rows_only][i].cpu().double().numpy().reshape(S, -1)
            rel = ((got - want)[want > 1] / want[want > 1])
            # About 5 of a piece's 16 terms are entries of a row, each cut by
            # half of 2^-24 of the largest on average, against a sum of some
            # 3 times the largest: near 2^-24; twice that is allowed.  In rows,
            # roundings to nearest cancel.
            assert abs(rel.mean()) <= (2.0 ** -26 if rows_only else 2.0 ** -23), (rows_only, rel.mean())
            far[rows_only], rms[rows_only] = np.abs(rel).max(), np.sqrt((rel ** 2).mean())
        assert far[False] <= far[True] + 2.0 ** -22, far
        assert rms[False] <= rms[True], rms
