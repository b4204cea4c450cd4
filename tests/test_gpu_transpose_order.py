"""Rays along grid lines hold some pixels twice; the transpose keeps such a
ray's two entries in the order in which the ray meets them, in every build of
the plan."""
import numpy as np
import pytest
import torch

from paper_2009_07226_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def xct():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2009_07226_gb300 import xct as x
    return x


def _transposed(rowptr, col, val, ncol):
    """The columns of a CSR matrix, each in the order of its rows."""
    at = np.argsort(col, kind="stable")
    rows = np.repeat(np.arange(len(rowptr) - 1), np.diff(rowptr))
    return np.searchsorted(col[at], np.arange(ncol + 1)), rows[at], val[at]


def _repeats(rowptr, col, val):
    """Places whose entry has the row and column of the one before, and
    another value."""
    rows = np.repeat(np.arange(len(rowptr) - 1), np.diff(rowptr))
    return np.nonzero((np.diff(col) == 0) & (np.diff(rows) == 0) & (np.diff(val) != 0))[0] + 1


# At 90 degrees (the table's cosine there is 6e-17, not 0) rays lie along grid
# lines: of an odd grid through its bins at half integers, and of an even grid
# with the bins 4e-16 from the integers.  Each holds one pixel in two pieces
# (0.5 and 0.5 but for rounding; 0.75 and 0.25).
@pytest.mark.parametrize("kind", ["f32", "f16"])
@pytest.mark.parametrize("n,m,nd,off", [(33, 4, 34, 0.0), (32, 2, 33, 4.4e-16)])
def test_repeated_entries_keep_their_order(xct, kind, n, m, nd, off):
    g = torch.Generator(device="cuda").manual_seed(n)
    y = torch.rand((5, m, nd), device="cuda", generator=g)
    backs = []
    for _ in range(2):
        with xct.Plan(n, m, nd, kind, cos_sin=inputs.angle_table(m), det_offset=off,
                      keep_f64=True) as p:
            rp, col, val = xct.xct_plan_export(p.handle, xct.XCT_EXPORT_A_F64)
            trp, tcol, tval = xct.xct_plan_export(p.handle, xct.XCT_EXPORT_AT_F64)
            backs.append(p.backproject(y).cpu().double().reshape(5, -1))
        assert len(_repeats(rp, col, val)) > 0
        want = _transposed(rp, col, val, n * n)
        assert np.array_equal(trp, want[0]) and np.array_equal(tcol, want[1]) and np.array_equal(tval, want[2])
        # (two entries exchanged would be seen)
        k = _repeats(trp, tcol, tval)[0]
        tval[[k - 1, k]] = tval[[k, k - 1]]
        assert not np.array_equal(tval, want[2])
    assert torch.equal(backs[0], backs[1])
    a = np.zeros((m * nd, n * n))
    np.add.at(a, (np.repeat(np.arange(m * nd), np.diff(rp)), col), val)
    # the bound of the product tests: rounding to the storage, then FP32 sums
    v = y.cpu().double().numpy().reshape(5, -1)
    assert np.all(np.abs(backs[0].numpy() - v @ a) <= (1e-5 if kind == "f32" else 2.0 ** -9) * (v @ a) + 1e-30)
