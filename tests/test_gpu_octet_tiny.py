"""Slices whose largest value is 2^-128 or less have no finite scale: their
staged values are infinities and NaN, which reach exactly the rays that cross
them, on octet layouts as on row layouts."""
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


@pytest.mark.parametrize("kind", ["f16", "bf16"])
@pytest.mark.parametrize("S", [9, 64])
def test_tiny_slices_as_on_rows(xct, kind, S):
    n, m, nd = 48, 60, 81          # some rays miss the grid
    g = torch.Generator(device="cuda").manual_seed(S)
    x = torch.rand((S, n, n), device="cuda", generator=g)
    for s, top in ((1, 2.0 ** -128), (4, 1e-42), (8, 2.0 ** -127)):
        x[s] = top * (x[s] < 0.5)
    with xct.Plan(n, m, nd, kind, cos_sin=inputs.angle_table(m)) as p:
        got = p.project(x)
        want = torch.empty_like(got)
        xct.xct_project_rows(p.handle, x, want, S)
        torch.cuda.synchronize()
    assert torch.equal(torch.isnan(got), torch.isnan(want))
    assert torch.equal(torch.isinf(got), torch.isinf(want))
    assert torch.isnan(want[1]).any() and (want[1] == 0).any() and torch.isfinite(want[8]).all()
    fine = [s for s in range(S) if s not in (1, 4)]
    assert torch.isfinite(got[fine]).all()
