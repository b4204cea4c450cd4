"""A call that the launch limits refuse fails alone: the calls after it, the
library's and torch's, succeed."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def xct():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2009_07226_gb300 import xct as x
    return x


@pytest.mark.parametrize("kind,tile", [("f32", 32), ("f16", 64)])
def test_too_many_slice_tiles(xct, kind, tile):
    """A grid has at most 65535 slice tiles."""
    x = torch.rand((4, 1, 1), device="cuda")
    with xct.Plan(1, 1, 1, kind) as p:
        want = p.project(x)
        with pytest.raises(xct.XctError) as e:
            p.project(torch.zeros((65535 * tile + 1, 1, 1), device="cuda"))
        assert e.value.status == xct.XCT_ERR_CUDA
        assert torch.equal(p.project(x) * 1.0, want)
        torch.cuda.synchronize()
