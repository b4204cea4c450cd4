"""A product whose bounded waits run out leaves nothing in flight behind it:
products that run right after it on the stream, in the shared memory that it
gave up, give the results that they give alone."""
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


# a few stages in all (they fit the descriptor slots, so that no request is
# waited for), and many
@pytest.mark.parametrize("kind", ["f16", "f32"])   # octet and row products
@pytest.mark.parametrize("n,m,nd", [(24, 24, 24), (96, 144, 100)])
def test_products_right_after_one_that_gave_up(xct, kind, n, m, nd):
    S = 64
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.rand((S, n, n), device="cuda", generator=g)
    x2 = torch.rand((S, 128, 128), device="cuda", generator=g)
    with xct.Plan(n, m, nd, kind, cos_sin=inputs.angle_table(m)) as p, \
            xct.Plan(128, 160, 128, kind, cos_sin=inputs.angle_table(160)) as q:
        ref, ref2 = p.project(x), q.project(x2)
        torch.cuda.synchronize()
        for _ in range(20):
            prev = xct.xct_set_wait_limit(0)
            p.project(x)                      # gives up, wholly or in part
            assert xct.xct_set_wait_limit(prev) == 0
            got, got2 = p.project(x), q.project(x2)
            torch.cuda.synchronize()
            try:
                xct.xct_plan_check(p.handle)
            except xct.XctError as e:
                assert e.status == xct.XCT_ERR_TIMEOUT
            xct.xct_plan_check(q.handle)
            assert torch.equal(got, ref) and torch.equal(got2, ref2)
