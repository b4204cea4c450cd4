"""Matrix-free projection with little working memory: in passes over rays and
slices, without the interleaved copy of the slices, and without the rays'
set-up."""
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


def _project(xct, p, x):
    y = torch.full((x.shape[0], p.m, p.nd), float("nan"), device="cuda")
    xct.xct_project_matfree(p.handle, x, y, x.shape[0])
    return y


# 64 x 96 rays need 442 KB of set-up, 24 slices of 96^2 885 KB
@pytest.mark.parametrize("most", [700 << 10, 64 << 10])
@pytest.mark.parametrize("S", [1, 2, 3, 24])
def test_without_room_for_working_memory(xct, S, most):
    n, m, nd = 96, 96, 64
    g = torch.Generator(device="cuda").manual_seed(S)
    x = torch.rand((S, n, n), device="cuda", generator=g)
    refused = []

    def alloc(nbytes, stream):
        if nbytes > most:
            refused.append(nbytes)
            return 0
        return torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device(), stream or 0)

    with xct.Plan(n, m, nd, "f32", cos_sin=inputs.angle_table(m)) as p:
        want = _project(xct, p, x)
        xct.xct_set_allocator(alloc, lambda ptr, nbytes, stream: torch.cuda.caching_allocator_delete(ptr))
        try:
            got = _project(xct, p, x)
        finally:
            xct.xct_set_allocator(None, None)
    assert bool(refused) == (most < 442 << 10 or S == 24)
    # the same lengths but for their rounding, in the same order
    assert float((got - want).abs().max()) <= 2.0 ** -22 * float(want.abs().max())


def test_slices_in_several_passes(xct):
    """80 slices of 2048^2: ten tiles, eight of them fill the copy's 1 GiB."""
    n, m, nd, S = 2048, 4, 70, 80
    g = torch.Generator(device="cuda").manual_seed(2)
    x = torch.rand((S, n, n), device="cuda", generator=g)
    with xct.Plan(n, m, nd, "f32", cos_sin=inputs.angle_table(m)) as p:
        got = _project(xct, p, x)
        for s in range(0, S, 8):
            assert torch.equal(got[s:s + 8], _project(xct, p, x[s:s + 8]))


@pytest.mark.parametrize("S", [1, 3])
def test_rays_in_several_batches(xct, S):
    """4,202,000 rays (most of them miss the grid), of which 4,194,304 fill a
    batch."""
    n, m, nd = 32, 2101, 2000
    g = torch.Generator(device="cuda").manual_seed(S)
    x = torch.rand((S, n, n), device="cuda", generator=g)
    with xct.Plan(n, m, nd, "f32", cos_sin=inputs.angle_table(m)) as p:
        got, want = _project(xct, p, x), p.project(x)
    # FP32 sums of at most 2 n + 1 terms in two orders
    assert float((got - want).abs().max()) <= 2 * (2 * n + 1) * 2.0 ** -24 * n * 1.5
    assert float(want[:, -1].abs().max()) > 0
