"""The library's scratch pool gives its memory back: to an allocation that
would fail without it, and when no plan is left."""
import pytest
import torch

from paper_2009_07226_gb300 import inputs

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module")
def xct():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2009_07226_gb300 import xct as x
    return x


def _free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _fill(leave):
    """Takes the device's free memory but for `leave` bytes."""
    return torch.empty(_free() - leave, dtype=torch.uint8, device="cuda")


def _plan(xct, n, m, kind="f32"):
    return xct.Plan(n, m, n, kind, cos_sin=inputs.angle_table(m))


def test_idle_scratch_makes_room_for_a_plan(xct):
    n, m = 256, 384
    with _plan(xct, n, m):                     # modules loaded; about what it keeps
        with_one = _free()
    kept = _free() - with_one
    assert kept > 300 * MB
    with _plan(xct, 512, 8) as p:
        x = torch.ones((2048, 512, 512), device="cuda")
        want = p.project(x)                    # 2 GiB of scratch
        del x
        hold = _fill(kept // 2)
        with _plan(xct, n, m) as q:            # fits only with the pool's memory
            img = torch.rand((2, n, n), device="cuda")
            y = q.project(img)
            assert torch.isfinite(y).all()
        del hold
        again = p.project(torch.ones((2048, 512, 512), device="cuda"))
        assert torch.equal(again, want)


def test_a_failed_build_leaves_nothing_mapped(xct):
    with _plan(xct, 64, 64):
        pass
    free = _free()
    hold = _fill(1500 * MB)
    with pytest.raises(xct.XctError) as e:
        _plan(xct, 512, 768)                   # needs over 4 GB
    assert e.value.status == xct.XCT_ERR_OOM
    del hold
    assert _free() > free - 64 * MB
    with _plan(xct, 64, 64) as p:              # and the library works on
        assert torch.isfinite(p.project(torch.rand((3, 64, 64), device="cuda"))).all()
