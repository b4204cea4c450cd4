"""What octet layouts cost and what a plan does without them: their bytes are
reported, and a plan whose memory did not suffice for them gives the products
of its row layouts."""
import numpy as np
import pytest
import torch

from paper_2009_07226_gb300 import inputs

pytestmark = pytest.mark.gpu

N, M, ND, S = 48, 60, 50, 20


@pytest.fixture(scope="module")
def xct():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2009_07226_gb300 import xct as x
    return x


class _Budget:
    """Allocator callbacks that serve `ok` allocations, then fail (None:
    never)."""

    def __init__(self, ok=None):
        self.ok, self.count, self.live = ok, 0, {}

    def alloc(self, nbytes, stream):
        self.count += 1
        if self.ok is not None and self.count > self.ok:
            return 0
        ptr = torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device(), stream or 0)
        self.live[ptr] = nbytes
        return ptr

    def release(self, ptr, nbytes, stream):
        assert self.live.pop(ptr) == nbytes
        torch.cuda.caching_allocator_delete(ptr)


@pytest.mark.parametrize("kind", ["f32", "f16a"])
def test_plans_of_fp32_slices_hold_no_octets(xct, kind):
    with xct.Plan(N, M, ND, kind, cos_sin=inputs.angle_table(M)) as p:
        st = p.stats()
    assert st["bytes_a_octets"] == st["bytes_at_octets"] == 0


@pytest.mark.parametrize("kind", ["f16", "bf16"])
def test_plans_that_fell_back_from_octets(xct, kind):
    g = torch.Generator(device="cuda").manual_seed(7)
    x = torch.rand((S, N, N), device="cuda", generator=g)
    y = torch.rand((S, M, ND), device="cuda", generator=g)
    geom = xct.make_geometry(N, M, ND, inputs.angle_table(M))
    count = _Budget()
    xct.xct_set_allocator(count.alloc, count.release)
    try:
        h = xct.xct_plan(geom, kind)
        torch.cuda.synchronize()
        full = xct.xct_plan_stats(h)
        kept = sum(count.live.values())
        xct.xct_free(h)
    finally:
        xct.xct_set_allocator(None, None)
    assert full["bytes_a_octets"] > 288 * full["nnz"] / 128 < full["bytes_at_octets"]
    seen = set()
    for ok in range(count.count - 1, 0, -1):
        budget = _Budget(ok)
        xct.xct_set_allocator(budget.alloc, budget.release)
        try:
            try:
                h = xct.xct_plan(geom, kind)
            except xct.XctError as e:
                assert e.status == xct.XCT_ERR_OOM
                break                            # the plan's other parts need the rest
            st = xct.xct_plan_stats(h)
            state = (st["bytes_a_octets"] > 0, st["bytes_at_octets"] > 0)
            if state not in seen:
                seen.add(state)
                # the reported bytes are what the layouts took
                assert kept - sum(budget.live.values()) == sum(
                    full[k] - st[k] for k in ("bytes_a_octets", "bytes_at_octets"))
                budget.ok = None
                got, rows = torch.empty_like(y), torch.empty_like(y)
                back = torch.empty_like(x)
                xct.xct_project(h, x, got, S)
                xct.xct_project_rows(h, x, rows, S)
                xct.xct_backproject(h, y, back, S)
                torch.cuda.synchronize()
                xct.xct_plan_check(h)
                if not state[0]:
                    assert torch.equal(got, rows)
                for out, what, v in ((got, xct.XCT_EXPORT_A_STORED, x), (back, xct.XCT_EXPORT_AT_STORED, y)):
                    rp, col, val = xct.xct_plan_export(h, what)
                    a = np.zeros((len(rp) - 1, v[0].numel()))
                    np.add.at(a, (np.repeat(np.arange(len(rp) - 1), np.diff(rp)), col), val)
                    v = v.cpu().double().numpy().reshape(S, -1)
                    # the vectors' rounding to 16 bits, then FP32 sums
                    eps = 2.0 ** (-11 if kind == "f16" else -8) + 1e-5
                    err = np.abs(out.cpu().double().numpy().reshape(S, -1) - v @ a.T)
                    assert np.all(err <= eps * (v @ a.T) + 1e-6)
            xct.xct_free(h)
        finally:
            xct.xct_set_allocator(None, None)
        torch.cuda.synchronize()
        assert budget.live == {}
    assert {(True, False), (False, False)} <= seen


# ---------------------------------------------------------------------------
# memory that runs out after the plan was built
# ---------------------------------------------------------------------------

MB = 1 << 20


def _free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _kept(xct, n, m):
    """Bytes that a binary16 plan of n^2 x m angles keeps."""
    b = _Budget()
    xct.xct_set_allocator(b.alloc, b.release)
    try:
        with xct.Plan(n, m, n, "f16", cos_sin=inputs.angle_table(m)):
            torch.cuda.synchronize()
            return sum(b.live.values())
    finally:
        xct.xct_set_allocator(None, None)


def _solve_at_the_limit(xct, p, S, idle, iters=2):
    """CGLS of S slices with less memory free (beside the `idle` bytes of the
    library's scratch pool) than its working memory needs, and enough with
    the plan's octet layouts; returns (y, x, status)."""
    n, m, nd = p.n, p.m, p.nd
    g = torch.Generator(device="cuda").manual_seed(1)
    y = torch.rand((S, m, nd), device="cuda", generator=g)
    x = torch.empty((S, n, n), device="cuda")
    st = p.stats()
    octets = st["bytes_a_octets"] + st["bytes_at_octets"]
    scratch = S * (12 * n * n + 8 * m * nd + 2 * (n * n + m * nd))
    assert octets > 400 * MB and scratch > idle + octets
    hold = torch.empty(_free() - (scratch - octets // 2 - idle), dtype=torch.uint8, device="cuda")
    try:
        xct.xct_cgls(p.handle, y, x, S, iters)
        status = xct.XCT_OK
    except xct.XctError as e:
        status = e.status
    del hold
    torch.cuda.empty_cache()
    return y, x, status


def test_a_solve_takes_the_octets_memory(xct):
    n, m, S = 256, 384, 2048
    kept = _kept(xct, n, m)
    img = torch.rand((20, n, n), device="cuda")
    before = _free()
    with xct.Plan(n, m, n, "f16", cos_sin=inputs.angle_table(m)) as p:
        want = p.project(img)
        y, x, status = _solve_at_the_limit(xct, p, S, before - _free() - kept)
        assert status == xct.XCT_OK
        assert p.stats()["bytes_a_octets"] == p.stats()["bytes_at_octets"] == 0
        got = p.project(img)
        assert float((got - want).norm() / want.norm()) <= 1e-6
        with xct.Plan(n, m, n, "f16", cos_sin=inputs.angle_table(m), rows_only=True) as q:
            assert torch.equal(x, q.cgls(y, 2))
            assert torch.equal(got, q.project(img))
            assert torch.equal(p.backproject(got), q.backproject(got))


def test_captured_products_keep_their_octets(xct):
    n, m, S = 256, 384, 2048
    kept = _kept(xct, n, m)
    img = torch.rand((20, n, n), device="cuda")
    before = _free()
    with xct.Plan(n, m, n, "f16", cos_sin=inputs.angle_table(m)) as p:
        want = p.project(img)
        idle = before - _free() - kept
        out = torch.empty_like(want)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            p.project(img, out=out)
        _, _, status = _solve_at_the_limit(xct, p, S, idle)
        assert status == xct.XCT_ERR_OOM
        assert p.stats()["bytes_a_octets"] > 0
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want)
        del graph


def test_building_octets_takes_no_other_plans(xct):
    """A second plan whose octets do not fit goes without; the first keeps
    its own."""
    n, m = 256, 384
    cs = inputs.angle_table(m)
    with xct.Plan(n, m, n, "f16", cos_sin=cs) as p:
        st = p.stats()
        # less and less room (the build's working memory lies idle in the
        # scratch pool since the first build)
        room = st["bytes_a"] + st["bytes_at"] + st["bytes_a_octets"]
        for leave in range(room, 0, -32 * MB):
            hold = torch.empty(_free() - leave, dtype=torch.uint8, device="cuda")
            with xct.Plan(n, m, n, "f16", cos_sin=cs) as q:
                sq = q.stats()
            del hold
            if sq["bytes_a_octets"] * sq["bytes_at_octets"] == 0:
                break
        assert sq["bytes_a_octets"] * sq["bytes_at_octets"] == 0
        assert p.stats() == st
