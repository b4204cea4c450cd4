"""Plans without octet layouts: products of 16-bit slices on the row layouts
(plain, narrow-tile, paired, wide-stage), which solves run on, against the
oracle's model of the 16-bit arithmetic, element by element."""
import numpy as np
import pytest
import torch

import oracle
from paper_2009_07226_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def xct():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2009_07226_gb300 import xct as x
    return x


def _matrices(n, m, nd, off):
    g = oracle.Geometry(n=n, m=m, nd=nd, cos_sin=inputs.angle_table(m), det_offset=off)
    a = oracle.siddon_csr(g)
    return g.table(), a, oracle.transpose(a)


# tiles of 8, 16, 32 and 64 slices, full and partly empty
@pytest.mark.parametrize("S", [3, 8, 16, 20, 32, 33, 64, 100])
@pytest.mark.parametrize("flags", [{}, {"narrow_tiles": True}, {"paired_rows": True}, {"few_slices": True},
                                   {"few_slices": True, "narrow_tiles": True, "paired_rows": True}],
                         ids=lambda f: "+".join(f) or "plain")
@pytest.mark.parametrize("kind", ["f16", "bf16"])
@pytest.mark.parametrize("n,m,nd,off", [(64, 96, 64, 0.0), (37, 23, 41, -0.4)])
def test_row_products_vs_oracle_model(xct, kind, flags, S, n, m, nd, off):
    cs, a, at = _matrices(n, m, nd, off)
    rng = np.random.default_rng(n + 7 * S)
    mag = 10.0 ** rng.uniform(-3, 3, size=(S, 1))
    x = torch.tensor(rng.uniform(-1, 1, size=(S, n * n)) * mag, dtype=torch.float32)
    y = torch.tensor(rng.uniform(-1, 1, size=(S, m * nd)) * mag, dtype=torch.float32)
    with xct.Plan(n, m, nd, kind, cos_sin=cs, det_offset=off, rows_only=True, **flags) as p:
        st = p.stats()
        assert st["bytes_a_octets"] == st["bytes_at_octets"] == 0
        yo = torch.full((S, m, nd), float("nan"), device="cuda")
        rows, xo = yo.clone(), torch.full((S, n, n), float("nan"), device="cuda")
        p.project(x.reshape(S, n, n).cuda(), out=yo)
        p.backproject(y.reshape(S, m, nd).cuda(), out=xo)
        xct.xct_project_rows(p.handle, x.cuda(), rows, S)
        torch.cuda.synchronize()
        xct.xct_plan_check(p.handle)
    assert torch.equal(yo, rows)
    for got, mat, v in ((yo, a, x), (xo, at, y)):
        v = v.double().numpy()
        absm = oracle.CSR(mat.nrow, mat.ncol, mat.rowptr, mat.col, np.abs(mat.val))
        err = np.abs(got.cpu().double().numpy().reshape(S, -1) - oracle.mixed_project(mat, v, kind))
        # FP32 sums of under 2 n terms, the bar of the product tests
        assert np.all(err <= 1e-5 * oracle.project(absm, np.abs(v)) + 1e-30)


def test_paired_and_plain_rows_agree(xct):
    """64 slices on paired and on plain layouts: the same products in another
    order, and not bit for bit the same (they are two kernels' results)."""
    n, m, nd, S = 64, 96, 64, 64
    g = torch.Generator(device="cuda").manual_seed(6)
    x = torch.rand((S, n, n), device="cuda", generator=g)
    cs = inputs.angle_table(m)
    with xct.Plan(n, m, nd, "f16", cos_sin=cs, paired_rows=True, rows_only=True) as pp, \
            xct.Plan(n, m, nd, "f16", cos_sin=cs, rows_only=True) as ps:
        y1, y0 = pp.project(x), ps.project(x)
        z1, z0 = pp.backproject(y0), ps.backproject(y0)
    for u, v in ((y1, y0), (z1, z0)):
        assert float((u - v).norm() / v.norm()) <= 1e-6 and not torch.equal(u, v)


@pytest.mark.parametrize("flags", [{}, {"narrow_tiles": True}, {"paired_rows": True}, {"few_slices": True}])
def test_solves_do_not_depend_on_octets(xct, flags):
    n, m, nd = 64, 96, 64
    g = torch.Generator(device="cuda").manual_seed(8)
    cs = inputs.angle_table(m)
    with xct.Plan(n, m, nd, "f16", cos_sin=cs, **flags) as p, \
            xct.Plan(n, m, nd, "f16", cos_sin=cs, rows_only=True, **flags) as q:
        for S in (3, 20, 64):
            y = torch.rand((S, m, nd), device="cuda", generator=g)
            (x1, l1), (x2, l2) = p.cgls(y, 4, resid=True), q.cgls(y, 4, resid=True)
            assert torch.equal(x1, x2) and torch.equal(l1, l2)


@pytest.mark.parametrize("flags", ["XCT_PLAN_PAIRED_ROWS", "XCT_PLAN_FEW_SLICES"])
def test_allocation_failures_in_the_last_layouts(xct, flags):
    """Without octets the paired or wide-stage layouts are built last: a
    failure in their build is reported, and nothing is leaked."""
    n, m, nd = 48, 60, 50
    geom = xct.make_geometry(n, m, nd, inputs.angle_table(m))
    fl = getattr(xct, flags) | xct.XCT_PLAN_ROWS_ONLY
    live, state = {}, {"count": 0, "ok": None}

    def alloc(nbytes, stream):
        state["count"] += 1
        if state["ok"] is not None and state["count"] > state["ok"]:
            return 0
        ptr = torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device(), stream or 0)
        live[ptr] = nbytes
        return ptr

    def release(ptr, nbytes, stream):
        assert live.pop(ptr) == nbytes
        torch.cuda.caching_allocator_delete(ptr)

    xct.xct_set_allocator(alloc, release)
    try:
        xct.xct_free(xct.xct_plan(geom, "f16", xct.XCT_PLAN_ROWS_ONLY))
        plain = state["count"]
        state["count"] = 0
        xct.xct_free(xct.xct_plan(geom, "f16", fl))
        total = state["count"]
        assert total > plain
        for ok in range(plain, total):
            state.update(count=0, ok=ok)
            with pytest.raises(xct.XctError) as e:
                xct.xct_plan(geom, "f16", fl)
            assert e.value.status == xct.XCT_ERR_OOM
            torch.cuda.synchronize()
            assert live == {}, ok
    finally:
        xct.xct_set_allocator(None, None)
