"""Products of 16-bit slices on octet layouts (tensor cores): against the
stored 16-bit matrix times 16-bit-exact inputs in float64, at the edges of
the layout -- blocks and octets past the matrix, columns past the last group
of 8, tiles other than 8 x 8, rays that hold a pixel twice, every tile width
and partly empty ones -- and against the row-ordered products where a slice
holds infinities and NaN."""
import numpy as np
import pytest
import torch

from paper_2009_07226_gb300 import inputs

pytestmark = pytest.mark.gpu

# n, angles, bins, detector offset, Hilbert tile.  64 x 64 with 65 bins: the
# rays at 90 degrees run along grid lines and hold some pixels twice.
GEOMS = [(1, 1, 1, 0.0, 0), (5, 3, 7, 0.3, 0), (37, 23, 41, -0.4, 0), (64, 96, 65, 0.0, 0),
         (64, 48, 64, 0.0, 16), (100, 33, 96, 0.0, 3)]


@pytest.fixture(scope="module")
def xct():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2009_07226_gb300 import xct as x
    return x


def _vectors(rng, S, k, kind):
    """Values that 16 bits hold exactly, with maximum 1 in every slice."""
    v = torch.tensor(rng.uniform(-1, 1, size=(S, k)), dtype=torch.float32)
    v = v.to(torch.float16 if kind == "f16" else torch.bfloat16).float()
    v[:, 0] = 1.0
    return v


def _stored(xct, plan, what, shape):
    """Dense float64 matrix (repeated entries added)."""
    rp, col, val = xct.xct_plan_export(plan.handle, what)
    a = np.zeros(shape)
    np.add.at(a, (np.repeat(np.arange(shape[0]), np.diff(rp)), col), val)
    return a


@pytest.mark.parametrize("kind", ["f16", "bf16"])
@pytest.mark.parametrize("n,m,nd,off,tile", GEOMS)
def test_octet_products_equal_the_stored_matrix(xct, kind, n, m, nd, off, tile):
    rng = np.random.default_rng(n + m)
    with xct.Plan(n, m, nd, kind, cos_sin=inputs.angle_table(m), det_offset=off, hilbert_tile=tile) as p:
        A = _stored(xct, p, xct.XCT_EXPORT_A_STORED, (m * nd, n * n))
        AT = _stored(xct, p, xct.XCT_EXPORT_AT_STORED, (n * n, m * nd))
        for S in (1, 8, 9, 17, 33, 64, 65, 100):
            x, y = _vectors(rng, S, n * n, kind), _vectors(rng, S, m * nd, kind)
            yo = torch.full((S, m, nd), float("nan"), device="cuda")
            xo = torch.full((S, n, n), float("nan"), device="cuda")
            p.project(x.reshape(S, n, n).cuda(), out=yo)
            p.backproject(y.reshape(S, m, nd).cuda(), out=xo)
            torch.cuda.synchronize()
            xct.xct_plan_check(p.handle)
            for got, mat, v in ((yo, A, x), (xo, AT, y)):
                got, v = got.cpu().double().numpy().reshape(S, -1), v.double().numpy()
                want, bound = v @ mat.T, np.abs(v) @ np.abs(mat).T
                assert np.all(np.abs(got - want) <= 1e-5 * bound + 1e-30), (S, mat.shape)


@pytest.mark.parametrize("kind", ["f16", "bf16"])
@pytest.mark.parametrize("S", [9, 20, 64])
def test_octet_products_keep_infinities_and_nan_to_their_rays(xct, kind, S):
    """An infinity and a NaN in two slices reach exactly the rays that cross
    them (a chunk's unused cells hold zeros, and 0 times either is NaN)."""
    n, m, nd = 48, 60, 47
    rng = np.random.default_rng(S)
    x = _vectors(rng, S, n * n, kind).reshape(S, n, n)
    x[1, 20, 13] = float("inf")
    x[min(8, S - 1), 31, 40] = float("nan")
    with xct.Plan(n, m, nd, kind, cos_sin=inputs.angle_table(m)) as p:
        got = p.project(x.cuda())
        want = torch.empty_like(got)
        xct.xct_project_rows(p.handle, x.cuda(), want, S)
        torch.cuda.synchronize()
    assert torch.equal(torch.isnan(got), torch.isnan(want))
    assert torch.equal(torch.isinf(got), torch.isinf(want))
    fine = torch.isfinite(want)
    assert 0 < int((~fine).sum()) < fine.numel() // 4
    # FP32 sums of at most 2 n + 1 terms of at most sqrt(2)
    assert float((got - want)[fine].abs().max()) <= 2 * (2 * n + 1) * 2.0 ** -24 * (2 * n + 1) * 1.5


def test_octet_product_unaligned_buffers(xct):
    """Inputs and outputs that start 4 bytes past an aligned address."""
    n, m, nd, S = 40, 50, 44, 20
    gen = torch.Generator().manual_seed(3)
    x = torch.rand((S, n, n), generator=gen).cuda()
    with xct.Plan(n, m, nd, "f16", cos_sin=inputs.angle_table(m)) as p:
        want = p.project(x)
        xs = torch.empty(x.numel() + 1, device="cuda")[1:].view_as(x).copy_(x)
        ys = torch.full((want.numel() + 1,), float("nan"), device="cuda")[1:].view_as(want)
        xct.xct_project(p.handle, xs, ys, S)
        torch.cuda.synchronize()
    assert torch.equal(ys, want)


def test_octet_product_of_wide_footprints(xct):
    """Rays 8 pixels apart: a block of 128 rays crosses more groups of columns
    than are ordered along them (8192), and the back projection's blocks
    fewer."""
    import scipy.sparse as sp
    n, m, nd, S = 720, 16, 90, 9
    rng = np.random.default_rng(5)
    with xct.Plan(n, m, nd, "f16", cos_sin=inputs.angle_table(m), det_spacing=8.0) as p:
        mats = [sp.csr_matrix((v, c, r), shape=s) for (r, c, v), s in
                ((xct.xct_plan_export(p.handle, xct.XCT_EXPORT_A_STORED), (m * nd, n * n)),
                 (xct.xct_plan_export(p.handle, xct.XCT_EXPORT_AT_STORED), (n * n, m * nd)))]
        x, y = _vectors(rng, S, n * n, "f16"), _vectors(rng, S, m * nd, "f16")
        got = [p.project(x.reshape(S, n, n).cuda()), p.backproject(y.reshape(S, m, nd).cuda())]
    # the groups (4 x 2 pixels) of one Hilbert tile of rays, half a block
    c = np.concatenate([mats[0][k * nd + 40:k * nd + 48].indices for k in range(8)])
    assert len(np.unique(c // n // 2 * (n // 4) + c % n // 4)) > 8192
    for g, mat, v in zip(got, mats, (x, y)):
        g, v = g.cpu().double().numpy().reshape(S, -1), v.double().numpy()
        assert np.all(np.abs(g - (mat @ v.T).T) <= 1e-5 * (abs(mat) @ np.abs(v).T).T + 1e-30)
