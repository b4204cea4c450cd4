"""Matrix-free projection on a large grid: the lengths of rays through tens of
thousands of grid lines against an FP64 trace, at their shortest pieces, where
an error of the crossings shows."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

N, ND, SP = 16384, 7, 1500.3


@pytest.fixture(scope="module")
def xct():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2009_07226_gb300 import xct as x
    return x


def _row(c, s, t, min_seg=1e-9):
    """Pixels and lengths of one ray, every crossing on its own in FP64."""
    h = N / 2
    ends, cross = [], []
    for p, d in ((t * c, -s), (t * s, c)):
        a = (np.arange(N + 1) - h - p) / d
        ends.append((a.min(), a.max()))
        cross.append(a)
    lo, hi = max(e[0] for e in ends), min(e[1] for e in ends)
    a = np.concatenate(cross)
    a = np.sort(np.concatenate([[lo, hi], a[(a > lo) & (a < hi)]]))
    ln, mid = np.diff(a), 0.5 * (a[1:] + a[:-1])
    ix = np.clip(np.floor(t * c - mid * s + h), 0, N - 1).astype(np.int64)
    iy = np.clip(np.floor(t * s + mid * c + h), 0, N - 1).astype(np.int64)
    keep = ln >= min_seg
    return (iy * N + ix)[keep], ln[keep]


@pytest.mark.parametrize("S", [1, 3])
def test_short_pieces_of_long_rays(xct, S):
    th = np.radians([33.0, 44.9, 45.3, 52.0, 128.0, 135.1, 146.0])
    cs = np.stack([np.cos(th), np.sin(th)], 1)
    rows, short = [], []
    for c, s in cs:
        for k in range(ND):
            pix, ln = _row(c, s, (k - 0.5 * (ND - 1)) * SP)
            rows.append((pix, ln))
            at = np.argsort(ln)[:1]
            short.append(pix[at[ln[at] > 1e-7]])
    marked = np.unique(np.concatenate(short))
    x = torch.zeros((S, N * N), device="cuda")
    x[S - 1, torch.tensor(marked, device="cuda")] = 1.0
    with xct.Plan(N, len(th), ND, "f32", cos_sin=cs, det_spacing=SP) as p:
        y = torch.empty((S, len(th), ND), device="cuda")
        xct.xct_project_matfree(p.handle, x, y, S)
        torch.cuda.synchronize()
    got = y[S - 1].double().cpu().numpy().ravel()
    checked = 0
    for r, (pix, ln) in enumerate(rows):
        ln = ln[np.isin(pix, marked)]
        if ln.sum() > 1e-2:
            continue                       # crosses another ray's pixel widely
        checked += 1
        d = np.abs(cs[r // ND]).min()
        # a crossing's FP64 difference and quotient, in both traces, at both
        # ends of a piece; the FP32 length; the FP32 sum
        bound = len(ln) * 8 * 2.0 ** -53 * N / d + (1 + len(ln)) * 2.0 ** -24 * ln.sum()
        assert abs(got[r] - ln.sum()) <= bound, (r, got[r] - ln.sum(), bound, ln)
    assert checked > 30
    assert float(y[:S - 1].abs().sum()) == 0.0
