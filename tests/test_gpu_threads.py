"""Host threads that build and use plans of different sizes at the same time:
every call succeeds and gives what it gives alone."""
import threading

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


@pytest.mark.parametrize("kind", ["f16", "f32"])
def test_plans_of_different_sizes_built_at_once(xct, kind):
    # footprints and rows of a column that need from a few to over 100 KB of
    # a block's shared memory
    sizes = [(12, 10, 12, 3), (96, 140, 96, 9), (250, 60, 250, 20), (40, 1500, 40, 40)]
    data, want = [], []
    for n, m, nd, S in sizes:
        g = torch.Generator(device="cuda").manual_seed(n)
        x = torch.rand((S, n, n), device="cuda", generator=g)
        with xct.Plan(n, m, nd, kind, cos_sin=inputs.angle_table(m)) as p:
            y = p.project(x)
            data.append((x, y))
            want.append(p.backproject(y))
    torch.cuda.synchronize()
    errors = []

    def work(i):
        n, m, nd, S = sizes[i]
        x, y = data[i]
        stream = torch.cuda.Stream()
        try:
            with torch.cuda.stream(stream):
                for _ in range(12):
                    with xct.Plan(n, m, nd, kind, cos_sin=inputs.angle_table(m)) as p:
                        got, back = p.project(x), p.backproject(y)
                        stream.synchronize()
                    if not (torch.equal(got, y) and torch.equal(back, want[i])):
                        errors.append((i, "another result"))
        except Exception as e:
            errors.append((i, repr(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(sizes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:4]


def test_many_small_and_large_plans_built_at_once(xct):
    """Eight threads, 4400 builds: a block's footprint needs 1 KB of shared
    memory in some and over 100 KB in the others, rays 8 pixels apart."""
    errors = []

    def work(n, m, nd, spacing, builds):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(builds):
                try:
                    with xct.Plan(n, m, nd, "f16", cos_sin=inputs.angle_table(m), det_spacing=spacing):
                        pass
                except xct.XctError as e:
                    errors.append(str(e))

    threads = [threading.Thread(target=work, args=a)
               for a in [(12, 10, 12, 1.0, 800)] * 4 + [(360, 16, 45, 8.0, 300)] * 4]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, (len(errors), errors[:2])
