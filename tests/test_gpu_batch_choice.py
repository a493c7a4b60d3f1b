"""Which launches a batch takes (launches per step) and that the choice changes
no bit: few small events tiled launches of their own, events whose lines would
leave most of a tile unused the shared streaming launches."""
import numpy as np
import pytest

from paper_1206_0919_gb300 import shasta as S
from paper_1206_0919_gb300 import workloads as W
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


def prims(shape, seed):
    return W.random_state(shape, seed=seed, vmax=0.5, e_range=(0.3, 3.0)).as_list()


def batch(events, steps, **kw):
    """events: (shape, equation of state, steps taken before the next is added)."""
    with S.Batch(sum(int(np.prod(e[0])) for e in events) + 64 * len(events), **kw) as b:
        ids = []
        for i, (shape, eos, ahead) in enumerate(events):
            ids.append(b.add_primitives(shape, prims(shape, i), eos=eos))
            b.step(ahead)
        b.step(steps)
        return [b.get_conserved(i) for i in ids], [b.counters(i) for i in ids], b.info()


def same(a, b):
    return a[1] == b[1] and all(np.array_equal(x, y) for u, v in zip(a[0], b[0]) for x, y in zip(u, v))


@pytest.mark.parametrize("shape,tiles", [((48, 48, 48), True), ((16, 16, 16), True), ((512, 512, 1), False),
                                         ((4, 500, 500), False)])
def test_thin_events_stream(monkeypatch, shape, tiles):
    require_gpu()
    events = [(shape, "ideal", 0)] * 2
    monkeypatch.setenv("SHASTA_TILE", "off")
    ref = batch(events, 8)
    assert ref[2]["launches_per_step"] == 3
    monkeypatch.setenv("SHASTA_TILE", "")
    got = batch(events, 8)
    assert got[2]["launches_per_step"] == (6 if tiles else 3)
    assert same(ref, got)
