"""Which launches a batch takes (launches per step) and that the choice changes
no bit: few small events tiled launches of their own, events whose lines would
leave most of a tile unused the shared streaming launches."""
import time

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


def us_per_step(b, n=12):
    best = 1e9
    b.step(n)
    b.sync()
    for _ in range(5):
        t = time.perf_counter()
        b.step(n)
        b.sync()
        best = min(best, time.perf_counter() - t)
    return best / n * 1e6


@pytest.mark.parametrize("shape,count,ahead", [((16, 16, 1024), 12, 0), ((1024, 16, 16), 12, 1), ((12, 700, 20), 10, 0)])
def test_long_lines_are_cut_beside_other_launches(monkeypatch, shape, count, ahead):
    """Long lines of several launches in a slot (two equations of state, events
    at different phases) are cut into ranges: the bits of whole line groups, in
    well under the time of those (measured at 0.3 to 0.6 of it)."""
    require_gpu()
    events = [(shape, "ideal" if ahead or i % 2 else "bag", ahead) for i in range(count)]
    res, us = [], []
    for forced in ("0", None):  # whole line groups, the rule
        if forced:
            monkeypatch.setenv("SHASTA_BATCH_RANGE", forced)
        else:
            monkeypatch.delenv("SHASTA_BATCH_RANGE")
        res.append(batch(events, 8, autotune=False))
        with S.Batch(count * int(np.prod(shape)) + 64 * count, autotune=False) as b:
            for i, (sh, eos, n) in enumerate(events):
                b.add_primitives(sh, prims(sh, i), eos=eos)
                b.step(n)
            us.append(us_per_step(b))
    assert same(*res)
    assert us[1] < 0.8 * us[0], us


def test_two_equations_of_state_are_tuned():
    """The autotuner times launches that differ for two equations of state side
    by side: two flat events (measured: 771 us a step with the ranges it picks,
    913 by the untimed rule, 854 with the other register variant alone), with
    the same bits."""
    require_gpu()
    shape = (500, 500, 30)
    events = [(shape, eos, 0) for eos in ("ideal", "bag")]
    pr = [prims(shape, i) for i in range(2)]
    res, us = [], []
    for tune in (True, False):
        with S.Batch(2 * int(np.prod(shape)) + 128, autotune=tune) as b:
            ids = [b.add_primitives(sh, p, eos=eos) for (sh, eos, _), p in zip(events, pr)]
            b.step(1)
            res.append(([b.get_conserved(i) for i in ids], [b.counters(i) for i in ids]))
            us.append(us_per_step(b))
    assert same(*res)
    assert us[0] < 0.9 * us[1], us


def test_phases_apart_skip_the_shares():
    """With events at different phases no share of the trials is used, so only
    the two register variants are timed: of sweeps over 0.2 ms four an axis, about
    four steps (eight with the shares)."""
    require_gpu()
    shape, ratio = (224, 224, 224), []
    with S.Batch(3 * 224 ** 3 + 192, autotune=False) as b:
        for i in range(3):
            b.add_primitives(shape, prims(shape, i))
            b.step(1)
        step = us_per_step(b)
        for _ in range(5):
            t = time.perf_counter()
            b.autotune()
            b.sync()
            ratio.append((time.perf_counter() - t) * 1e6 / step)
    assert min(ratio) < 5.5, ratio
