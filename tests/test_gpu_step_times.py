"""Time per step of small sets, one way of stepping against another on the same card in turn: the
ratios that hold where the choice between resident launches and launches per step, and the chain
of launches, are sound.  Margins are wide against noise and narrow against what they catch."""
import time

import pytest

from paper_2010_04144_gb300 import synth as S

pytestmark = pytest.mark.gpu


def _us_per_step(ctx, steps, calls, repeats=7):
    ctx.step(steps)
    ctx.sync()
    times = []
    for _ in range(repeats):
        t = time.perf_counter()
        for _ in range(calls):
            ctx.step(steps)
        ctx.sync()
        times.append((time.perf_counter() - t) / (steps * calls) * 1e6)
    return min(times)


def _context(gpu, geo, storage, scheme, launches):
    ctx = gpu.Context(storage=storage, scheme=scheme)
    ctx.domain(geo.xyz, geo.iolets)
    if launches:
        ctx.inject_fault(gpu.FAULT_LAUNCH, 1)  # the set is then stepped launch by launch
    ctx.step(2)
    ctx.sync()
    return ctx


def test_launched_steps_of_many_iolets(gpu):
    """100 narrow tubes: both schemes are bound by the chain stream-collide, iolet update, next
    stream-collide, and take the same time (13 us; A/B took 17 with the update launched early)."""
    geo = S.parallel_tubes(100, radius=3, length=12)
    us = {}
    for scheme in ("ab", "aa"):
        ctx = _context(gpu, geo, "f32", scheme, launches=True)
        us[scheme] = _us_per_step(ctx, 100, 4)
        ctx.close()
    assert us["ab"] < 1.2 * us["aa"], us


@pytest.mark.parametrize("geo,storage,scheme,steps", [
    (lambda: S.cylinder(100, 12), "f32", "ab", 100),                # 31k slots an iolet: 72 us resident, 28 launched
    (lambda: S.parallel_tubes(100, radius=3, length=12), "f16", "aa", 20),  # 200 iolets: 28 us, 14 launched
    (lambda: S.cylinder(40, 10), "f32", "aa", 1),                   # single steps: 41 us, 22 launched
    (lambda: S.cylinder(50, 50), "f16", "ab", 1),                   # 64 us, 26 launched
    (lambda: S.tree(S.TreeSpec(depth=4, scale=0.5), period=100.0), "f32", "ab", 1),
])
def test_way_of_stepping_is_the_faster_one(gpu, geo, storage, scheme, steps):
    """Left to itself, a set takes no longer than launch by launch."""
    geo = geo()
    us = {}
    for launches in (True, False):
        ctx = _context(gpu, geo, storage, scheme, launches)
        us[launches] = _us_per_step(ctx, steps, max(1, 100 // steps))
        ctx.close()
    assert us[False] < 1.2 * us[True], us
