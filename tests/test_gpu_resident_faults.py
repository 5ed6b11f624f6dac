"""Resident launches that cannot be had: the set is stepped launch by launch, with the bits of
the resident launches.  The failures are made on the host; no GPU fault is made."""
import numpy as np
import pytest

from paper_2010_04144_gb300 import synth as S

pytestmark = pytest.mark.gpu


def _run(gpu, scheme, calls, prepare=lambda ctx: None):
    geos = [S.cylinder(radius=4, length=30, inlet=dict(kind=S.VELOCITY, value=0.02, pulse=S.PULSE_SINE, period=41.0)),
            S.tree(S.TreeSpec(depth=3, scale=0.25), period=37.0)]
    ctx = gpu.Context(storage="f32", scheme=scheme)
    doms = [ctx.domain(g.xyz, g.iolets) for g in geos]
    prepare(ctx)
    for n in calls:
        ctx.step(n)
    ctx.sync()
    out = []
    for d in doms:
        out += [d.state().copy(), d.iolet_stats(), d.boundary_values(), *d.adjacent_moments(), d.step]
    ctx.close()
    return out


@pytest.mark.parametrize("scheme", ["ab", "aa"])
@pytest.mark.parametrize("refused", [1, 2, 4])
def test_refused_launch_steps_launch_by_launch(gpu, scheme, refused):
    """The first launch of the first call, a later one of the same call (1024 steps each, so the
    rest begins at an even or, after the odd call, an odd step), and one of a later call."""
    calls = (2051, 37, 3)
    ref = _run(gpu, scheme, calls)
    got = _run(gpu, scheme, calls, lambda ctx: ctx.inject_fault(gpu.FAULT_LAUNCH, refused))
    for a, b in zip(ref, got):
        assert np.array_equal(a, b)
