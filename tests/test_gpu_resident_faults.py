"""Resident launches that cannot be had: the set is stepped launch by launch, with the bits of
the resident launches.  Bounded waits in them that give up: the launch ends, hg_sync reports it,
and the next launch is sound.  The failures are made on the host, or by a limit on the polls of a
wait; no GPU fault is made."""
import numpy as np
import pytest

from paper_2010_04144_gb300 import synth as S

pytestmark = pytest.mark.gpu


def _run(gpu, scheme, calls, prepare=lambda ctx: None, after=lambda ctx: None):
    geos = [S.cylinder(radius=4, length=30, inlet=dict(kind=S.VELOCITY, value=0.02, pulse=S.PULSE_SINE, period=41.0)),
            S.tree(S.TreeSpec(depth=3, scale=0.25), period=37.0)]
    ctx = gpu.Context(storage="f32", scheme=scheme)
    doms = [ctx.domain(g.xyz, g.iolets) for g in geos]
    prepare(ctx)
    for n in calls:
        ctx.step(n)
    ctx.sync()
    after(ctx)
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


def test_no_memory_for_tables(gpu):
    """The plan's eight buffers are had, the resident tables are not: the set is stepped launch by
    launch, and the call that returned HG_OK leaves no error text behind."""
    errors = []
    ref = _run(gpu, "ab", (37, 3))
    got = _run(gpu, "ab", (37, 3), lambda ctx: ctx.inject_fault(gpu.FAULT_ALLOC, 9),
               lambda ctx: errors.append(gpu.lib().hg_last_error(ctx.h)))
    assert errors == [b""]
    for a, b in zip(ref, got):
        assert np.array_equal(a, b)


def _coupled(gpu, scheme):
    from paper_2010_04144_gb300 import serve

    art, ven = (S.tree(S.TreeSpec(depth=3, scale=0.35), venous=v, period=37.0) for v in (False, True))
    pairs = serve.coupled_job_from_trees(0, 0.0, 1, art, ven, [0.3] * len(ven.iolets)).pairs
    ctx = gpu.Context(storage="f32", scheme=scheme)
    doms = [ctx.domain(g.xyz, g.iolets) for g in (art, ven)]
    ctx.couple(doms[0], doms[1], pairs)
    ctx.step(10)
    return ctx, doms


@pytest.mark.parametrize("scheme", ["ab", "aa"])
@pytest.mark.parametrize("polls", [1, 2, 3])
def test_waits_that_give_up(gpu, scheme, polls):
    """Every wait of a coupled set's launch (the step barrier, the coupled values, the iolet
    blocks' wait) runs out after a few polls, three launches in a row; after the states are loaded
    again the set steps to the bits of an undisturbed one."""
    got = []
    for disturbed in (False, True):
        ctx, doms = _coupled(gpu, scheme)
        saved = [d.save_state() for d in doms]
        if disturbed:
            ctx.inject_fault(gpu.FAULT_WAIT_LIMIT, polls)
            ctx.step(2100)
            with pytest.raises(gpu.HgError) as e:
                ctx.sync()
            assert e.value.code == gpu.HG_ERR_TIMEOUT
            assert [d.step for d in doms] == [2110, 2110]
            ctx.sync()  # reported once
            ctx.inject_fault(gpu.FAULT_WAIT_LIMIT, 0)
            for d, s in zip(doms, saved):
                d.load_state(s)
        ctx.step(57)
        ctx.sync()
        out = []
        for d in doms:
            out += [d.state().copy(), d.iolet_stats(), d.boundary_values(), *d.adjacent_moments(), d.step]
        got.append(out)
        ctx.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)


def _live(ctx):
    return sum(t.numel() for t in ctx._alloc.live.values())


@pytest.mark.parametrize("storage,scheme", [("f32", "ab"), ("f16", "aa")])
def test_device_memory_of_small_sets(gpu, storage, scheme):
    """What domains and their stepping hold stays below the server's estimate, and sets that are
    stepped in turn share one buffer of boundary values and moments."""
    from paper_2010_04144_gb300 import serve

    geos = [S.parallel_tubes(12, radius=4, length=20), S.cylinder(radius=9, length=30),
            S.tree(S.TreeSpec(depth=4, scale=0.2), period=37.0)]
    ctx = gpu.Context(storage=storage, scheme=scheme)
    before = _live(ctx)
    doms = [ctx.domain(g.xyz, g.iolets) for g in geos]
    ctx.step(100)
    ctx.sync()
    held = _live(ctx) - before
    assert held <= sum(serve.geometry_footprint(g, ctx.storage, ctx.scheme) for g in geos)
    for sub in (doms[:1], doms[1:], doms[:2]):
        ctx.step_domains(sub, 100)
    ctx.sync()
    # three more plans: tables (a tile of 16 bytes per 64 sites or more, descriptors), no scratch
    tables = 3 * (sum(g.n for g in geos) / 2 + 512 * sum(len(g.iolets) for g in geos) + 32 * 256)
    assert _live(ctx) - before - held <= tables
    # a larger set replaces the buffer; the first set steps on with new tables
    big = ctx.domain(*(lambda g: (g.xyz, g.iolets))(S.parallel_tubes(40, radius=3, length=12)))
    ctx.step(100)
    ctx.step_domains(doms, 100)
    ctx.sync()
    assert [d.step for d in doms + [big]] == [500, 500, 400, 100]
    ctx.close()


def test_launch_setting_keeps_plans(gpu):
    """A launch setting selects nothing, so setting one frees and builds nothing again."""
    geo = S.cylinder(radius=4, length=20)
    ctx = gpu.Context(storage="f16", scheme="aa")
    d = ctx.domain(geo.xyz, geo.iolets)
    ctx.step(20)
    held = set(ctx._alloc.live)
    for launch in ((128, 2, 14), (256, 1, 0), (128, 2, 1)):
        ctx.set_launch(*launch)
        assert set(ctx._alloc.live) == held
        ctx.step(20)
        assert set(ctx._alloc.live) == held
    assert d.step == 80
    ctx.close()
