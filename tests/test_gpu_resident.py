"""Resident multi-step launches against the per-step kernels (hg_step_profiled launches every
step's kernels one by one), bit for bit: fields, iolet means, boundary values, boundary moments
and step counts, for single domains, packed ones and coupled pairs, at the edges of the launch
shapes (blocks of 128 to 512 sites, one to eight tiles a block, links in shared memory or not)."""
import numpy as np
import pytest

from paper_2010_04144_gb300 import synth as S

pytestmark = pytest.mark.gpu


def _snapshot(doms):
    out = []
    for d in doms:
        out += [d.state().copy(), d.iolet_stats(), d.boundary_values(), *d.adjacent_moments(), d.step]
    return out


def _tree(scale, depth=3, **kw):
    return S.tree(S.TreeSpec(depth=depth, scale=scale), period=37.0, **kw)


def _pair(scale):
    from paper_2010_04144_gb300 import serve

    art, ven = _tree(scale), _tree(scale, venous=True)
    job = serve.coupled_job_from_trees(0, 0.0, 1, art, ven, [0.3] * len(ven.iolets))
    return [art, ven], job.pairs


SETS = {
    "tube": lambda: ([S.cylinder(radius=5, length=31, inlet=dict(kind=S.VELOCITY, value=0.02, pulse=S.PULSE_SINE,
                                                                 period=41.0))], []),
    "closed box": lambda: ([S.box(16, 8, 8)], []),
    "ragged": lambda: ([S.cylinder(radius=3 + j % 4, length=9 + 13 * j, axis=j % 3) for j in range(9)], []),
    "many iolets": lambda: ([S.parallel_tubes(48, radius=3, length=12)], []),
    "pair": lambda: _pair(0.35),
    "two tiles": lambda: ([S.box(128, 64, 32)], []),
    "table from memory": lambda: ([_tree(1.45, depth=4)], []),
}


@pytest.mark.parametrize("name", list(SETS))
@pytest.mark.parametrize("scheme", ["ab", "aa"])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_resident_bit_identical(gpu, storage, scheme, name):
    geos, pairs = SETS[name]()
    for ordering in ("morton", "rows"):
        got = []
        for resident in (True, False):
            ctx = gpu.Context(storage=storage, scheme=scheme)
            doms = [ctx.domain(g.xyz, g.iolets, tau=0.7, ordering=ordering) for g in geos]
            if pairs:
                ctx.couple(doms[0], doms[1], pairs)
            if name == "closed box":
                buf = doms[0].save_state()
                v = S.random_state(doms[0].n, 1, 1e-3, np.float32)
                v = v if storage == "f32" else v.astype(np.float16) if storage == "f16" else \
                    (v.view(np.uint32) >> 16).astype(np.uint16)
                buf[40:] = np.frombuffer(v.tobytes(), np.uint8)
                doms[0].load_state(buf)
            for n in (2, 37, 3, 1, 66):
                (ctx.step if resident else ctx.step_profiled)(n)
            ctx.sync()
            got.append(_snapshot(doms))
            ctx.close()
        for a, b in zip(*got):
            assert np.array_equal(a, b)


def test_resident_mixed_progress_and_many_steps(gpu):
    """Domains at different step counts in one launch; more steps than one launch takes."""
    geos = [S.cylinder(radius=3, length=14), _tree(0.2), S.cylinder(radius=4, length=20, axis=0)]
    got = []
    for resident in (True, False):
        ctx = gpu.Context(storage="f32", scheme="aa")
        doms = [ctx.domain(g.xyz, g.iolets) for g in geos]
        if resident:
            ctx.step_domains(doms[:1], 3)
            ctx.step_domains(doms, 10)
            ctx.step_domains(doms, 4099)
        else:  # every domain alone, step by step
            for d, n in zip(doms, (4112, 4109, 4109)):
                for _ in range(n):
                    ctx.step_domains([d], 1)
        ctx.sync()
        got.append(_snapshot(doms))
        ctx.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)


def test_resident_two_contexts_at_once(gpu):
    """Two contexts on two streams, driven by two threads, both with full-size resident grids:
    each result is that of the context alone."""
    import threading

    geos = [_tree(1.1, depth=4), S.tree(S.TreeSpec(depth=4, scale=1.0, seed=7))]

    def run(geo, out, k):
        ctx = gpu.Context(storage="f32", scheme="ab")
        d = ctx.domain(geo.xyz, geo.iolets)
        for _ in range(6):
            ctx.step(150)
        ctx.sync()
        out[k] = _snapshot([d])
        ctx.close()

    alone, both = {}, {}
    for k, g in enumerate(geos):
        run(g, alone, k)
    threads = [threading.Thread(target=run, args=(g, both, k)) for k, g in enumerate(geos)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for k in range(2):
        for a, b in zip(alone[k], both[k]):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("scheme", ["ab", "aa"])
def test_steps_under_stream_capture(gpu, scheme):
    """A caller's capture records plain launches (no resident launch, no graph of the library's
    own), chained as on the stream: replays give the bits of stepping."""
    torch = pytest.importorskip("torch")
    geos, pairs = _pair(0.3)
    got = []
    for captured in (True, False):
        ctx = gpu.Context(storage="f32", scheme=scheme)
        doms = [ctx.domain(g.xyz, g.iolets, ordering=o) for g, o in zip(geos, ("rows", "morton"))]
        ctx.couple(doms[0], doms[1], pairs)
        ctx.step(2)
        if captured:
            ctx.sync()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=ctx.stream):
                ctx.step(4)
            with torch.cuda.stream(ctx.stream):
                for _ in range(6):
                    g.replay()
            ctx.sync()
        else:
            ctx.step(24)
        got.append([d.state().copy() for d in doms] + [d.iolet_stats() for d in doms]
                   + [d.boundary_values() for d in doms])
        ctx.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)


def test_resident_shapes_in_turn(gpu):
    """Sets of different launch shapes (much and little shared memory) stepped in turn."""
    geos = [S.box(128, 64, 32), S.cylinder(radius=4, length=20), S.parallel_tubes(3, radius=5, length=40)]
    ctxs = [gpu.Context(storage="f32", scheme="aa") for _ in geos]
    doms = [c.domain(g.xyz, g.iolets) for c, g in zip(ctxs, geos)]
    for n in (2, 3, 4):
        for c in ctxs:
            c.step(n)
    for c, g, d in zip(ctxs, geos, doms):
        c.sync()
        ref = gpu.Context(storage="f32", scheme="aa")
        r = ref.domain(g.xyz, g.iolets)
        ref.step_profiled(9)
        for a, b in zip(_snapshot([d]), _snapshot([r])):
            assert np.array_equal(a, b)
        ref.close()
        c.close()
