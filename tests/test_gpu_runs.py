"""The run-encoded stream-collide kernel against the 18-row table's, bit for bit, where their
tiles end: site counts around multiples of the tiles, runs that end anywhere, sites with iolet
links, every storage and scheme, one domain per launch and domains of mixed parity in one."""
import numpy as np
import pytest

from paper_2010_04144_gb300 import synth as S

pytestmark = pytest.mark.gpu


def _state(d, seed):
    """A saved state of domain d with every population perturbed."""
    buf = d.save_state()
    raw = S.random_state(d.n, seed, 2e-3, np.float32)
    off = 40 + 28 * d.n_iolets
    if d.ctx.storage == 0:
        buf[off:off + 76 * d.n] = np.frombuffer(raw.tobytes(), np.uint8)
    elif d.ctx.storage == 1:
        buf[off:off + 38 * d.n] = np.frombuffer(raw.astype(np.float16).tobytes(), np.uint8)
    else:
        buf[off:off + 38 * d.n] = np.frombuffer((raw.view(np.uint32) >> 16).astype(np.uint16).tobytes(), np.uint8)
    return buf


def _geometries():
    """Flat slabs (rows of 64 sites: runs) cut to counts around tile edges, a tube with iolets
    along x and a tree."""
    out = []
    for n in (127, 128, 129, 255, 257, 511, 513, 1025):
        g = S.box(64, 4, 8)
        order = np.lexsort((g.xyz[:, 0], g.xyz[:, 1], g.xyz[:, 2]))
        out.append(S.Geometry(xyz=g.xyz[order][:n], iolets=[]))
    out.append(S.cylinder(radius=5, length=50, axis=0,
                          inlet=dict(kind=S.VELOCITY, value=0.03, profile=S.PARABOLIC, pulse=S.PULSE_COSINE,
                                     period=50.0)))
    out.append(S.tree(S.TreeSpec(depth=3, scale=0.4)))
    return out


@pytest.mark.parametrize("scheme", ["ab", "aa"])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_run_and_table_kernels_tile_edges(gpu, storage, scheme):
    """Rows ordering has runs, Morton ordering none: the two kernels on the same state."""
    for geo in _geometries():
        got = []
        for ordering in ("rows", "morton"):
            ctx = gpu.Context(storage=storage, scheme=scheme)
            d = ctx.domain(geo.xyz, geo.iolets, ordering=ordering)
            assert (d.info()["n_runs"] > 0) == (ordering == "rows")
            d.load_state(_state(d, 3))
            ctx.step_profiled(5)  # one launch per step, whatever the size of the set
            got.append((d.state().copy(), d.iolet_stats(), d.boundary_values()))
            ctx.close()
        for a, b in zip(*got):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("scheme", ["ab", "aa"])
@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_packed_and_mixed_parity_launches(gpu, storage, scheme):
    """Several domains in one launch, at the same and at different step parities, with and
    without runs (one domain without them takes the whole launch to the table form)."""
    geos = [S.tree(S.TreeSpec(depth=3, scale=s)) for s in (0.3, 0.35, 0.4)]
    got = []
    for orderings in (("rows",) * 3, ("morton",) * 3, ("rows", "morton", "rows")):
        ctx = gpu.Context(storage=storage, scheme=scheme)
        doms = [ctx.domain(g.xyz, g.iolets, ordering=o) for g, o in zip(geos, orderings)]
        for j, d in enumerate(doms):
            d.load_state(_state(d, 5 + j))
        ctx.step_profiled(3)
        ctx.step_domains(doms[:1], 1)
        ctx.step_profiled(7)
        got.append([d.state().copy() for d in doms])
        ctx.close()
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert np.array_equal(a, b)
