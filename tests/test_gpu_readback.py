"""Read-back after even and odd steps, with and without a run encoding, against the exported
state and one another: fields, the FP64 mass to the bit, checkpoints, NaN and Inf counts,
subnormal and signed-zero values, at site counts around the 8192-site chunks of the mass."""
import numpy as np
import pytest

from paper_2010_04144_gb300 import synth as S

pytestmark = pytest.mark.gpu

W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)


def _values(ctx, raw):
    """Stored values (19, n) as float32."""
    if ctx.storage == 2:
        return (raw.astype(np.uint32) << 16).view(np.float32)
    return raw.astype(np.float32)


def _mass(h, scaled):
    """The mass as documented: chunks of 8192 sites, 256 threads each with every 256th site in
    direction order, a fixed tree, chunk sums by thread in turn and the same tree."""
    v = h.astype(np.float64)
    if scaled:
        v = v * W[:, None]

    def tree(x):  # 256 partial sums: shuffles inside 8 warps, then over the warps
        x = x.reshape(8, 32)
        for o in (16, 8, 4, 2, 1):
            x = np.concatenate([x[:, :o] + x[:, o:2 * o], x[:, o:]], axis=1)
        y = np.concatenate([x[:, 0], np.zeros(24)])
        for o in (16, 8, 4, 2, 1):
            y = np.concatenate([y[:o] + y[o:2 * o], y[o:]])
        return y[0]

    n, parts = v.shape[1], []
    for lo in range(0, n, 8192):
        acc = np.zeros(256)
        for c in range(lo, min(lo + 8192, n), 256):
            w = v[:, c:min(c + 256, lo + 8192, n)]
            for i in range(19):
                acc[:w.shape[1]] += w[i]
        parts.append(tree(acc))
    acc = np.zeros(256)
    for j in range(0, len(parts), 256):
        acc[:len(parts[j:j + 256])] += parts[j:j + 256]
    return tree(acc)


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_read_back(gpu, storage):
    fields = {}
    for scheme in ("ab", "aa"):
        for ordering in ("morton", "rows"):
            _read_back(gpu, storage, scheme, ordering, fields)
    for got in fields.values():
        assert len(got) == 4
        for m in got[1:]:
            assert np.array_equal(m, got[0])


def _read_back(gpu, storage, scheme, ordering, fields):
    for n in (1, 8191, 8193):
        g = S.box(32, 16, 20)
        order = np.lexsort((g.xyz[:, 0], g.xyz[:, 1], g.xyz[:, 2]))
        ctx = gpu.Context(storage=storage, scheme=scheme)
        d = ctx.domain(g.xyz[order][:n], [], ordering=ordering)
        buf = d.save_state()
        v = S.random_state(n, 11, 1e-3, np.float32)
        v[:, ::5] *= 1e-37 if storage != "f16" else 1e-4  # subnormals of the storage type
        v[:, 2::7] = -0.0
        raw = v if storage == "f32" else v.astype(np.float16) if storage == "f16" else \
            (v.view(np.uint32) >> 16).astype(np.uint16)
        buf[40:] = np.frombuffer(raw.tobytes(), np.uint8)
        d.load_state(buf)
        for steps in (0, 1, 2):  # t = 0, 1, 3
            ctx.step_profiled(steps)
            raw = d.state()
            h = _values(ctx, raw)
            mass, bad, _ = d.state_check()
            assert bad == 0 and mass == _mass(h, storage != "f32")
            m = d.macroscopic()
            if storage == "f32":  # FP32 sums in direction order, to the bit
                drho = np.zeros(n, np.float32)
                for i in range(19):
                    drho = drho + h[i]
                assert np.array_equal(m[:, 0], drho)
            fields.setdefault((n, steps), []).append(m)  # every arrangement: the same bits
            saved = d.save_state()
            d.load_state(saved)
            assert np.array_equal(d.state(), raw) and np.array_equal(d.save_state(), saved)
        ctx.close()


@pytest.mark.parametrize("storage,scheme", [("f32", "aa"), ("f16", "ab"), ("bf16", "aa")])
def test_nonfinite_counted(gpu, storage, scheme):
    ctx = gpu.Context(storage=storage, scheme=scheme)
    d = ctx.domain(S.box(12, 12, 12).xyz, [], ordering="rows")
    buf = d.save_state()
    raw = np.zeros((19, d.n), {"f32": np.float32, "f16": np.float16, "bf16": np.uint16}[storage])
    nan, inf = (0x7FC0, 0xFF80) if storage == "bf16" else (np.nan, -np.inf)
    raw[3, 5], raw[18, 700], raw[0, d.n - 1] = nan, inf, nan
    buf[40:] = np.frombuffer(raw.tobytes(), np.uint8)
    d.load_state(buf)
    assert d.state_check()[1] == 3
    ctx.close()
