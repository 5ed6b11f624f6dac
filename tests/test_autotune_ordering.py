"""The site ordering is chosen by the time of the way a set is really stepped (CPU only, stub
contexts): not by its stream-collide launches, which a small set's resident launches do not make."""
from paper_2010_04144_gb300 import autotune as AT

LAUNCHED = {"morton": 3.0, "rows": 1.0, "bricks": 2.0}  # ms per stream-collide launch
STEPPED = {"morton": 0.5, "rows": 0.7, "bricks": 0.6}   # ms per step of Context.step


class _Dom:
    n, ordering = 1000, 0

    def save_state(self):
        return b""

    def load_state(self, buf):
        pass


class _Ctx:
    device, storage, scheme = 0, 0, 0
    closed = timed = 0

    def __init__(self, ordering):
        self.o, self.domains = ordering, [_Dom()]
        self.domains[0].ordering = sorted(LAUNCHED).index(ordering)

    def set_launch(self, *launch):
        pass

    def step(self, n):
        pass

    def step_profiled(self, n):
        return LAUNCHED[self.o] * n, 0.0

    def close(self):
        _Ctx.closed += 1


def _step_ms(ctx, *args, **kw):
    _Ctx.timed += 1
    return STEPPED[ctx.o]


def test_ordering_by_the_way_the_set_is_stepped(tmp_path, monkeypatch):
    monkeypatch.setenv("HEMEGB_TUNE_CACHE", str(tmp_path / "tune.json"))
    monkeypatch.setattr(AT, "step_ms", _step_ms, raising=False)
    monkeypatch.setattr(_Ctx, "closed", 0)
    monkeypatch.setattr(_Ctx, "timed", 0)
    o, setting, table = AT.tune_ordering(_Ctx, candidates=[(256, 1, 0)])
    assert o == "morton" and setting == (256, 1, 0)
    assert {k: v[1] for k, v in table.items()} == STEPPED
    assert _Ctx.closed == 3 and _Ctx.timed == 3
    again = AT.tune_ordering(_Ctx, candidates=[(256, 1, 0)])  # from the cache, nothing timed
    assert again == (o, setting, table) and _Ctx.timed == 3
    other = AT.tune_ordering(_Ctx, candidates=[(256, 1, 0)], use_cache=False)
    assert other[0] == "morton" and _Ctx.timed == 6
