"""Autotuner: the site ordering of a set's domains, and the launch setting of its context.

The ordering decides: the device layout is fixed when a domain is built, so `tune_ordering` builds
the set in each ordering and times `Context.step`, the way the set is then stepped (resident
launches for small sets, per-step kernels for others, where the orderings compare differently).

The setting (threads per block, sites per thread, kernel variant) selects nothing: the library
itself picks the kernel form and launch shape of every launch (see kernel_variant in hemegb.h).
`autotune` still times each accepted one, with CUDA events around every stream-collide launch
(hg_step_profiled), keeps the fastest, and restores every domain's state, step count, boundary
values and iolet means afterwards (hg_save_state / hg_load_state), so tuning never changes the
simulation; the candidates of one context time alike and compute the same bits.

Results are kept in a JSON cache (``$HEMEGB_TUNE_CACHE``, default
``~/.cache/hemegb/tune.json``) keyed by device, storage, scheme, domain sizes
and device orderings, so a later process on the same machine reuses the choice instead of
re-timing (and a run under a profiler, whose timings are distorted, picks the
same as the plain run before it).
"""
from __future__ import annotations

import hashlib
import json
import os

DEFAULT_CANDIDATES = (
    (256, 1, 0), (128, 1, 0), (512, 1, 0), (256, 2, 0), (128, 2, 0), (512, 2, 0),
    (128, 1, 1), (256, 1, 1), (128, 2, 1), (256, 2, 1), (64, 2, 1),
    (128, 2, 2), (256, 2, 2), (256, 1, 2),  # variant 2: AA scheme only
    (256, 1, 3), (128, 1, 3), (256, 2, 3), (128, 2, 3), (512, 2, 3), (128, 4, 3), (256, 4, 3),
    (128, 2, 5), (256, 2, 5), (512, 2, 5),  # variant 5: A/B with 16-bit storage only
    (128, 2, 6), (256, 2, 6), (256, 2, 7), (512, 2, 7),  # variants 6, 7: AA only
    (256, 1, 8), (256, 2, 9), (256, 2, 10), (256, 2, 11), (128, 1, 12), (128, 2, 13), (128, 2, 14),
)
AA_ONLY = (2, 4, 6, 7, 10, 11, 12, 14)
AB_16BIT_ONLY = (5, 9)


def allowed(ctx, candidates):
    """The candidates the context's storage and scheme support."""
    if ctx.scheme != 1:
        candidates = [c for c in candidates if c[2] not in AA_ONLY]
    if ctx.scheme != 0 or ctx.storage == 0:
        candidates = [c for c in candidates if c[2] not in AB_16BIT_ONLY]
    return candidates


def _cache_path():
    return os.environ.get("HEMEGB_TUNE_CACHE",
                          os.path.join(os.path.expanduser("~"), ".cache", "hemegb", "tune.json"))


def _key(ctx, candidates):
    try:
        import torch

        dev = torch.cuda.get_device_name(ctx.device)
    except Exception:
        dev = "cuda"
    sizes = ",".join(f"{d.n}/{getattr(d, 'ordering', 0)}" for d in ctx.domains)
    cands = hashlib.sha1(repr(sorted(tuple(c) for c in candidates)).encode()).hexdigest()[:8]
    return f"{dev}|storage={ctx.storage}|scheme={ctx.scheme}|sites={sizes}|candidates={cands}"


def _load():
    try:
        with open(_cache_path()) as f:
            return json.load(f)
    except Exception:
        return {}


def _store(key, best, timing):
    _put(key, {"best": list(best), "ms": {"x".join(map(str, k)): v for k, v in timing.items()}})


def _put(key, entry):
    path = _cache_path()
    try:
        os.makedirs(os.path.dirname(path), exist_ok=True)
        data = _load()
        data[key] = entry
        tmp = path + f".{os.getpid()}.tmp"
        with open(tmp, "w") as f:
            json.dump(data, f, indent=1)
        os.replace(tmp, path)
    except OSError:
        pass


def autotune(ctx, candidates=DEFAULT_CANDIDATES, steps=12, warmup=2, use_cache=True):
    """Pick the fastest launch setting for `ctx`; returns (best, {candidate: ms per launch})."""
    if not ctx.domains:
        raise ValueError("autotune needs at least one domain in the context")
    candidates = allowed(ctx, candidates)
    key = _key(ctx, candidates)
    if use_cache:
        hit = _load().get(key)
        if hit:
            best = tuple(hit["best"])
            ctx.set_launch(*best)
            return best, {tuple(int(x) for x in k.split("x")): v for k, v in hit["ms"].items()}
    steps += steps & 1  # balance odd and even steps of the AA scheme
    saved = [(d, d.save_state()) for d in ctx.domains]
    timing = {}
    try:
        for cand in candidates:
            ctx.set_launch(*cand)
            ctx.step(warmup)
            ms_sc, _ = ctx.step_profiled(steps)
            timing[tuple(cand)] = ms_sc / steps
    finally:
        for d, buf in saved:
            d.load_state(buf)
    best = min(timing, key=timing.get)
    ctx.set_launch(*best)
    if use_cache:
        _store(key, best, timing)
    return best, timing


def step_ms(ctx, steps=64, repeats=5):
    """Milliseconds per step of ctx.step(steps): the fastest of `repeats`, CUDA events on the
    context's stream.  Advances the domains."""
    import torch

    ctx.step(2)
    ms = []
    for _ in range(repeats):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(ctx.stream)
        ctx.step(steps)
        e1.record(ctx.stream)
        e1.synchronize()
        ms.append(e0.elapsed_time(e1) / steps)
    return min(ms)


def tune_ordering(make_ctx, orderings=("morton", "rows", "bricks"), candidates=DEFAULT_CANDIDATES,
                  use_cache=True):
    """Site ordering as a tuning dimension: the device layout is fixed when a domain is
    built, so ``make_ctx(ordering)`` builds a fresh context with its domains in that
    ordering; each is launch-tuned, stepped and closed again.  Returns (best ordering, its
    launch setting, {ordering: (setting, ms per step of Context.step)}).  Every ordering
    computes bit-identical results."""
    table = {}
    for o in orderings:
        ctx = make_ctx(o)
        try:
            best, _ = autotune(ctx, candidates, use_cache=use_cache)
            key = _key(ctx, ()) + "|step"
            hit = _load().get(key) if use_cache else None
            ms = hit["ms_per_step"] if hit else step_ms(ctx)
            if use_cache and not hit:
                _put(key, {"ms_per_step": ms})
            table[o] = (best, ms)
        finally:
            ctx.close()
    o = min(table, key=lambda k: table[k][1])
    return o, table[o][0], table


def autotune_split(ctx, split, candidates=DEFAULT_CANDIDATES, steps=12, warmup=2):
    """Launch setting of a split domain's context (it selects nothing, as for `autotune`): every
    candidate timed with CUDA events around `steps` whole steps.  A split keeps no checkpoint,
    so tuning advances it; every setting computes the same bits.  Returns (best, {candidate: ms per step})."""
    import torch

    candidates = allowed(ctx, candidates)
    timing = {}
    for cand in candidates:
        ctx.set_launch(*cand)
        split.step(warmup)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(ctx.stream)
        split.step(steps)
        e1.record(ctx.stream)
        e1.synchronize()
        timing[tuple(cand)] = e0.elapsed_time(e1) / steps
    best = min(timing, key=timing.get)
    ctx.set_launch(*best)
    return best, timing
