"""Autotuner of the compositing launches.

Two parameters of a launch change its time and no result: the forward's tile
batch (the splats of a tile's list staged per pass through shared memory: a
larger batch takes fewer barriers per list but more shared memory, and so
fewer resident CTAs) and the backward's tables per pass (one, or groups of
four, faster where the tables have opacity at the same scalars).  The best
choice depends on the tables, the image and the scene.  `tune` times the
launches that differ, as the pipeline names them (`launch_choices`; every
(group, batch) pair for a pipeline that names none), on the caller's actual
buffers with CUDA events and keeps the fastest; results are cached per
(device, problem signature) in a JSON file so a shape is tuned once.
"""
from __future__ import annotations

import json
import os

import torch

FWD_GROUPS = (1, 2, 4, 8)
BWD_GROUPS = (1, 2, 4)
BATCHES = (128, 256, 512)


def _cache_path():
    base = os.environ.get("XDG_CACHE_HOME", os.path.join(os.path.expanduser("~"), ".cache"))
    return os.path.join(base, "veg_gb300", "autotune.json")


def _load():
    try:
        with open(_cache_path()) as fh:
            return json.load(fh)
    except (OSError, ValueError):
        return {}


def _store(cache):
    path = _cache_path()
    try:
        os.makedirs(os.path.dirname(path), exist_ok=True)
        with open(path + ".tmp", "w") as fh:
            json.dump(cache, fh, indent=1, sort_keys=True)
        os.replace(path + ".tmp", path)
    except OSError:
        pass


def _time(fn, reps):
    fn()
    torch.cuda.synchronize()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    for _ in range(reps):
        fn()
    b.record()
    b.synchronize()
    return a.elapsed_time(b) / reps


def signature(p, n_tf):
    dev = torch.cuda.get_device_name(p.device)
    return f"{dev}|n={p.n}|V={p.V}|{p.W}x{p.H}|T={n_tf}|cap={p.capacity // (1 << 20)}"


def _choices(p, luts, n_tf):
    """({"fwd": [(group, batch), ...], "bwd": [...]}, cache tag)"""
    own = getattr(p, "launch_choices", None)
    if own is not None:
        return own(luts), "|launches"
    every = lambda groups: [(g, b) for g in groups if g == 1 or g // 2 < n_tf for b in BATCHES]
    return {"fwd": every(FWD_GROUPS), "bwd": every(BWD_GROUPS)}, "|batch"


def tune(p, luts, dout=None, reps=3, use_cache=True):
    """Chooses p.tf_group and p.tile_batch (forward), p.tf_group_bwd and
    p.tile_batch_bwd (backward, with `dout`) for pipeline `p` whose binning
    is current (project + bin_sort already run).  Returns {"fwd": group,
    "fwd_batch": batch, "bwd": group, "bwd_batch": batch, "times": ...}; a pass
    with a single launch to choose from is not timed."""
    n_tf = luts.shape[0]
    choices, tag = _choices(p, luts, n_tf)
    key = signature(p, n_tf) + ("|bwd" if dout is not None else "") + tag
    cache = _load() if use_cache else {}
    if key in cache:
        res = cache[key]
    else:
        times = {}

        def fastest(kind, group, batch, run):
            took = []
            for g, b in choices[kind]:
                setattr(p, group, g)
                setattr(p, batch, b)
                if len(choices[kind]) > 1:
                    times[f"{kind}{g}x{b}"] = _time(run, reps)
                    took.append((times[f"{kind}{g}x{b}"], (g, b)))
            best = min(took)[1] if took else choices[kind][0]
            setattr(p, group, best[0])
            setattr(p, batch, best[1])
            return best

        fwd, fwd_b = fastest("fwd", "tf_group", "tile_batch", lambda: p.composite(luts))
        p.composite(luts)
        bwd, bwd_b = (4, 256) if tag == "|batch" else (0, 0)
        if dout is not None:
            bwd, bwd_b = fastest("bwd", "tf_group_bwd", "tile_batch_bwd",
                                 lambda: p.backward_2d(dout))
        res = {"fwd": fwd, "fwd_batch": fwd_b, "bwd": bwd, "bwd_batch": bwd_b, "times": times}
        if use_cache:
            cache[key] = res
            _store(cache)
    p.tf_group, p.tile_batch = res["fwd"], res["fwd_batch"]
    p.tf_group_bwd, p.tile_batch_bwd = res["bwd"], res["bwd_batch"]
    return res
