"""Project autotuner: picks launch shapes by timing them on the device and
caches the choice as JSON (one file per machine, next to the built library).

Two searches:
  * single cavity: the (bx, by) block shape of the stream-collide kernels;
  * ensemble: (threads per block, nodes per thread) of the persistent kernel.
An entry is for the device, what the choice depends on (edge lengths, heated
face, storage, nodes per thread, conduction in the solid; for an ensemble its
members' edges and faces) and the library's sources: shapes measured with other
kernels, or before the default was one of the candidates, are measured anew.
Timing is by CUDA events on the handle's stream; the state advances while
tuning (tune before the run you care about, or on a scratch copy).
"""
from __future__ import annotations

import functools
import hashlib
import json
import os

from . import build as _build

CACHE = os.path.join(_build.BUILD, "autotune.json")
CAVITY_SHAPES = ((0, 0), (128, 1), (64, 2), (32, 4))  # (0, 0): the default
ENSEMBLE_SHAPES = ((64, 2), (128, 1), (128, 2), (128, 4), (128, 8), (256, 1), (256, 2), (256, 4))


def _device_key():
    import torch
    return torch.cuda.get_device_name()


@functools.lru_cache(maxsize=None)
def _code_key():
    h = hashlib.sha1()
    for path in sorted(_build._deps()):
        with open(path, "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:12]


def _cavity_key(cav):
    return "cavity|%s|%s|face%d|p%d|pairs%d|solid%d|%s" % (
        _device_key(), "x".join(map(str, cav.shape)), cav.face, cav.precision, cav.node_pairs, cav.solid, _code_key())


def _ensemble_key(ens):
    members = hashlib.sha1(repr(ens.dims).encode()).hexdigest()[:12]
    return "ensemble|%s|n%d|%s|p%d|%s" % (_device_key(), ens.n, members, ens.precision, _code_key())


def _load():
    try:
        with open(CACHE) as fh:
            return json.load(fh)
    except (OSError, ValueError):
        return {}


def _save(d):
    os.makedirs(os.path.dirname(CACHE), exist_ok=True)
    tmp = CACHE + ".tmp%d" % os.getpid()
    with open(tmp, "w") as fh:
        json.dump(d, fh, indent=1, sort_keys=True)
    os.replace(tmp, CACHE)


def _time(step, sync, steps, stream):
    import torch
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    step(2)
    sync()
    e0.record(stream)
    step(steps)
    e1.record(stream)
    sync()
    torch.cuda.synchronize()
    return e0.elapsed_time(e1) / steps


def tune_cavity(cav, steps=20, shapes=CAVITY_SHAPES, use_cache=True):
    """Best (bx, by) for this cavity; applied to cav."""
    import torch
    key = _cavity_key(cav)
    cache = _load()
    if use_cache and key in cache:
        bx, by = cache[key]["shape"]
        cav.set_launch(bx, by)
        return tuple(cache[key]["shape"]), cache[key]
    stream = torch.cuda.current_stream()
    res = {}
    for bx, by in shapes:
        cav.set_launch(bx, by)
        res["%dx%d" % (bx, by)] = _time(cav.step, cav.sync, steps, stream)
    best = min(res, key=res.get)
    shape = tuple(int(v) for v in best.split("x"))
    cav.set_launch(*shape)
    cache[key] = {"shape": shape, "ms_per_step": res}
    _save(cache)
    return shape, cache[key]


def tune_ensemble(ens, steps=8, shapes=ENSEMBLE_SHAPES, use_cache=True, graph_steps=8):
    """Best (block, nodes per thread) of the persistent kernel; applied."""
    import torch
    key = _ensemble_key(ens)
    cache = _load()
    if use_cache and key in cache:
        b, k = cache[key]["shape"]
        ens.set_launch(b, k, graph_steps)
        return tuple(cache[key]["shape"]), cache[key]
    stream = torch.cuda.current_stream()
    res = {}
    for b, k in shapes:
        ens.set_launch(b, k, graph_steps)
        res["%dx%d" % (b, k)] = _time(ens.step, ens.sync, steps, stream)
    best = min(res, key=res.get)
    shape = tuple(int(v) for v in best.split("x"))
    ens.set_launch(shape[0], shape[1], graph_steps)
    cache[key] = {"shape": shape, "ms_per_step": res}
    _save(cache)
    return shape, cache[key]
