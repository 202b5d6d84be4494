"""Launch-configuration autotuner of the FP32 step.

The knobs are the z chunk of the pair kernel (planes one CTA marches) and the
tail chunk: long chunks re-read fewer boundary planes and pay fewer unit
prologues, short chunks fill the SMs; a tail of short chunks at the end of
each column (launched last) lets the SMs run out of work together (256^3 on
GB300: 397 us per step with 16-plane chunks, 383 us with 32-plane chunks
ending in 8-plane ones).  The first candidate is z chunk 0, the library's own
choice, which also has chunks of two lengths a plane apart and tails of other
lengths; it is kept unless another is faster by more than the timing's noise
(us per step, own choice against the best of the others: 64^3 10.3, 11.4;
128^3 60.2, 62.1; 192 x 128 x 128 82.8, 86.5; 300 x 80 x 80 56.9, 58.3; 256^3
383, 383).  "tiled64" names the same kernel as "tiled" and takes its
measurements.  The best choice depends on the grid's shape and the SM count,
so it is measured: each candidate runs a few steps of the sim's own state on a
scratch copy of the sim (its own workspace, so the user's state and step count
are untouched), timed with CUDA events on the scratch sim's stream; the choice
is applied and cached per (device, grid, precision, scheme, boundary kinds,
candidates, kernel form and sources) in a JSON file (LBM_TUNE_CACHE, default
~/.cache/paper_1010_4135_gb300/launch.json), so each shape is tuned once.
FP64 sims always use the plain kernel and are not tuned.
"""
from __future__ import annotations

import functools
import glob
import hashlib
import json
import os
import threading

import torch

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "csrc")
ZCHUNKS = (0, 1, 2, 4, 6, 8, 12, 14, 16, 20, 24, 28, 32, 40, 48)  # 0: the library's own choice
ZTAILS = (0, 8, 16)  # 0: equal chunks; a tail length is tried only below the chunk length
VARIANTS = ("tiled", "tiled64")
# another launch has to take less than this share of the automatic one's time
# (ten timed steps of one launch repeat to 2 %, of the smallest grids to 6 %)
FASTER = 0.97
_lock = threading.Lock()


def cache_path() -> str:
    return os.environ.get("LBM_TUNE_CACHE") or os.path.join(
        os.path.expanduser("~"), ".cache", "paper_1010_4135_gb300", "launch.json")


def _load(path):
    try:
        with open(path) as fh:
            return json.load(fh)
    except (OSError, ValueError):
        return {}


def _store(path, key, value):
    with _lock:
        data = _load(path)
        data[key] = value
        os.makedirs(os.path.dirname(path) or ".", exist_ok=True)
        tmp = f"{path}.tmp{os.getpid()}"
        with open(tmp, "w") as fh:
            json.dump(data, fh, indent=1, sort_keys=True)
        os.replace(tmp, path)


def key_of(sims, batched: bool, device_name: str | None = None, sms: int | None = None,
           variants=None) -> str:
    """Cache key: device, SM count, the candidate tile shapes and tail lengths,
    and per sim the grid, precision, scheme and boundary kinds."""
    if device_name is None or sms is None:
        props = torch.cuda.get_device_properties(sims[0].device)
        device_name, sms = props.name, props.multi_processor_count
    parts = [device_name.replace(" ", "_"), str(int(sms)), "batch" if batched else "single",
             ",".join(variants or VARIANTS), "tails" + ",".join(str(t) for t in ZTAILS)]
    for s in sims:
        c = s.config
        parts.append("x".join(str(int(v)) for v in (c["nx"], c["ny"], c["nz"])) + f":{c['precision']}:{c['scheme']}:"
                     + "".join(str(int(k)) for k in tuple(c["bc_lo"]) + tuple(c["bc_hi"])))
    return "|".join(parts)


@functools.lru_cache(maxsize=None)
def kernel_hash() -> str:
    """Hash of the library's sources: a measurement is of one version of the kernels."""
    h = hashlib.sha256()
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        h.update(os.path.basename(path).encode())
        with open(path, "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def entry_of(sims, batched: bool, zchunks=ZCHUNKS, variants=None, device_name: str | None = None,
             sms: int | None = None) -> str:
    """Name of a cache entry: key_of, the z chunks measured, the kernels'
    version, and what else a sim's kernel form goes by (dt = tau, recovery)."""
    forms = [("dt=tau" if s.config["dt"] == s.config["tau"] else "dt!=tau") + (":recovery" if s.t_recovery else "")
             for s in sims]
    chunks = "chunks" + ",".join(str(int(z)) for z in zchunks)
    return "|".join([key_of(sims, batched, device_name, sms, variants), chunks, ",".join(forms), kernel_hash()])


def _time(run, steps: int, warmup: int) -> float:
    run(warmup)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    run(steps)
    e1.record()
    e1.synchronize()
    return e0.elapsed_time(e1) / steps


def candidates(zchunks=ZCHUNKS, variants=VARIANTS) -> list:
    """(variant, zchunk, ztail) launches to measure: every tile shape and z
    chunk (0: the automatic one) with equal chunks, and with each tail length
    below the chunk."""
    return [(v, int(zc), int(zt)) for v in variants for zc in zchunks for zt in ZTAILS if not zt or zt < zc]


def measure(sims, zchunks=ZCHUNKS, steps: int = 10, warmup: int = 2, batched: bool = False,
            variants=VARIANTS) -> dict:
    """{(variant, zchunk, ztail): ms per step} of the given sims' current states on scratch copies."""
    from . import sim as S
    scratch = []
    try:
        with torch.cuda.stream(torch.cuda.Stream(device=sims[0].device)):
            for s in sims:
                f = torch.empty((15,) + s.shape, dtype=torch.float32, device=s.device)
                s.sync()
                s.get_f(out=f)
                s.sync()
                c = s.clone(stream=torch.cuda.current_stream(s.device))
                c.set_t_recovery(s.t_recovery)
                scratch.append((c, f))

            def ms(launch):
                for c, f in scratch:
                    c.set_launch(*launch)
                    c.set_f(f)
                if batched:
                    run = lambda n: S.step_batch([c for c, _ in scratch], n)
                else:
                    run = scratch[0][0].step
                return _time(run, steps, warmup)

            out = {}
            for v, zc, zt in candidates(zchunks, variants):
                if v == "tiled64" and ("tiled", zc, zt) in out:
                    out[(v, zc, zt)] = out[("tiled", zc, zt)]
                else:
                    out[(v, zc, zt)] = ms((v, zc, zt))
            # the automatic launch once more: the first one timed bears the clocks' rise
            again = {}
            for a in [k for k in out if k[1] == 0]:
                name = "tiled" if a[0] == "tiled64" else a[0]
                if name not in again:
                    again[name] = ms(a)
                out[a] = min(out[a], again[name])
            return out
    finally:
        for c, _ in scratch:
            c.close()


def choose(timings) -> tuple:
    """The fastest launch, but the automatic one (z chunk 0) unless another is
    faster by more than the timing's noise."""
    best = min(timings, key=timings.get)
    auto = min((k for k in timings if k[1] == 0), key=timings.get, default=best)
    return best if timings[best] < FASTER * timings[auto] else auto


def tune(sim, zchunks=ZCHUNKS, steps: int = 10, use_cache: bool = True, path: str | None = None,
         variants=VARIANTS) -> dict:
    """Choose and apply the tile shape, z chunk (0: automatic) and tail of one FP32 sim;
    returns {"variant", "zchunk", "ztail", "ms", "cached", "timings"}."""
    return _tune([sim], zchunks, steps, use_cache, path, batched=False, variants=variants)


def tune_batch(sims, zchunks=ZCHUNKS, steps: int = 10, use_cache: bool = True, path: str | None = None,
               variants=VARIANTS) -> dict:
    """Choose and apply one tile shape, z chunk and tail for sims stepped together (lbm_step_batch)."""
    return _tune(list(sims), zchunks, steps, use_cache, path, batched=True, variants=variants)


def _tune(sims, zchunks, steps, use_cache, path, batched, key=None, variants=VARIANTS):
    if any(s.config["precision"] not in ("fp32", 1) for s in sims):
        return {"variant": None, "zchunk": None, "ztail": None, "ms": None, "cached": False, "timings": {}}
    path = path or cache_path()
    key = key or entry_of(sims, batched, zchunks, variants)
    hit = _load(path).get(key) if use_cache else None
    if hit is not None:
        for s in sims:
            s.set_launch(hit["variant"], int(hit["zchunk"]), int(hit.get("ztail", 0)))
        return {**hit, "cached": True}
    timings = measure(sims, zchunks, steps, batched=batched, variants=variants)
    best = choose(timings)
    for s in sims:
        s.set_launch(*best)
    rec = {"variant": best[0], "zchunk": best[1], "ztail": best[2], "ms": timings[best],
           "timings": {f"{v}:{z}:{t}": ms for (v, z, t), ms in timings.items()}}
    _store(path, key, rec)
    return {**rec, "cached": False}
