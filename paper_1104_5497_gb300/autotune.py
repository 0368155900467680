"""Autotuner for the trackers, per (ring size, GPU): launch shapes, threads per path of
the FP64 lists, and the FP32 pass's step-control constants.

Stage 1 (scheduling: every path's arithmetic is unchanged, so a tuned solve gives the
same endpoints bit for bit): the FP32 tracker over its resident warps per SM
(`nphc_options.blocks_per_sm`), then the FP64 continuation of the sample's hand-offs with
one path per warp at 1 to 4 blocks per SM (`list_blocks_per_sm`).

Stage 2 (gated by parity): the FP64 lists' threads per path (`threads_per_path`: a warp or
four lanes per path by the list's length, or one path per thread; their rounding differs)
and the FP32 pass's step control, the corrector's iteration cap (`max_newton_fp32`) and
tolerance (`eps_fp32`), which decide which steps it accepts and which paths it hands to
FP64.  Each candidate runs the calibration sample through the FP32 pass, the FP64
continuation of its hand-offs and the certification, and is kept only if every sample
path ends with the class it has under the options as given and every certified endpoint
equals theirs within 1e-10 relative; among those the fastest wins.  With the default
sample (every path up to N = 10) the gate covers the whole ring.

The list tracker's best shape depends on how long the hand-off list is, so the sample
must reproduce it: by default it is every path up to N = 10 (262,144).  The result is
cached in a JSON file under a key made of N, the GPU's name, its SM count and the trackers'
sources: what was measured on other kernels says nothing about these.

Every step runs through the C ABI (nphc_track, nphc_refine_certify on caller-owned device
buffers); this module only chooses options and times calls with CUDA events.
"""
from __future__ import annotations

import ctypes
import functools
import hashlib
import json
import os

import numpy as np

from . import nphc as N_

# resident warps per SM; 0 = the occupancy maximum (7 or 8 with a path per thread, about 16 in blocks
# of four with four lanes per path)
FP32_CANDIDATES = (0, 12, 8, 6, 4)
LIST_CANDIDATES = (2, 1, 3, 4)      # blocks of 4 warps per SM (the default, 2, first)
# FP32 step control: (max_newton_fp32, eps_fp32); the defaults first
STEP_CANDIDATES = ((3, 1e-5), (2, 1e-5), (3, 3e-5), (2, 3e-5))
THREADS_PER_PATH = (0, 1)           # FP64 lists; 0 = the library's automatic choice
DEFAULT_CACHE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "_build", "autotune.json")


def calibration_paths(npaths: int, sample: int) -> np.ndarray:
    """`sample` path indices spread evenly over [0, npaths) (all of them if fewer)."""
    if sample >= npaths:
        return np.arange(npaths, dtype=np.int64)
    return (np.arange(sample, dtype=np.int64) * npaths) // sample


def pick(timings: dict) -> int:
    """The fastest candidate; ties go to the one listed first (the default)."""
    best, best_t = None, None
    for k, t in timings.items():
        if best_t is None or t < best_t:
            best, best_t = k, t
    return int(best)


@functools.lru_cache(maxsize=None)
def kernels() -> str:
    """A hash of the trackers' sources (csrc/xy_*, what they include, and their launchers)."""
    d = os.path.join(os.path.dirname(os.path.abspath(__file__)), "csrc")
    h = hashlib.sha256()
    for f in sorted(os.listdir(d)):
        if f.startswith("xy_") or f in ("f32_step.cuh", "nphc_internal.cuh", "nphc_api.cu"):
            with open(os.path.join(d, f), "rb") as fh:
                h.update(f.encode() + b"\0" + fh.read())
    return h.hexdigest()[:16]


def cache_key(N: int, device_name: str, sms: int) -> str:
    return f"N={N}|{device_name}|sms={sms}|kernels={kernels()}"


def load_cache(path: str) -> dict:
    try:
        with open(path) as fh:
            return json.load(fh)
    except (OSError, ValueError):
        return {}


def store_cache(path: str, key: str, entry: dict) -> None:
    d = load_cache(path)
    d[key] = entry
    os.makedirs(os.path.dirname(path), exist_ok=True)
    tmp = f"{path}.tmp{os.getpid()}"
    with open(tmp, "w") as fh:
        json.dump(d, fh, indent=1, sort_keys=True)
    os.replace(tmp, path)


def apply(opts, entry: dict):
    """A copy of opts with the tuned values (the keys entry has)."""
    o = N_.nphc_options()
    ctypes.memmove(ctypes.byref(o), ctypes.byref(opts), ctypes.sizeof(o))
    o.blocks_per_sm = int(entry["blocks_per_sm"])
    o.list_blocks_per_sm = int(entry["list_blocks_per_sm"])
    if "threads_per_path" in entry:
        o.threads_per_path = int(entry["threads_per_path"])
    if "max_newton_fp32" in entry:
        o.max_newton_fp32 = int(entry["max_newton_fp32"])
        o.eps_fp32 = float(entry["eps_fp32"])
    return o


def same_certified(a: dict, b: dict, rel: float = 1e-10) -> bool:
    """Two runs of the calibration sample agree: every path has the same class, and every
    certified endpoint the same value within rel (1 + |z|)."""
    if not np.array_equal(a["cls"], b["cls"]):
        return False
    c = np.isin(a["cls"], [N_.END_REAL, N_.END_NONREAL, N_.END_UNDECIDED])
    if not c.any():
        return True
    d = np.abs(a["z"][c] - b["z"][c]).max(axis=1)
    return bool((d <= rel * (1 + np.abs(b["z"][c]).max(axis=1))).all())


def _median_ms(fn, reps: int) -> float:
    import torch
    ts = []
    for _ in range(reps):
        a = torch.cuda.Event(enable_timing=True)
        b = torch.cuda.Event(enable_timing=True)
        a.record()
        fn()
        b.record()
        torch.cuda.synchronize()
        ts.append(a.elapsed_time(b))
    return float(np.median(ts))


def tune(system, opts, sample: int = 262144, reps: int = 3, cache: str | None = DEFAULT_CACHE,
         refresh: bool = False, measure: bool = True):
    """Returns (tuned options, report).  report: the key, the chosen values, the timings
    (ms per candidate) and whether it came from the cache.  measure=False: the cached
    entry if there is one, else opts unchanged (no kernel launches)."""
    import torch
    if system.N == 0:   # generic quadratic systems: FP64 only, nothing to choose
        return apply(opts, dict(blocks_per_sm=opts.blocks_per_sm,
                                list_blocks_per_sm=opts.list_blocks_per_sm)), dict(cached=False)
    props = torch.cuda.get_device_properties(torch.cuda.current_device())
    key = cache_key(system.N, props.name, props.multi_processor_count)
    if cache and not refresh:
        hit = load_cache(cache).get(key)
        if hit:
            return apply(opts, hit), dict(hit, key=key, cached=True)
    if not measure:
        same = dict(blocks_per_sm=opts.blocks_per_sm, list_blocks_per_sm=opts.list_blocks_per_sm)
        return apply(opts, same), dict(same, key=key, cached=False)
    paths = calibration_paths(system.npaths, sample)
    ep = N_.DeviceEndpoints.empty(system.n, paths)
    ws = torch.empty(system.workspace_size(ep.count), dtype=torch.uint8, device="cuda")
    # FP32 tracker: every candidate tracks the whole sample from its start points
    fp32 = {}
    for bps in FP32_CANDIDATES:
        o = apply(opts, dict(blocks_per_sm=bps, list_blocks_per_sm=0))
        N_.track(system, o, N_.PREC_MIXED, ep, ws)   # warm-up (kernel attributes, caches)
        fp32[bps] = _median_ms(lambda: N_.track(system, o, N_.PREC_MIXED, ep, ws), reps)
    bps32 = pick(fp32)
    # FP64 list tracker: the sample's hand-offs, continued from the same state each time
    o = apply(opts, dict(blocks_per_sm=bps32, list_blocks_per_sm=0))
    N_.track(system, o, N_.PREC_MIXED, ep, ws)
    torch.cuda.synchronize()
    st = ep.tensors["status"]
    ho = torch.nonzero((st == N_.PATH_HANDOFF) | (st == N_.PATH_HANDOFF_COND)).flatten().to(torch.int32)
    lists = {}
    if ho.numel() > 0:
        count = torch.tensor([ho.numel()], dtype=torch.int32, device="cuda")
        saved = {k: v.clone() for k, v in ep.tensors.items() if k != "path"}

        def restore():
            for k, v in saved.items():
                ep.tensors[k].copy_(v)

        for lb in LIST_CANDIDATES:
            ol = apply(opts, dict(blocks_per_sm=bps32, list_blocks_per_sm=lb, threads_per_path=32))
            run = lambda: N_.track(system, ol, N_.PREC_FP64, ep, ws, ho, count, resume=True)
            restore()
            run()                                      # warm-up
            ts = []
            for _ in range(reps):
                restore()
                torch.cuda.synchronize()
                ts.append(_median_ms(run, 1))
            lists[lb] = float(np.median(ts))
        restore()
    lb = pick(lists) if lists else 0
    shapes = dict(blocks_per_sm=bps32, list_blocks_per_sm=lb)

    # stage 2: threads per path and FP32 step control, each candidate gated on the
    # certified sample of the options as given
    def sample_run(o):
        N_.track(system, o, N_.PREC_MIXED, ep, ws)
        s32 = ep.tensors["status"]
        h = torch.nonzero((s32 == N_.PATH_HANDOFF) | (s32 == N_.PATH_HANDOFF_COND)).flatten().to(torch.int32)
        if h.numel() > 0:
            n = torch.tensor([h.numel()], dtype=torch.int32, device="cuda")
            N_.track(system, o, N_.PREC_FP64, ep, ws, h, n, resume=True)

    cands = [(opts.threads_per_path, opts.max_newton_fp32, opts.eps_fp32)]   # as given: the reference
    cands += [(t, mn, eps) for t in THREADS_PER_PATH for mn, eps in STEP_CANDIDATES
              if (t, mn, eps) != cands[0]]
    steps, gate = {}, {}
    ref = None
    for tpp, mn, eps in cands:
        o = apply(opts, dict(shapes, threads_per_path=tpp, max_newton_fp32=mn, eps_fp32=eps))
        sample_run(o)                                  # warm-up
        steps[(tpp, mn, eps)] = _median_ms(lambda: sample_run(o), reps)
        sample_run(o)
        N_.refine_certify(system, o, ep)
        torch.cuda.synchronize()
        got = dict(cls=ep.tensors["cls"].cpu().numpy(),
                   z=(ep.tensors["z_re"] + 1j * ep.tensors["z_im"]).cpu().numpy().T)
        if ref is None:
            ref = got
        gate[(tpp, mn, eps)] = same_certified(got, ref)
    ok = [k for k in cands if gate[k]]
    tpp, mn, eps = min(ok, key=lambda k: (steps[k], cands.index(k)))
    key_s = lambda k: f"{k[0]},{k[1]},{k[2]:g}"
    entry = dict(shapes, threads_per_path=tpp, max_newton_fp32=mn, eps_fp32=eps,
                 sample=int(ep.count), handoffs=int(ho.numel()),
                 fp32_ms={str(k): v for k, v in fp32.items()},
                 list_ms={str(k): v for k, v in lists.items()},
                 step_ms={key_s(k): v for k, v in steps.items()},
                 step_gate={key_s(k): bool(v) for k, v in gate.items()})
    if cache:
        store_cache(cache, key, entry)
    return apply(opts, entry), dict(entry, key=key, cached=False)
