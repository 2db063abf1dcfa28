"""Autotuner for the rasteriser launch shape.

Times, on the caller's own model and views, every tile size (8, 16, 32) with
every pixels-per-thread (1, 2, 4 where a tile fills whole warps) of the two
rasteriser kernels, and picks the tile size whose projection + sort + best
forward + best backward is fastest. Every shape computes the same image and
resume record; a shape's batch changes nothing and is not timed.
"""
from __future__ import annotations

import dataclasses
import json

import torch

from . import lib


@dataclasses.dataclass
class RasterTuning:
    tile: int
    fwd: tuple[int, int]  # (pixels per thread, batch)
    bwd: tuple[int, int]
    table: dict

    def to_json(self) -> str:
        return json.dumps(dataclasses.asdict(self))


def _time(fn, reps: int) -> float:
    fn()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(reps):
        fn()
    e1.record()
    torch.cuda.synchronize()
    return e0.elapsed_time(e1) / reps


def retile(cam: lib.GsCamera, tile: int) -> lib.GsCamera:
    c = lib.GsCamera()
    ctypes_copy = bytes(memoryview(cam).cast("B"))
    memoryview(c).cast("B")[:] = ctypes_copy
    c.tile = tile
    return c


def time_shapes(run, ppts, batches, reps: int) -> dict:
    """Milliseconds of run(cfg) by (pixels per thread, batch). No kernel depends
    on the batch, so that each pixels-per-thread is timed once for all of them."""
    times = {}
    for ppt in ppts:
        cfg = lib.raster_config(ppt, batches[0])
        t = _time(lambda: run(cfg), reps)
        times.update({(ppt, b): t for b in batches})
    return times


def pick(times: dict) -> tuple[int, int]:
    """The (pixels per thread, batch) to take: of the shapes within 5% of the
    fastest the smallest batch, then the fastest. Of time_shapes' times, where
    the batches of a pixels-per-thread are equal, that is the fastest
    pixels-per-thread with the smallest batch."""
    best = min(times.values())
    return min((k for k, t in times.items() if t <= 1.05 * best), key=lambda k: (k[1], times[k]))


def tune(model, cams, targets, tiles=(8, 16, 32), ppts=(1, 2, 4), batches=(32, 64, 128, 256), reps: int = 3,
         n_views: int = 2) -> RasterTuning:
    """``cams``/``targets``: a few representative views (camera, target image)."""
    table = {}
    best = None
    all_ppts = ppts
    for tile in tiles:
        ppts = [p for p in all_ppts if tile * tile // p >= 32]  # whole warps per tile
        views = [retile(c, tile) for c in cams[:n_views]]
        cap = model.measure_capacity(views)
        v = model.make_view(views[0], cap)
        t_ps = t_f = t_b = 0.0
        fwd_times, bwd_times = {}, {}
        for cam, gt in zip(views, targets[:n_views]):
            model.retarget(v, cam)
            t_ps += _time(lambda: (lib.gs_project(model.P, model.n, model.sh_degree, v.cam, model.splats),
                                   lib.gs_sort(model.splats, model.n, v.cam, v.sort_ws, v.capacity, v.vals, v.ranges,
                                               v.count)), reps)
            for k, t in time_shapes(lambda cfg: model.render_fwd(v, cfg), ppts, batches, reps).items():
                fwd_times[k] = fwd_times.get(k, 0.0) + t
            model.loss(v, gt)
            for k, t in time_shapes(lambda cfg: model.raster_bwd(v, cfg), ppts, batches, reps).items():
                bwd_times[k] = bwd_times.get(k, 0.0) + t
        model.grad2d.zero_()
        bf, bb = pick(fwd_times), pick(bwd_times)
        total = t_ps + fwd_times[bf] + bwd_times[bb]
        table[tile] = dict(project_sort_ms=t_ps / n_views, fwd_ms={f"{k[0]}x{k[1]}": t / n_views
                                                                  for k, t in fwd_times.items()},
                           bwd_ms={f"{k[0]}x{k[1]}": t / n_views for k, t in bwd_times.items()},
                           best_fwd=bf, best_bwd=bb, total_ms=total / n_views)
        if best is None or total < best[0]:
            best = (total, tile, bf, bb)
        del v
    return RasterTuning(tile=best[1], fwd=best[2], bwd=best[3], table=table)
