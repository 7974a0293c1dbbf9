"""Autotuning and reporting of the batched (many-atmosphere) solve.

``tune_batch`` sweeps the persistent launch's knobs (grid size, probes per
work item, items per queue claim, block-table staging, register budget) by
coordinate descent; ``tune_threshold`` picks the fastest IoD threshold whose J
error meets a bar; ``batch_report`` builds a seeded set of independent
atmospheres, then times one step three ways -- a sequential launch per
atmosphere, one persistent launch, and the whole step (line synthesis, grids,
MIPs and the persistent solve) replayed from a captured CUDA graph -- and writes
a JSON report with aggregate dense-equivalent segment throughput and
per-atmosphere completion times.

Usage: python -m paper_2511_08498_gb300.autotune [--scale S] [--out FILE]
"""

from __future__ import annotations

import argparse
import json
import sys

import numpy as np
import torch

from . import api

DISTANCE_LIMITS = [6.0, 24.0, 96.0]


def _time(fn, reps=3):
    fn()
    torch.cuda.synchronize()
    best = float("inf")
    for _ in range(reps):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        fn()
        e1.record()
        e1.synchronize()
        best = min(best, e0.elapsed_time(e1))
    return best


WALKS = {"per_batch": api.TRAVERSAL_PER_BATCH, "paired": api.TRAVERSAL_PAIRED}


def run_config(ctx, items, W, cfg, queue=None, **kw):
    """``dex_batch_solve_config`` with the knobs of ``cfg``; its ``walk`` (one walk
    per batch, or one per mirror pair of batches) is set on the context for the
    call."""
    cfg = dict(cfg)
    ctx.set_traversal(WALKS[cfg.pop("walk", "per_batch")])
    try:
        return api.batch_solve_config(ctx, items, W, queue=queue, **cfg, **kw)
    finally:
        ctx.set_traversal(api.TRAVERSAL_PER_BATCH)


def default_config(items, W, sms, walk="per_batch"):
    """The launch that ``dex_batch_solve`` makes of ``items`` when the grid is left to it."""
    packets = 0
    for it in items:
        n = -(-it.n_lambda // W)
        packets += it.capacity * (n if walk == "per_batch" else -(-n // 2))  # pairs and a lone batch
    small = packets < 6 * sms
    staging = int(all((it.nx // 16) * (it.nz // 16) <= 8192 for it in items))
    return dict(ctas=(6 if small else 3) * sms, packet=128 if small else 256, chunk=1, staging=staging, occupancy=0,
                walk=walk)


def tune_batch(ctx, items, W, reps=3, rounds=2):
    """Coordinate descent over the launch knobs of ``dex_batch_solve_config`` --
    persistent grid size, probes per work item (packet), work items per queue
    claim (chunk), block-table staging, register budget and the walk (one per
    wavelength batch, or one per mirror pair of batches, W = 8) -- starting from
    the default configuration; every knob is swept with the others fixed, twice.
    Returns ``{"best", "best_ms", "default", "default_ms", "trials"}``."""
    sms = torch.cuda.get_device_properties(ctx.device).multi_processor_count
    queue = torch.zeros(1, dtype=torch.int32, device=torch.device("cuda", ctx.device))
    default = default_config(items, W, sms)
    space = [("walk", ["per_batch", "paired"] if W == 8 else ["per_batch"]),
             ("ctas", [k * sms for k in (1, 2, 3, 4, 6, 8)]), ("packet", [256, 128, 64]), ("chunk", [1, 2, 4, 8, 16]),
             ("staging", [0, 1]), ("occupancy", [0, 1] if W == 8 else [0])]
    trials = {}

    def timed(cfg):
        key = tuple(sorted(cfg.items()))
        if key not in trials:
            trials[key] = _time(lambda: run_config(ctx, items, W, cfg, queue=queue), reps)
        return trials[key]

    best, best_t = dict(default), timed(default)
    for _ in range(rounds):
        for name, values in space:
            for v in values:
                cand = dict(best, **{name: v})
                t = timed(cand)
                if t < best_t:
                    best, best_t = cand, t
    return {"best": best, "best_ms": best_t, "default": default, "default_ms": trials[tuple(sorted(default.items()))],
            "trials": [{"config": dict(k), "ms": v} for k, v in trials.items()]}


def tune_threshold(ctx, atms, W, cfg, thresholds=(0.0, 1e-4, 1e-3, 1e-2, 1.0, 1e30), bar_pct=0.5, reps=3):
    """The IoD threshold of the batch: the fastest of ``thresholds`` whose J error
    against the full-resolution solve (MIP 0 only) has a 99.9th percentile of at
    most ``bar_pct`` % over every probe and wavelength of every atmosphere; if
    none meets it, the most accurate one (threshold 0 leaves only the
    always-average rule of Section 2.2)."""
    queue = torch.zeros(1, dtype=torch.int32, device="cuda")
    ref = []
    for a in atms:
        a.build(max_mip=0)
    items = [a.item() for a in atms]
    run_config(ctx, items, W, cfg, queue=queue)
    ctx.check()
    ref = [a.J.clone() for a in atms]
    out = []
    for thr in thresholds:
        for a in atms:
            a.iod = thr
            a.build()
        items = [a.item() for a in atms]
        t = _time(lambda: run_config(ctx, items, W, cfg, queue=queue), reps)
        ctx.check()
        errs = []
        for a, r in zip(atms, ref):
            mask = r > 0
            errs.append((((a.J - r).abs() / r.clamp_min(1e-30))[mask] * 100.0).double().cpu().numpy())
        e = np.concatenate(errs)
        out.append({"iod": thr, "ms": t, "j_err_pct_p99.9": float(np.percentile(e, 99.9)),
                    "j_err_pct_max": float(e.max())})
    ok = [o for o in out if o["j_err_pct_p99.9"] <= bar_pct]
    best = min(ok, key=lambda o: o["ms"]) if ok else min(out, key=lambda o: o["j_err_pct_p99.9"])
    return {"bar": f"J error p99.9 <= {bar_pct}% vs the full-resolution solve", "trials": out,
            "best_iod": best["iod"], "bar_met": bool(ok)}


class Atmosphere:
    """Device-resident model parameters and buffers of one atmosphere of the batch."""

    def __init__(self, ctx, spec, W, iod):
        import synth
        self.spec, self.ctx, self.W, self.iod = spec, ctx, W, iod
        m = synth.sparse_line_atmosphere(spec["nx"], spec["nz"], n_lambda=spec["n_lambda"],
                                         empty_frac=spec["empty_frac"], seed=spec["seed"])
        self.params = {k: torch.from_numpy(np.ascontiguousarray(m[k]).reshape(-1)).cuda()
                       for k in ("chi_c", "s_c", "s_l", "ratio", "dld", "dlam")}
        n = spec["nx"] * spec["nz"]
        self.eta = torch.empty((spec["n_lambda"], n), device="cuda")
        self.chi = torch.empty_like(self.eta)
        self.J = torch.empty_like(self.eta)
        dirs, w = synth.directions(spec["n_dir"])
        self.dirs, self.w = dirs, w
        self.dirs_dev, self.w_dev = torch.from_numpy(dirs).cuda(), torch.from_numpy(w).cuda()
        self.grid = None
        self.mips = None
        self.build()

    def build(self, max_mip=3):
        p = self.params
        api.synth_static_line(self.ctx, p["chi_c"], p["s_c"], p["s_l"], p["ratio"], p["dld"], p["dlam"],
                              eta=self.eta, chi=self.chi)
        self.grid = api.grid_build(self.ctx, self.spec["nx"], self.spec["nz"], self.eta, self.chi, out=self.grid)
        if self.mips is not None and self.mips.max_mip != max_mip:
            self.mips = None
        self.mips = api.mips_build(self.ctx, self.grid, self.eta, self.chi, self.W, max_mip, self.iod, self.iod,
                                   0.25, out=self.mips)

    def solve(self):
        api.formal_solve_hdda(self.ctx, self.grid, self.mips, self.dirs, self.w, J=self.J, band=DISTANCE_LIMITS)

    def item(self):
        return api.batch_item(self.grid, self.mips, self.dirs_dev, self.w_dev, self.J, band=DISTANCE_LIMITS)

    def dense_seg_lambda(self):
        """Full-resolution voxel segments x wavelengths of this atmosphere's probes (one plain pass)."""
        g = self.grid
        act = torch.nonzero(g.block_offset >= 0).reshape(-1)
        bx, bz = act % g.nbx, act // g.nbx
        loc = torch.arange(256, device="cuda")
        cells = ((bz[:, None] * 16 + loc[None, :] // 16) * g.nx + bx[:, None] * 16 + loc[None, :] % 16)
        cells = cells.reshape(-1).to(torch.int32)
        planes = api.pack_planes(self.ctx, self.eta, self.chi, self.W)
        _, _, seg = api.formal_solve_dense(self.ctx, g.nx, g.nz, self.spec["n_lambda"], self.W, planes, self.dirs,
                                           self.w, probes=cells, count_segments=True)
        return int(seg.item()) * self.W


def batch_report(scale=1.0, n_atm=24, W=8, iod=1e30, seed=None, reps=3, tune_iod=True):
    import synth
    ctx = api.Context(0)
    specs = synth.batch_specs(n_atm, scale=scale) if seed is None else synth.batch_specs(n_atm, seed=seed, scale=scale)
    atms = [Atmosphere(ctx, sp, W, iod) for sp in specs]
    torch.cuda.synchronize()
    dense = [a.dense_seg_lambda() for a in atms]
    items = [a.item() for a in atms]
    tuned = tune_batch(ctx, items, W, reps=reps)
    cfg = tuned["best"]
    ctas = cfg["ctas"]
    queue = torch.zeros(1, dtype=torch.int32, device="cuda")
    # sequential: one launch per atmosphere (solve only, with the tuned walk), and the whole step
    def sequential():
        ctx.set_traversal(WALKS[cfg["walk"]])
        for a in atms:
            a.solve()
        ctx.set_traversal(api.TRAVERSAL_PER_BATCH)
    t_seq = _time(sequential, reps)
    t_pers = _time(lambda: run_config(ctx, items, W, cfg, queue=queue), reps)
    t_pers_default = _time(lambda: run_config(ctx, items, W, tuned["default"], queue=queue), reps)

    def whole_step():
        for a in atms:
            a.build()
        run_config(ctx, items, W, cfg, queue=queue)

    t_step_eager = _time(whole_step, reps)
    # capture the whole step in a CUDA graph (the library calls enqueue on the capture stream)
    g = torch.cuda.CUDAGraph()
    old = ctx.stream
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        ctx.set_stream(s)
        whole_step()          # warm up on the side stream (kernel attributes, lazy loading)
        s.synchronize()
        with torch.cuda.graph(g, stream=s):
            whole_step()
    ctx.set_stream(old)
    torch.cuda.current_stream().wait_stream(s)
    t_graph = _time(g.replay, reps)
    done, start = run_config(ctx, items, W, cfg, queue=queue, timing=True)
    ctx.check()
    per_atm_ms = ((done.cpu().numpy() - int(start.item())) / 1e6).tolist()
    total_dense = float(sum(dense))
    return {
        "workload": f"{n_atm} independent sparse static-line atmospheres (scale {scale}), VLM mip 0-3, "
                    f"IoD threshold {iod:g}, distance limits {DISTANCE_LIMITS}, W={W}",
        "atmospheres": specs,
        "dense_seg_lambda": dense,
        "tuning": tuned,
        "sequential_solve_ms": t_seq,
        "persistent_solve_ms": t_pers,
        "persistent_default_config_ms": t_pers_default,
        "persistent_speedup_vs_sequential": t_seq / t_pers,
        "tuned_speedup_vs_default_config": t_pers_default / t_pers,
        "step_eager_ms": t_step_eager,
        "step_graph_ms": t_graph,
        "aggregate_seg_lambda_per_s": {"sequential": total_dense / (t_seq / 1e3),
                                       "persistent": total_dense / (t_pers / 1e3),
                                       "graph_step": total_dense / (t_graph / 1e3)},
        "per_atmosphere_done_ms": per_atm_ms,
        "threshold_tuning": tune_threshold(ctx, atms, W, cfg, reps=reps) if tune_iod else None,
    }


def main(argv=None):
    ap = argparse.ArgumentParser()
    ap.add_argument("--scale", type=float, default=1.0)
    ap.add_argument("--n-atm", type=int, default=24)
    ap.add_argument("--reps", type=int, default=3)
    ap.add_argument("--out", default=None)
    args = ap.parse_args(argv)
    rep = batch_report(scale=args.scale, n_atm=args.n_atm, reps=args.reps)
    s = json.dumps(rep)
    if args.out:
        with open(args.out, "w") as f:
            f.write(s + "\n")
    print(s)


if __name__ == "__main__":
    sys.exit(main())
