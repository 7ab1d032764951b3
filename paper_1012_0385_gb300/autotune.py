"""Autotuner for the launches of a domain-schedule context and of a batch.

Knobs, each timed on a short probe with CUDA events:

* the plan, the "tile" of the resident kernel: how many CTAs one sample is
  spread over (1 = whole samples in one CTA; 2..16 = a thread-block cluster,
  i.e. G/cluster columns of 2D sites per CTA) and how many small samples
  share one CTA;
* balanced launches (``asep_set_balance``): whole launches per sample
  group, or persistent CTAs taking (group, chunk of sweeps) items so that
  groups move between SMs -- off, or the chunk length;
* sweeps per launch (``asep_set_launch_sweeps``): the automatic bound (the
  32-bit per-lane hop counters) or shorter launches;
* for a batch: eager persistent launches (``asep_batch_sweep``) or one
  captured CUDA graph replayed per step (``asep_batch_graph``).

The words each thread handles are not a knob: a thread holds one column, the
2D/32 words of a domain pair, and the domain size D is part of the schedule's
definition -- another D gives other (equally valid) trajectories, so it is a
parameter of the job, not of the launch.  No knob changes a result: as a
guard, every probe's lattices must be bit-identical to the first one's
before its timing is accepted.
"""
from __future__ import annotations

import json
import os
from dataclasses import dataclass

import numpy as np

from . import asep as A


@dataclass
class Choice:
    """`cluster` and `samples_per_group` (streamed plans: the tile width) as
    ``asep_set_plan`` takes them; 0, 0 where the automatic plan spreads its
    launches over clusters, which only the automatic plan does."""
    cluster: int
    samples_per_group: int
    ms_per_sweep: float
    launch_sweeps: int = 0  # 0 = automatic
    balance: int = 0  # sweeps per chunk of a balanced launch (0 = off)


def candidates(ctx, sms: int | None = None) -> list[tuple[int, int]]:
    """Plans worth trying: the automatic one, the one-CTA plan with other
    sample counts per CTA, cluster splits that leave >= 32 columns per CTA,
    and the streamed tier at tile widths that leave >= 2 tiles per sample --
    for streamed contexts, and for contexts with fewer samples than the
    device has SMs (`sms`), where one CTA per sample leaves SMs idle and
    tiles spread the samples over all of them, at the cost of one launch
    per phase and a staging pass."""
    info = A.asep_get_info(ctx)
    L, D = info["L"], info["D"]
    G = L // (2 * D)
    out = [(0, 0)]
    if G <= 1024:
        spc = 1
        while spc * G <= 1024 and spc <= info["S"]:
            out.append((1, spc))
            spc *= 2
    for nc in (2, 4, 8, 16):
        if G // nc >= 32:
            out.append((nc, 0))
    few = sms is not None and info["S"] < sms
    if (info["cluster"] == 32 or few) and (L // 32) % 4 == 0:  # streamed: the tile width in columns
        for cols in STREAM_TILE_COLUMNS:
            if 2 * cols <= G:
                out.append((32, cols))
    return out


def _probe(ctx, n_sweeps: int, seed: int) -> tuple[float, np.ndarray]:
    import torch

    stream = torch.cuda.current_stream()
    A.asep_reset(ctx, seed=seed)
    A.asep_sweep(ctx, 2)  # warm the plan's kernel
    A.asep_reset(ctx, seed=seed)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    A.asep_sweep(ctx, n_sweeps)
    e1.record(stream)
    torch.cuda.synchronize()
    words, _ = A.asep_state(ctx)
    return e0.elapsed_time(e1) / n_sweeps, words


def _sm_count() -> int:
    import torch

    return torch.cuda.get_device_properties(torch.cuda.current_device()).multi_processor_count


def launch_sweep_candidates(probe_sweeps: int) -> list[int]:
    """0 (automatic: the whole probe in one launch) and shorter launches."""
    out = [0]
    for k in (2, 4, 8):
        if probe_sweeps // k >= 1 and probe_sweeps // k not in out:
            out.append(probe_sweeps // k)
    return out


BALANCE_CHUNKS = (16, 32, 64)
STREAM_TILE_COLUMNS = (64, 128, 256, 512, 1024)


def autotune(ctx, probe_sweeps: int = 32, seed: int = 12345, launch_sweeps: bool = True,
             balance: bool = True) -> tuple[Choice, list[dict]]:
    """Time every valid plan on `ctx` (its state is reset; re-seed or reset it
    afterwards) and, for plans that keep samples in single CTAs with more
    sample groups than SMs, also balanced launches in chunks of 16/32/64
    sweeps; when balanced launches are among the candidates every candidate
    runs the same longer probe (16 of the longest chunks) so that chunking
    shows.  Every candidate's lattices must equal the first one's.  The
    fastest (plan, chunk) is applied; then, on it and on the same probe, the
    sweeps-per-launch caps are timed and the fastest applied.  Returns the choice and the table
    (rows with knob "plan" or "launch_sweeps")."""
    sms = _sm_count()
    plans = []
    for cluster, spc in candidates(ctx, sms):
        try:
            A.asep_set_plan(ctx, cluster, spc)
        except A.AsepError:
            continue  # does not fit this device
        info = A.asep_get_info(ctx)
        plans.append((cluster, spc, info["cluster"] == 1 and info["groups"] > sms))
    n = 16 * max(BALANCE_CHUNKS) if balance and any(b for *_, b in plans) else probe_sweeps
    table, ref_words, best, best_ms = [], None, None, None
    for cluster, spc, can_balance in plans:
        A.asep_set_plan(ctx, cluster, spc)
        info = A.asep_get_info(ctx)
        for chunk in (0,) + (BALANCE_CHUNKS if balance and can_balance else ()):
            A.asep_set_balance(ctx, chunk)
            ms, words = _probe(ctx, n, seed)
            if ref_words is None:
                ref_words = words
            elif not np.array_equal(words, ref_words):
                raise RuntimeError(f"plan cluster={cluster} spc={spc} balance={chunk} changed the result")
            launched = A.asep_launch_cluster(ctx)
            second = info["tile_columns"] if info["cluster"] == 32 else info["samples_per_group"]
            table.append({"knob": "plan", "cluster": info["cluster"], "launch_cluster": launched,
                          "samples_per_group": info["samples_per_group"], "tile_columns": info["tile_columns"],
                          "balance_chunk_sweeps": chunk or "off", "ms_per_sweep": ms, "probe_sweeps": n,
                          "requested": [cluster, spc]})
            if best is None or ms < best_ms:
                automatic = launched != info["cluster"]  # spread: the plan that info names runs another kernel
                best = Choice(0 if automatic else info["cluster"], 0 if automatic else second, ms, 0, chunk)
                best_ms = ms
        A.asep_set_balance(ctx, 0)
    A.asep_set_plan(ctx, best.cluster, best.samples_per_group if best.cluster in (1, 32) else 0)
    A.asep_set_balance(ctx, best.balance)
    if launch_sweeps:  # on the same probe as the plans: a cap below it must not hide the chunking
        best_cap, cap_ms = 0, None
        for cap in launch_sweep_candidates(n):
            A.asep_set_launch_sweeps(ctx, cap)
            ms, words = _probe(ctx, n, seed)
            if not np.array_equal(words, ref_words):
                raise RuntimeError(f"{cap} sweeps per launch changed the result")
            table.append({"knob": "launch_sweeps", "launch_sweeps": cap or "auto", "ms_per_sweep": ms,
                          "probe_sweeps": n})
            # shorter launches only when measurably faster (1 %): noise must not split long runs
            if cap_ms is None or ms < 0.99 * cap_ms:
                best_cap, cap_ms = cap, ms
        A.asep_set_launch_sweeps(ctx, best_cap)
        best.launch_sweeps = best_cap
    return best, table


def tune_batch_mode(make_contexts, step_sweeps, steps: int = 20) -> tuple[str, list[dict]]:
    """Eager persistent launches or a captured CUDA graph for a batch of
    contexts advanced in equal steps: `make_contexts()` returns fresh
    contexts (same parameters every call), each advanced `steps` times by
    `step_sweeps` (one value per context).  Both modes run the same steps
    from the same start; their final lattices must agree bit for bit.
    Returns "graph" or "eager" and the table (ms per step)."""
    import torch

    stream = torch.cuda.current_stream()
    rows, finals = [], {}
    for mode in ("eager", "graph"):
        ctxs = make_contexts()
        with A.asep_batch_create(max_jobs=max(1, len(ctxs)), max_items=1 << 20) as b:
            # one warm-up step (the graph mode captures here), then the timed steps
            if mode == "eager":
                A.asep_batch_sweep(b, ctxs, step_sweeps)
            else:
                A.asep_batch_graph(b, ctxs, step_sweeps, 1)
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            if mode == "eager":
                for _ in range(steps):
                    A.asep_batch_sweep(b, ctxs, step_sweeps)
            else:
                A.asep_batch_graph(b, ctxs, step_sweeps, steps)
            e1.record(stream)
            torch.cuda.synchronize()
            rows.append({"knob": "batch_mode", "mode": mode, "contexts": len(ctxs),
                         "ms_per_step": e0.elapsed_time(e1) / steps})
            finals[mode] = [A.asep_state(c)[0] for c in ctxs]
        for c in ctxs:
            c.close()
    if not all(np.array_equal(a, b) for a, b in zip(finals["eager"], finals["graph"])):
        raise RuntimeError("graph replay changed the result")
    best = min(rows, key=lambda r: r["ms_per_step"])["mode"]
    return best, rows


class PlanCache:
    """Chosen plans by workload shape, kept in a JSON file."""

    def __init__(self, path: str):
        self.path = path
        self.data = {}
        if os.path.exists(path):
            with open(path) as f:
                self.data = json.load(f)

    @staticmethod
    def key(params) -> str:
        return (f"s{params.schedule}-m{params.model}-d{params.dis_kind}-L{params.L}-D{params.domain_sites}-"
                f"S{params.n_realizations * params.samples_per_real}-f{params.flags}")

    def get(self, params):
        return self.data.get(self.key(params))

    def put(self, params, choice: Choice):
        self.data[self.key(params)] = {"cluster": choice.cluster, "samples_per_group": choice.samples_per_group,
                                       "launch_sweeps": choice.launch_sweeps, "balance": choice.balance,
                                       "ms_per_sweep": choice.ms_per_sweep}
        tmp = self.path + ".tmp"
        with open(tmp, "w") as f:
            json.dump(self.data, f, indent=1, sort_keys=True)
        os.replace(tmp, self.path)
