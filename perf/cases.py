"""Measured workloads of the scoring library, through its Python entry points.

Two kinds of pass.  A "fleet" pass is a monitor at work: some calls of Guard.ingest, each followed by
Guard.score (and, where asked for, Guard.node_verdict), on a context that has been running before, or on one
that starts over with every pass.  A "sweep" pass is one qualification of repeated benchmark results.  Fleet
telemetry and sweep results come from the package's own seeded generators; the named sizes are those of its
workload configurations and tests, or lie between them.
"""
import math

import torch

from paper_2605_17879_b200 import guard, synth

# What a fleet case may leave out.
#   in_place   the producer has written the telemetry into the ring (else ingest copies it there)
#   deferred   evaluations are left running beside the next ingest and joined at the end of the pass
#   step_stats ingest also returns every step's cross-rank median and MAD
#   nodes      every evaluation is folded into node verdicts
#   timers     values as coarse timers and counters report them: whole milliseconds, tokens/s, TFLOP/s
#   restart    every pass starts over on an empty window (an incident replayed), else the monitor goes on
FLEET = dict(kind="fleet", in_place=False, deferred=False, step_stats=False, nodes=False, timers=False, restart=False)


def listed():
    return [
        # One call pair of a small job: a block the length of the window, 64 ranks (the tiny configuration).
        dict(FLEET, name="tiny_block", ranks=64, metrics=4, W=50, topk=8, block=50, calls=1),
        # A mid-sized job scored block by block, in the pipeline mode (the medium configuration).
        dict(FLEET, name="medium_blocks", ranks=1024, metrics=8, W=100, topk=16, block=100, calls=4, in_place=True,
             deferred=True),
        # The large configuration: the benchmark's own pass, four blocks of it.
        dict(FLEET, name="large_blocks", ranks=16384, metrics=8, W=200, topk=64, block=200, calls=4, in_place=True,
             deferred=True),
        # An incident replayed on an empty context, with every step's baseline returned; a ragged fleet.
        dict(FLEET, name="replay", ranks=12345, metrics=8, W=180, topk=33, block=180, calls=1, step_stats=True, restart=True),
        # Blocks of a fleet wider than the large configuration; each block is half of the window.
        dict(FLEET, name="wide_blocks", ranks=24000, metrics=8, W=100, topk=64, block=50, calls=2, deferred=True),
        # Twice as many indicators per rank, windows twice as long as the blocks.
        dict(FLEET, name="many_metrics", ranks=4096, metrics=16, W=120, topk=32, block=60, calls=2, in_place=True),
        # The streaming configuration: a step at a time, an evaluation after every step.
        dict(FLEET, name="stream_wide", ranks=32768, metrics=8, W=200, topk=64, block=1, calls=6, deferred=True),
        # A monitor that acts on every step as it comes: one step, one evaluation, node verdicts.
        dict(FLEET, name="stream_nodes", ranks=2048, metrics=8, W=100, topk=16, block=1, calls=1, nodes=True),
        # A window of hours, polled a tenth of it at a time.
        dict(FLEET, name="long_window", ranks=1024, metrics=8, W=1000, topk=16, block=100, calls=1),
        # Telemetry with the resolution of real timers and counters: many ranks report the same value.
        dict(FLEET, name="coarse_timers", ranks=8192, metrics=8, W=100, topk=64, block=100, calls=1, timers=True),
        # Acceptance of a new rack: few GPUs, few repetitions.
        dict(kind="sweep", name="sweep_rack", nodes=37, gpus_per_node=8, reps=33, metrics=6),
        # The node-sweep configuration.
        dict(kind="sweep", name="sweep_fleet", nodes=2048, gpus_per_node=8, reps=200, metrics=6),
    ]


def _log_uniform(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    if rng.random() < 0.2:
        nodes, reps, metrics = _log_uniform(rng, 8, 2048), _log_uniform(rng, 20, 250), rng.choice([4, 5, 6, 6, 8])
        while nodes * 8 * reps * metrics > 20_000_000:
            nodes //= 2
        return dict(kind="sweep", nodes=nodes, gpus_per_node=8, reps=reps, metrics=metrics)
    ranks, metrics = _log_uniform(rng, 64, 32768), rng.choice([3, 4, 4, 6, 8, 8, 8, 12, 16])
    if rng.random() < 0.6:
        ranks = max(64, ranks // 8 * 8)
    case = dict(FLEET, ranks=ranks, metrics=metrics, topk=min(ranks, _log_uniform(rng, 8, 64)))
    way = rng.random()
    if way < 0.35:      # a step (or a few) at a time
        case.update(W=_log_uniform(rng, 40, 240), block=rng.choice([1, 1, 1, 2, 4]), calls=rng.choice([1, 2, 4]),
                    deferred=rng.random() < 0.5, nodes=ranks % 8 == 0 and rng.random() < 0.5)
    elif way < 0.9:     # block by block, or one block on an empty context
        W = _log_uniform(rng, 40, 240)
        case.update(W=W, block=max(8, rng.choice([W, W, W // 2, W // 3])), calls=rng.choice([1, 2, 3]),
                    in_place=rng.random() < 0.5, deferred=rng.random() < 0.5, step_stats=rng.random() < 0.2,
                    timers=rng.random() < 0.15, restart=rng.random() < 0.15)
    else:               # a long window
        case.update(W=_log_uniform(rng, 300, 1500), block=_log_uniform(rng, 20, 150), calls=1)
    # coarse values and other numbers of metrics cost several times as much per value: no more than their listed cases
    most = 25_000_000 if metrics in (4, 8) and not case["timers"] else 6_000_000
    while case["ranks"] * metrics * case["block"] * case["calls"] > most or case["ranks"] * metrics * case["W"] > 40_000_000:
        case["ranks"] = max(64, case["ranks"] // 16 * 8)
    case["topk"] = min(case["topk"], case["ranks"])
    return case


def _telemetry(case, steps, seed):
    R, M = case["ranks"], case["metrics"]
    cfg = synth.FleetConfig("case", ranks=R, steps=steps, metrics=M, sigma=0.03, seed=seed, W=case["W"], k=1, topk=1,
                            block=case["block"], node_sigma=0.005, n_persistent=max(1, R // 1000), persistent_lo=1.05,
                            persistent_hi=1.5, spike_p=0.002, spike_lo=2.0, spike_hi=5.0, n_ramp=max(1, R // 1000),
                            ramp_len=max(1, steps), ramp_start_max=steps // 2, heavy_tail=0.01, stall_p=1e-4)
    x = synth.fleet_tensor(cfg, device="cuda", chunk=64)
    if case["timers"]:
        whole = torch.tensor([m in (3, 7) for m in range(M)], device="cuda")
        x = torch.where(whole, torch.round(x), torch.round(x * 1000.0) * 0.001)
    return x


def _prepare_fleet(case, seed):
    R, M, W, B, calls = (case[k] for k in ("ranks", "metrics", "W", "block", "calls"))
    # enough telemetry that no window holds a step twice, in whole passes
    per_pass = B * calls
    steps = per_pass if case["restart"] else per_pass * max(2, -(-(W + 8) // per_pass))
    capacity = max(W, steps) if case["in_place"] else max(W + 2 * B, 512 if B == 1 else 0)
    g = guard.Guard(R, M, W, max(1, (3 * W) // 5), dir=synth.fleet_dir(M), capacity=capacity, topk=case["topk"])
    g.set_deferred(case["deferred"])
    data = _telemetry(case, steps, seed)
    if case["in_place"]:
        ring = g.ring_reserve(steps)
        ring.copy_(data)
        data = ring
    state = {"g": g, "case": case, "at": 0, "blocks": [data[t:t + B] for t in range(0, steps, B)],
             "out": [g.alloc_outputs() for _ in range(calls)], "stats": None, "nodes": None}
    if case["step_stats"]:
        state["stats"] = [tuple(torch.empty((B, M), dtype=torch.float32, device="cuda") for _ in range(2)) for _ in range(calls)]
    if case["nodes"]:
        state["nodes"] = [{"node_flag": torch.empty(R // 8, dtype=torch.uint8, device="cuda"),
                           "node_tier": torch.empty(R // 8, dtype=torch.uint8, device="cuda"),
                           "node_stall": torch.empty(R // 8, dtype=torch.uint16, device="cuda")} for _ in range(calls)]
    if not case["restart"]:
        # the monitor has been running: the window is full and the evaluations have settled
        first = max(0, W // B - 1) if B <= 8 else 0
        for b in range(first):
            g.ingest(state["blocks"][b])
        for b in range(first, len(state["blocks"])):
            g.ingest(state["blocks"][b])
            g.score(state["out"][0])
        g.join()
    return state


def _prepare_sweep(case, seed):
    cfg = synth.SweepConfig(nodes=case["nodes"], gpus_per_node=case["gpus_per_node"], reps=case["reps"],
                            metrics=case["metrics"], seed=seed)
    S = synth.sweep_tensor(cfg, device="cuda")
    G, M = cfg.gpus, cfg.metrics
    kw = dict(dir=synth.sweep_dir(M), thr=3.5, floor_rel=1e-4, floor_abs=synth.sweep_floor_abs(M), pct_ppm=cfg.pct_ppm)
    size = int(guard.lib().guard_sweep_workspace_bytes(G, cfg.reps, M))
    out = {"gpu_med": torch.empty((G, M), device="cuda"), "fleet_med": torch.empty(M, device="cuda"),
           "fleet_mad": torch.empty(M, device="cuda"), "fleet_cut": torch.empty(M, device="cuda"),
           "fail_mask": torch.empty(G, dtype=torch.uint32, device="cuda"),
           "gpu_pass": torch.empty(G, dtype=torch.uint8, device="cuda"),
           "node_pass": torch.empty(cfg.nodes, dtype=torch.uint8, device="cuda"),
           "status": torch.zeros(1, dtype=torch.uint32, device="cuda")}
    return {"case": case, "S": S, "kw": kw, "ws": torch.empty(size, dtype=torch.uint8, device="cuda"), "out": out}


def prepare(case, seed):
    return (_prepare_sweep if case["kind"] == "sweep" else _prepare_fleet)(case, seed)


def run(state):
    case = state["case"]
    if case["kind"] == "sweep":
        return guard.sweep_qualify(state["S"], case["nodes"], case["gpus_per_node"], workspace=state["ws"],
                                   out=state["out"], **state["kw"])
    g, blocks, stats, nodes = state["g"], state["blocks"], state["stats"], state["nodes"]
    if case["restart"]:
        g.reset()
        state["at"] = 0
    at = state["at"]
    for i, out in enumerate(state["out"]):
        if stats:
            g.ingest(blocks[at], *stats[i])
        else:
            g.ingest(blocks[at])
        g.score(out)
        if nodes:
            g.node_verdict(nodes[i])
        at += 1
    state["at"] = at % len(blocks)
    if case["deferred"]:
        g.join()
    return [state["out"], stats, nodes]


def work(case):
    """Telemetry read once (and stored once where ingest copies it), every result written once."""
    M = case["metrics"]
    if case["kind"] == "sweep":
        G = case["nodes"] * case["gpus_per_node"]
        return {"bytes": 4 * G * case["reps"] * M + G * (4 * M + 5) + case["nodes"] + 12 * M, "flops": 0}
    R, calls = case["ranks"], case["calls"]
    cells = case["block"] * calls * R * M
    result = R * (10 * M + 6) + 8 * M + 8 * case["topk"]
    if case["step_stats"]:
        result += 8 * M * case["block"]
    if case["nodes"]:
        result += 4 * (R // 8)
    return {"bytes": cells * (4 if case["in_place"] else 8) + calls * result, "flops": 0}


def tolerance(case):
    """Everything is a selection, a count, or single float32 operations in a fixed order."""
    return "exact"
