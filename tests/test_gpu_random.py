"""Random sequences of calls (sizes, values, options, modes and their changes; ingests of all lengths, copied and in place;
evaluations, node verdicts, resets, states exported and imported) against the CPU oracle: what the library enqueues on streams
of its own must not show in any result."""
import random

import numpy as np
import pytest
import torch

from oracle import guard_oracle as go
from parity_util import assert_bit_equal, compare_score, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2605_17879_b200 import build
    build.build_library()


def _values(kind, T, R, M, rng):
    n, u = rng.standard_normal((T, R, M)), rng.random((T, R, M))
    x = {"levels": (1.0 + 0.1 * rng.random((1, R, M))) * np.exp(0.03 * n),
         "coarse": np.round(20.0 * (1.0 + 0.03 * n)) / 20.0,
         "two": np.where(u < 0.5, 1.0, 2.0),
         "bimodal": np.where(u < 0.5, 1.0, 3.0) + 0.01 * n,
         "zeros": np.where(u < 0.6, 0.0 * n, n),
         "jumps": (1.0 + 0.02 * n) * (1 + np.arange(T) // 7 % 5)[:, None, None],
         "decades": np.exp(10.0 * n), "large": 1e25 * (1.0 + 0.01 * n), "small": 1e-30 * (1.0 + 0.01 * n)}[kind]
    return x.astype(np.float32)


@pytest.mark.parametrize("seed", range(24))
def test_random_calls_match_the_oracle(seed):
    from paper_2605_17879_b200 import guard
    pick = random.Random(seed)
    rng = np.random.default_rng(seed)
    # small fleets, single CTAs, the one-pass path (odd widths too), the paths beyond 32 768 ranks
    R, M = [(pick.randrange(1, 200), pick.randrange(1, 33)), (pick.randrange(200, 4096), pick.choice([2, 4, 7, 8, 16])),
            (pick.randrange(4096, 12000), pick.choice([4, 8])), (32768 + pick.choice([1, 4, 232]), pick.choice([1, 2, 4]))][seed % 4]
    W = pick.choice([pick.randrange(1, 12), pick.randrange(12, 40)] + ([pick.randrange(260, 400)] if R < 200 else []))
    K, spare = min(R, pick.choice([0, 5, 130, 500])), pick.choice([0, 1, 9, W, 2 * W])
    steps = 4 * W + 40
    X = _values(pick.choice(["levels", "levels", "coarse", "two", "bimodal", "zeros", "jumps", "decades", "large", "small"]), steps, R, M, rng)
    kw = dict(dir=[pick.choice([1, -1]) for _ in range(M)], thr=pick.choice([3.5, 1.0, 0.3]), primary=pick.randrange(M),
              min_signals=pick.choice([1, 2]), n_consec=pick.choice([1, 2]))
    o = go.Oracle(R, M, W, max(1, W // 3), K, **kw)
    g = guard.Guard(R, M, W, max(1, W // 3), capacity=W + spare, topk=K, ranks_per_node=1, **kw)
    deferred = pick.random() < 0.7
    g.set_deferred(deferred)
    Xd, t, due = torch.from_numpy(X).cuda(), 0, []

    def check():
        for what, got, want in due:
            if "wmed" in got:
                compare_score(got, want, what)
            for key in want:
                if key in ("step_med", "step_mad", "node_flag", "node_tier", "node_stall"):
                    assert_bit_equal(to_np(got[key]), want[key], what + " " + key)
        due.clear()
    while t < steps:
        op = pick.random()
        if op < 0.08:
            deferred = not deferred
            g.set_deferred(deferred)
        elif op < 0.16:
            pick.choice([g.set_sliding, g.set_row_hints, g.set_overlap])(pick.random() < 0.5)
        elif op < 0.22:
            state = g.state_export()
            torch.cuda.synchronize()
            check()
            g.close()
            g = guard.Guard(R, M, W, max(1, W // 3), capacity=W + spare, topk=K, ranks_per_node=1, **kw)
            g.set_deferred(deferred)
            g.state_import(state)
        B = min(pick.choice([1, 1, 2, 5, W, W + spare]), W + spare, steps - t)
        block = Xd[t:t + B]
        if pick.random() < 0.3:
            try:
                block = g.ring_reserve(B).copy_(block)
            except guard.GuardError:               # the slots wrap around, or are still read
                pass
        stats = [torch.empty((B, M), device="cuda") for _ in range(2)] if pick.random() < 0.3 else [None, None]
        g.ingest(block, *stats)
        ref = o.ingest(X[t:t + B])
        if stats[0] is not None:
            due.append(("steps from %d" % t, {"step_med": stats[0], "step_mad": stats[1]}, ref))
        t += B
        if pick.random() < 0.8:
            due.append(("t=%d" % t, g.score(), o.score()))
            if pick.random() < 0.4:
                due.append(("t=%d" % t, g.node_verdict(), o.node_verdict(1)))
        if pick.random() < 0.15:
            g.join()
            check()
    g.join()
    assert g.sync_status() == 0
    check()
    g.close()
