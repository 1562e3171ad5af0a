"""GPU parity: the CUDA library against the CPU oracle, element by element, on the same
seeded buffers, through the C ABI (via the ctypes binding)."""
import numpy as np
import pytest
import torch

from oracle import guard_oracle as go
from paper_2605_17879_b200 import synth
from parity_util import assert_bit_equal, compare_score, run_both, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2605_17879_b200 import build
    build.build_library()


def _rand_fleet(T, R, M, seed, quant=None, slow=True):
    rng = np.random.default_rng(seed)
    s = np.exp(0.03 * rng.normal(size=(T, R, 1)))
    X = s * np.exp(0.015 * rng.normal(size=(T, R, M))) * (1.0 + np.arange(M))
    dirs = [1 if m % 4 != 3 else -1 for m in range(M)]
    for m in range(M):
        if dirs[m] < 0:
            X[..., m] = 100.0 / X[..., m]
    if slow and R > 3:
        for r in (1, R // 2):
            f = 1.25
            for m in range(M):
                X[:, r, m] *= f if dirs[m] > 0 else 1 / f
    if quant:
        X = np.round(X * quant) / quant
    return X.astype(np.float32), dirs


@pytest.mark.parametrize("R,M,W,k,K,T,blocks,cap", [
    (64, 4, 50, 30, 8, 200, [50], None),          # shape of the tiny configuration
    (1, 1, 1, 1, 1, 5, [1], None),                # degenerate: one rank, one metric, window of one
    (2, 3, 4, 2, 2, 9, [1, 2, 3], 5),             # ring wrap, metrics not a multiple of 4
    (7, 5, 6, 3, 7, 20, [4], 9),                  # odd rank count, top-k of all ranks
    (33, 8, 16, 9, 5, 40, [16, 7], 24),
    (600, 2, 10, 6, 3, 25, [10], 16),             # more ranks than threads in a CTA
    (130, 9, 12, 7, 4, 30, [5], 16),              # 32-bit exceedance masks (more than 8 metrics)
    (40, 32, 8, 4, 0, 16, [8], None),             # maximum metric count, no top-k
    (257, 8, 3, 2, 16, 12, [3], 6),
    (96, 4, 33, 17, 8, 70, [33, 2], 40),          # odd window, 2 keys per lane
    (80, 8, 101, 51, 8, 210, [101, 4], 128),      # odd window, 4 keys per lane
    (70, 4, 255, 128, 8, 300, [255, 3], 256),     # odd window, 8 keys per lane, ring wrap
    (50, 3, 77, 40, 5, 160, [77, 1], 90),         # rows not 16-byte aligned: cp.async staging
])
def test_small_fleets_match_oracle(R, M, W, k, K, T, blocks, cap):
    X, dirs = _rand_fleet(T, R, M, seed=R * 1000 + M)
    run_both(X, W, k, K, dirs, blocks, capacity=cap, min_signals=min(2, M))


@pytest.mark.parametrize("R,M,W,T,quant", [
    (4096, 8, 6, 12, None),        # smallest fleet on the bracketed cross-rank path
    (5000, 4, 5, 10, None),        # ragged last chunk
    (4100, 16, 4, 8, None),
    (4096, 32, 3, 6, None),
    (6001, 8, 4, 8, None),         # odd rank count: a single middle element
    (20001, 3, 4, 8, None),        # few columns at a time, wide: a cluster of four CTAs per column; odd rank count (byte-wise mask atomics)
    (17000, 9, 3, 6, None),        # the same with 32-bit exceedance masks
    (32768, 2, 3, 6, 40),          # widest column the clusters hold (8 keys per thread), quantised values (ties)
    (4096, 8, 4, 8, 50),           # quantised: intervals collapse onto tied values, some steps fall back
    (8192, 4, 4, 8, 4),            # very coarse: candidate lists overflow, every step falls back
])
def test_bracketed_cross_rank_path(R, M, W, T, quant):
    X, dirs = _rand_fleet(T, R, M, seed=R + M, quant=quant)
    run_both(X, W, max(1, W // 2), 16, dirs, [W, 1, 2], capacity=2 * W, min_signals=2)


@pytest.mark.parametrize("R,M,B,T,quant", [
    (4096, 8, 12, 24, None),       # smallest fleet on the split path (blocks large enough to leave the column path)
    (5000, 4, 20, 40, None),       # four metrics; ragged last chunk
    (4100, 8, 9, 27, None),        # rank count not a multiple of 16: partial batches
    (16384, 8, 10, 20, None),      # width of the large configuration
    (20000, 8, 9, 9, None),        # beyond the split path's kept-list size: cluster path
    (32768, 8, 9, 9, None),        # cluster path with kept lists too long for its register selection
    (4096, 8, 12, 24, 50),         # quantised: intervals collapse onto tied values
    (8192, 4, 20, 20, 4),          # very coarse: kept lists overflow, every step takes the direct path
])
def test_wide_block_cross_rank_paths(R, M, B, T, quant):
    X, dirs = _rand_fleet(T, R, M, seed=3 * R + M, quant=quant)
    # continuous data must be served by the fast path itself (ragged chunks included), not by the fallback
    run_both(X, B, max(1, B // 2), 16, dirs, [B], capacity=2 * B, min_signals=2,
             max_fallback_steps=0 if quant is None else None)


@pytest.mark.parametrize("R,M,B,W,nblk,cap,quant,deferred", [
    (4096, 8, 50, 50, 4, 100, None, False),     # block = window; two sweep CTAs per step
    (4096, 8, 50, 50, 4, 100, None, True),      # the same in the deferred pipeline (alternating internal streams)
    (4100, 8, 64, 64, 3, 135, None, False),     # last sweep CTA of a step holds 4 ranks; ring wraps inside a block
    (5000, 4, 70, 70, 3, 140, None, True),      # four metrics: 4096-rank slices, ragged second slice
    (4096, 8, 60, 40, 3, 120, None, False),     # window shorter than the block
    (4096, 8, 50, 80, 4, 160, None, False),     # window longer than the block
    (4096, 8, 48, 48, 3, 96, 50, False),        # quantised: intervals collapse onto tied values, steps fall back
    (8192, 4, 48, 48, 2, 96, 4, False),         # very coarse: kept lists overflow, every step takes the direct path
    (16384, 8, 48, 48, 2, 96, None, True),      # width of the large configuration
    (18000, 8, 20, 20, 2, 40, None, False),     # wider than the split path takes: one cluster per step
])
def test_many_step_blocks_match_oracle(R, M, B, W, nblk, cap, quant, deferred):
    """Blocks of many steps on the split cross-rank path (per-step statistics, evaluations, with and without
    per-step outputs, default and deferred mode)."""
    from paper_2605_17879_b200 import guard
    T = nblk * B
    X, dirs = _rand_fleet(T, R, M, seed=11 * R + B + W, quant=quant)
    Xd = torch.from_numpy(X).cuda()
    k = max(1, W // 2)
    o = go.Oracle(R, M, W, k, 16, dir=dirs)
    g = guard.Guard(R, M, W, k, dir=dirs, capacity=cap, topk=16)
    g.set_deferred(deferred)
    bufs = [g.alloc_outputs() for _ in range(nblk)]
    stats = []
    for j in range(nblk):
        smed = torch.empty((B, M), dtype=torch.float32, device="cuda")
        smad = torch.empty((B, M), dtype=torch.float32, device="cuda")
        if deferred and j % 2 == 1:
            g.ingest(Xd[j * B:(j + 1) * B])               # no per-step outputs: the block goes to an internal stream
            stats.append(None)
        else:
            g.ingest(Xd[j * B:(j + 1) * B], smed, smad)
            stats.append((smed, smad))
        g.score(bufs[j])
    g.join()
    assert g.sync_status() == 0
    if quant is None:
        assert g.fallback_steps() == 0
    g.close()
    for j in range(nblk):
        ref_i = o.ingest(X[j * B:(j + 1) * B])
        ref = o.score()
        if stats[j] is not None:
            assert_bit_equal(to_np(stats[j][0]), ref_i["step_med"], "step_med block %d" % j)
            assert_bit_equal(to_np(stats[j][1]), ref_i["step_mad"], "step_mad block %d" % j)
        compare_score(bufs[j], ref, "block %d" % j)


def test_split_path_nonfinite_and_overflowing_deviation():
    from paper_2605_17879_b200 import guard
    R, M, B = 4096, 8, 48
    X, dirs = _rand_fleet(2 * B, R, M, seed=123)
    for m in (2, 7):
        X[..., m] = (X[..., m] / np.median(X[..., m])) * np.float32(1e38)
        for t in range(2 * B):
            X[t, (37 * t + 5) % 997:R:997, m] = np.float32(-3e38)
    g = guard.Guard(R, M, B, B // 2, dir=dirs, capacity=2 * B, topk=8)
    o = go.Oracle(R, M, B, B // 2, 8, dir=dirs)
    Xd = torch.from_numpy(X).cuda()
    for t in range(0, 2 * B, B):
        smed = torch.empty((B, M), dtype=torch.float32, device="cuda")
        smad = torch.empty((B, M), dtype=torch.float32, device="cuda")
        g.ingest(Xd[t:t + B], smed, smad)
        ref_i = o.ingest(X[t:t + B])
        out = g.score()
        assert g.sync_status() == 0                      # finite input whose deviation overflows is not an error
        assert_bit_equal(to_np(smed), ref_i["step_med"], "step_med")
        assert_bit_equal(to_np(smad), ref_i["step_mad"], "step_mad")
        compare_score(out, o.score(), "t=%d" % t)
    assert g.fallback_steps() == 0
    g.reset()
    Xd[B + 7, 4000, 5] = float("inf")                    # a value that is not finite, in the last tile
    g.ingest(Xd[:B])
    assert g.sync_status() == 0
    g.ingest(Xd[B:])
    with pytest.raises(guard.GuardError) as ei:
        g.sync_status()
    assert ei.value.code == -4
    g.close()


def test_wide_block_degenerate_columns():
    # constant, two-valued and single-valued steps inside a wide block: the sample cannot
    # bracket anything, the direct path must take over for those steps only
    X, dirs = _rand_fleet(24, 4096, 8, seed=78)
    X[2] = 1.0
    X[3, ::2] = 1.0
    X[3, 1::2] = 2.0
    X[5] = X[5, :1]
    X[7, :, 3] = 0.0
    X[8, ::3, 1] = -0.0
    X[8, 1::3, 1] = 0.0
    X[8, 2::3, 1] = 1e-30
    run_both(X, 12, 6, 8, dirs, [12], capacity=24)


def test_bracketed_path_constant_and_two_valued_fleets():
    # every element equal: nothing can be bracketed, the direct path must take over and
    # later healthy steps must run on the fast path again with clean counters
    X, dirs = _rand_fleet(9, 4096, 8, seed=77)
    X[2] = 1.0
    X[3, ::2] = 1.0
    X[3, 1::2] = 2.0
    X[5] = X[5, :1]
    run_both(X, 4, 2, 8, dirs, [3], capacity=6)


def test_ties_zero_mad_and_signed_zero():
    # quantised telemetry: many equal values, MAD of zero, floors binding
    X, dirs = _rand_fleet(60, 48, 4, seed=5, quant=20)
    run_both(X, 20, 10, 6, dirs, [20], floor_rel=[0.0, 1e-4, 1e-2, 1e-4], floor_abs=[0.0, 0.0, 0.0, 0.5])
    # values around zero with both signs and both zeros
    rng = np.random.default_rng(6)
    Y = rng.integers(-2, 3, (30, 17, 3)).astype(np.float32)
    Y[Y == 0] = np.where(rng.random((Y == 0).sum()) < 0.5, 0.0, -0.0)
    run_both(Y, 10, 5, 17, [1, -1, 1], [5], min_signals=1, floor_rel=0.0)
    # constant fleet: nothing may be flagged and all scores are zero
    Z = np.full((12, 16, 4), 1.25, np.float32)
    last = run_both(Z, 6, 3, 4, [1, 1, 1, -1], [6])
    assert not last["flags"].any() and not last["mask"].any()


def test_wide_dynamic_range():
    rng = np.random.default_rng(7)
    X = (rng.standard_cauchy((24, 50, 4)) * 10.0 ** rng.integers(-30, 30, (24, 50, 4))).astype(np.float32)
    X[~np.isfinite(X)] = 1.0
    run_both(X, 8, 4, 10, [1, -1, 1, -1], [8], min_signals=1)


def test_in_place_ingest_equals_copy_ingest():
    X, dirs = _rand_fleet(48, 40, 4, seed=8)
    a = run_both(X, 12, 6, 5, dirs, [12], capacity=24, in_place=True)
    b = run_both(X, 12, 6, 5, dirs, [12], capacity=24, in_place=False)
    for key in a:
        assert np.array_equal(a[key], b[key])


def test_overlap_stream_on_and_off_agree():
    """The window medians may run on an internal stream overlapping the preceding ingest; with
    that switched off the same results must come out (and both match the oracle)."""
    from paper_2605_17879_b200 import guard
    X, dirs = _rand_fleet(60, 4500, 8, seed=21)
    Xd = torch.from_numpy(X).cuda()
    res = []
    for overlap in (True, False):
        g = guard.Guard(4500, 8, 20, 10, dir=dirs, capacity=40, topk=8)
        g.set_overlap(overlap)
        outs = []
        for t in range(0, 60, 20):
            g.ingest(Xd[t:t + 20])
            o = g.score()
            g.sync_status()
            outs.append({k: to_np(v).copy() for k, v in o.items()})
        res.append(outs)
        g.close()
    o = go.Oracle(4500, 8, 20, 10, 8, dir=dirs)
    for i, t in enumerate(range(0, 60, 20)):
        o.ingest(X[t:t + 20])
        ref = o.score()
        for key in ("wmed", "fleet_med", "fleet_mad", "counts", "mask", "flags", "tier", "topk_idx"):
            assert_bit_equal(res[0][i][key], ref[key], key)
            assert_bit_equal(res[1][i][key], ref[key], key)


def test_deferred_evaluations_match_oracle():
    """Deferred mode: score() leaves the evaluation running beside the next ingest; every
    evaluation's outputs, read after the next score() / join(), match the oracle, in place and
    copied, including a ring that forces the library to join by itself (capacity < W + block)."""
    from paper_2605_17879_b200 import guard
    R, M, W, B, T = 4500, 8, 20, 20, 120
    X, dirs = _rand_fleet(T, R, M, seed=33)
    Xd = torch.from_numpy(X).cuda()
    o = go.Oracle(R, M, W, 10, 8, dir=dirs)
    refs = []
    for t in range(0, T, B):
        o.ingest(X[t:t + B])
        refs.append(o.score())
    for cap, in_place in ((60, True), (40, False), (30, False)):
        g = guard.Guard(R, M, W, 10, dir=dirs, capacity=cap, topk=8)
        g.set_deferred(True)
        bufs = [g.alloc_outputs() for _ in range(2)]
        got = []
        for i, t in enumerate(range(0, T, B)):
            if in_place:
                slot = g.ring_reserve(B)
                slot.copy_(Xd[t:t + B])
                g.ingest(slot)
            else:
                g.ingest(Xd[t:t + B])
            g.score(bufs[i % 2])                      # also completes the evaluation before it
            if i > 0:
                torch.cuda.current_stream().synchronize()
                got.append({k: to_np(v).copy() for k, v in bufs[(i - 1) % 2].items()})
        g.join()
        g.sync_status()
        got.append({k: to_np(v).copy() for k, v in bufs[(len(refs) - 1) % 2].items()})
        g.close()
        for i, ref in enumerate(refs):
            compare_score({k: torch.from_numpy(v) for k, v in got[i].items()}, ref, "cap=%d eval %d" % (cap, i))
    # a ring too small for the caller to write the next block in place while an evaluation is pending
    g = guard.Guard(R, M, W, 10, dir=dirs, capacity=30, topk=8)
    g.set_deferred(True)
    g.ingest(Xd[:B])
    g.score()
    with pytest.raises(guard.GuardError):
        g.ring_reserve(B)
    g.join()
    g.ring_reserve(10)
    g.close()


def test_long_window_paths():
    # windows too long for the warp-per-series path: 128-, 64- and 32-column staged tiles, and the
    # global-memory fallback
    for W, R in ((300, 40), (500, 24), (1200, 8), (2000, 4)):
        X, dirs = _rand_fleet(W + 7, R, 4, seed=W)
        run_both(X, W, W // 2, 2, dirs, [W, 7], capacity=W + 16, score_every=1)


@pytest.mark.parametrize("R,M,W,cap,gaps,quant", [
    (300, 4, 50, 64, [1], None),                # an evaluation every step: one step enters, one leaves
    (300, 4, 50, 60, [1, 3, 8, 2], None),       # several steps between evaluations, up to the sliding limit
    (64, 8, 200, 256, [1], None),               # window of the streaming configuration (8 keys per lane when rebuilding)
    (40, 3, 7, 9, [1, 2], None),                # tiny odd window, ring barely longer than it
    (96, 4, 33, 40, [1, 9, 1, 1, 20, 1], None), # gaps beyond the limit fall back to whole-window kernels in between
    (128, 4, 40, 64, [1], 25),                  # quantised: ties at the interval ends, lists that overflow
    (50, 2, 30, 32, [1], 3),                    # very coarse: most series cannot hold their ties and rebuild every time
])
def test_sliding_evaluations_match_oracle(R, M, W, cap, gaps, quant):
    from paper_2605_17879_b200 import guard
    T = 3 * W + 20
    X, dirs = _rand_fleet(T, R, M, seed=R + W, quant=quant)
    X[W + 3:W + 9, 5] *= 1.5                     # a level shift: medians leave their intervals
    Xd = torch.from_numpy(X).cuda()
    k = max(1, W // 2)
    for sliding in (True, False):
        g = guard.Guard(R, M, W, k, dir=dirs, capacity=cap, topk=min(8, R), min_signals=min(2, M))
        g.set_sliding(sliding)
        o = go.Oracle(R, M, W, k, min(8, R), dir=dirs, min_signals=min(2, M))
        t, i = 0, 0
        while t < T:
            b = min(gaps[i % len(gaps)], T - t)
            g.ingest(Xd[t:t + b])
            o.ingest(X[t:t + b])
            t += b
            i += 1
            out = g.score()
            assert g.sync_status() == 0
            compare_score(out, o.score(), "sliding=%s t=%d" % (sliding, t))
        rb = g.sliding_rebuilds()
        if sliding and quant is None and max(gaps) <= 8:
            assert R * M <= rb < 0.5 * R * M * i, rb      # state built once, then mostly slid
        if not sliding:
            assert rb == 0
        g.close()


def test_consecutive_evaluations_state():
    X, dirs = _rand_fleet(80, 32, 4, seed=9)
    run_both(X, 10, 6, 4, dirs, [10], n_consec=3)


def test_tiny_configuration_full():
    cfg = synth.paper_configs()["tiny"]
    X = synth.fleet_tensor(cfg).numpy()
    last = run_both(X, cfg.W, cfg.k, cfg.topk, synth.fleet_dir(cfg.metrics), [cfg.block])
    truth = synth.fleet_truth(cfg)
    assert sorted(np.nonzero(last["flags"])[0].tolist()) == sorted(truth["persistent"])


def test_medium_configuration_full():
    cfg = synth.paper_configs()["medium"]
    X = synth.fleet_tensor(cfg, device="cuda").cpu().numpy()
    last = run_both(X, cfg.W, cfg.k, cfg.topk, synth.fleet_dir(cfg.metrics), [cfg.block])
    truth = synth.fleet_truth(cfg)
    # slowdowns well above the per-step noise (sigma = 0.03) must be caught; 1.07x is inside it
    clear = {r for r, f in zip(truth["persistent"], truth["persistent_factor"]) if f >= 1.13}
    assert clear and clear <= set(np.nonzero(last["flags"])[0].tolist())


def test_large_configuration_sampled_blocks():
    """16 384 ranks x 8 metrics, W = 200: two of the hundred 200-step blocks, checked in full
    (tumbling windows with one evaluation per block make every block independent)."""
    cfg = synth.paper_configs()["large"]
    for t0 in (0, 15_800):
        X = synth.fleet_block(cfg, t0, t0 + cfg.block, device="cuda").cpu().numpy()
        run_both(X, cfg.W, cfg.k, cfg.topk, synth.fleet_dir(cfg.metrics), [cfg.block], capacity=cfg.block, in_place=True)


def test_large_configuration_bench_pipeline():
    """The launch configuration bench.py times: 16 384 ranks x 8 metrics, blocks of 200 steps written
    in place, deferred mode (evaluations and consecutive ingests on internal streams), a ring of
    several blocks.  Three consecutive blocks, every evaluation compared in full with the oracle:
    the second and third run the thread-per-series window kernel at full width."""
    from paper_2605_17879_b200 import guard
    cfg = synth.paper_configs()["large"]
    R, M, B, nb = cfg.ranks, cfg.metrics, cfg.block, 3
    dirs = synth.fleet_dir(M)
    g = guard.Guard(R, M, cfg.W, cfg.k, dir=dirs, capacity=nb * B, topk=cfg.topk)
    g.set_deferred(True)
    o = go.Oracle(R, M, cfg.W, cfg.k, cfg.topk, dir=dirs)
    ring = g.ring_reserve(nb * B)
    for j in range(nb):
        synth.fleet_block(cfg, j * B, (j + 1) * B, device="cuda", out=ring[j * B:(j + 1) * B])
    torch.cuda.synchronize()
    bufs = [g.alloc_outputs() for _ in range(nb)]
    for j in range(nb):
        g.ingest(ring[j * B:(j + 1) * B])
        g.score(bufs[j])
    g.join()
    g.sync_status()
    assert g.fallback_steps() == 0
    Xh = ring.cpu().numpy()
    for j in range(nb):
        o.ingest(Xh[j * B:(j + 1) * B])
        compare_score(bufs[j], o.score(), "block %d" % j)
    g.close()


def test_streaming_configuration_prefix():
    """32 768 ranks, one step per ingest into a 512-step ring; every step's cross-rank
    statistics are compared, evaluations at a few steps (an oracle evaluation sorts 262 144
    series)."""
    from paper_2605_17879_b200 import guard
    cfg = synth.paper_configs()["streaming"]
    T = 230
    X = synth.fleet_block(cfg, 0, T, device="cuda")
    Xh = X.cpu().numpy()
    dirs = synth.fleet_dir(cfg.metrics)
    g = guard.Guard(cfg.ranks, cfg.metrics, cfg.W, cfg.k, dir=dirs, capacity=cfg.ring_capacity, topk=cfg.topk)
    o = go.Oracle(cfg.ranks, cfg.metrics, cfg.W, cfg.k, cfg.topk, dir=dirs)
    smed = torch.empty((T, cfg.metrics), dtype=torch.float32, device="cuda")
    smad = torch.empty((T, cfg.metrics), dtype=torch.float32, device="cuda")
    for t in range(T):
        g.ingest(X[t:t + 1], smed[t:t + 1], smad[t:t + 1])
        os_ = o.ingest(Xh[t:t + 1])
        if t in (0, 3, 150, 229):
            gout = g.score()
            g.sync_status()
            compare_score(gout, o.score(), "t=%d" % t)
            assert_bit_equal(to_np(smed[t]), os_["step_med"][0], "step_med")
            assert_bit_equal(to_np(smad[t]), os_["step_mad"][0], "step_mad")
    g.close()


def test_nonfinite_input_sets_sticky_status():
    from paper_2605_17879_b200 import guard
    X, dirs = _rand_fleet(4, 16, 4, seed=10)
    X[2, 5, 1] = np.nan
    g = guard.Guard(16, 4, 4, 2, dir=dirs, topk=2)
    g.ingest(torch.from_numpy(X).cuda())
    with pytest.raises(guard.GuardError) as ei:
        g.sync_status()
    assert ei.value.code == -4
    g.reset()
    X[2, 5, 1] = 1.0
    g.ingest(torch.from_numpy(X).cuda())
    g.score()
    assert g.sync_status() == 0
    g.close()


def test_runtime_argument_errors():
    from paper_2605_17879_b200 import guard
    g = guard.Guard(8, 2, 4, 2, dir=[1, 1], capacity=6, topk=2)
    with pytest.raises(guard.GuardError) as ei:
        g.score()
    assert ei.value.code == -3                       # nothing ingested yet
    with pytest.raises(guard.GuardError):
        g.ingest(torch.ones((7, 8, 2), device="cuda"))   # more steps than the ring holds
    g.ingest(torch.ones((4, 8, 2), device="cuda"))
    with pytest.raises(guard.GuardError):
        g.ring_reserve(3)                            # would wrap: slot 4 + 3 > 6
    assert g.ring_reserve(2).shape == (2, 8, 2)
    assert g.steps_seen == 4
    g.close()


@pytest.mark.parametrize("nodes,gpn,N,M,seed", [(1, 1, 1, 1, 0), (3, 2, 5, 3, 1), (16, 8, 20, 6, 2), (5, 4, 33, 7, 3),
                                               (40, 8, 200, 6, 5),      # warp per GPU, 8 keys per lane, 128-bit loads
                                               (9, 3, 100, 5, 6),       # warp per GPU, blocks not 16-byte aligned
                                               (3, 8, 256, 32, 7),      # widest block a warp stages
                                               (2, 8, 300, 6, 8),       # staged tile of a CTA
                                               (2, 8, 600, 6, 4)])      # too long to stage: selection from global memory
def test_sweep_small_matches_oracle(nodes, gpn, N, M, seed):
    from paper_2605_17879_b200 import guard
    rng = np.random.default_rng(300 + seed)
    G = nodes * gpn
    S = np.round((1.0 + 0.01 * rng.normal(size=(G, 1, M))) * np.exp(0.003 * rng.normal(size=(G, N, M))) * 500) / 500
    S[0] *= 0.8
    S = S.astype(np.float32)
    dirs = [(-1 if m % 3 else 1) for m in range(M)]
    kw = dict(dir=dirs, thr=[3.5] * M, floor_rel=[1e-4] * M, floor_abs=[0.0 if m % 2 else 0.002 for m in range(M)],
              pct_ppm=100_000)
    out = guard.sweep_qualify(torch.from_numpy(S).cuda(), nodes, gpn, **kw)
    ref = go.sweep(S, nodes, gpn, **kw)
    assert int(out["status"].cpu()[0]) == 0
    for key in ref:
        assert_bit_equal(to_np(out[key]), ref[key], key)


def test_sweep_configuration_full():
    from paper_2605_17879_b200 import guard
    cfg = synth.SweepConfig()
    S = synth.sweep_tensor(cfg, device="cuda")
    kw = dict(dir=synth.sweep_dir(cfg.metrics), thr=3.5, floor_rel=1e-4, floor_abs=synth.sweep_floor_abs(cfg.metrics),
              pct_ppm=cfg.pct_ppm)
    out = guard.sweep_qualify(S, cfg.nodes, cfg.gpus_per_node, **kw)
    ref = go.sweep(S.cpu().numpy(), cfg.nodes, cfg.gpus_per_node, **kw)
    assert int(out["status"].cpu()[0]) == 0
    for key in ref:
        assert_bit_equal(to_np(out[key]), ref[key], key)
    bad, which, amount = synth.sweep_tables(cfg)
    failed = set(np.nonzero(ref["gpu_pass"] == 0)[0].tolist())
    strong = set(np.nonzero((bad & (amount > 0.10)).numpy())[0].tolist())
    assert strong <= failed                       # clearly degraded GPUs are caught
    assert len(failed) < 0.08 * cfg.gpus          # and the healthy bulk passes


@pytest.mark.parametrize("R,M,B,T,quant", [
    (64, 4, 50, 100, None),        # a warp per column
    (65, 5, 40, 80, None),         # odd rank count and number of metrics: one metric per CTA, masks bit by bit
    (1024, 8, 40, 80, None),       # two metrics per CTA, eight values per thread
    (2047, 6, 60, 120, None),      # the same with a ragged last round and rows that are not word aligned
    (4096, 16, 24, 48, None),      # 32 values per thread; 32-bit exceedance words
    (8200, 12, 26, 52, None),      # more than 256 threads per CTA
    (16386, 4, 80, 80, None),      # two metrics no longer fit one CTA
    (32768, 3, 12, 24, None),      # the widest column: 1 024 threads, all values in use
    (1024, 8, 40, 80, 40),         # ties: bins with more equal keys than are ranked, ranks in two bins
    (3000, 2, 80, 160, 3),         # a handful of distinct values
])
def test_columns_held_in_registers(R, M, B, T, quant):
    """Blocks whose columns live in registers: the second block starts from the first one's results, and a jump of
    every rank in between makes those miss for half of the steps."""
    X, dirs = _rand_fleet(T, R, M, seed=5 * R + M, quant=quant)
    if T > B:
        X[B + B // 2:] *= np.float32(1.75)
    run_both(X, B, max(1, B // 2), 16, dirs, [B], capacity=2 * B, min_signals=2)


@pytest.mark.parametrize("R,M,B,quant", [
    (4097, 8, 1, None),            # the narrowest column over eight CTAs; a ragged last one
    (4100, 9, 4, None),            # four CTAs per column, several rows
    (8192, 19, 1, None),           # bracketed rows of too many metrics for eight CTAs each; 32-bit exceedance words
    (16385, 4, 2, None),           # eight values per thread
    (32768, 1, 1, None),           # the widest column
    (32768, 6, 6, None),           # the same over four CTAs: sixteen values per thread
    (12345, 5, 1, 40),             # ties: lists of several CTAs, bins of equal keys
])
def test_columns_over_clusters(R, M, B, quant):
    """A few wide rows: columns spread over clusters, bracketed by the row before and (a jump of every rank) missed."""
    T = 3 * B + 4
    X, dirs = _rand_fleet(T, R, M, seed=3 * R + M, quant=quant)
    X[T - B - 2:] *= np.float32(1.75)
    run_both(X, 4, 2, 16, dirs, [B], capacity=max(B, 4), min_signals=2)


@pytest.mark.parametrize("R,M,K,quant", [
    (64, 4, 64, None),             # one warp; every rank is listed
    (129, 3, 1, None),             # groups of single threads; the slowest rank alone
    (130, 3, 100, None),           # more ranks wanted than there are groups for: the exact selection
    (4096, 2, 96, None),           # the widest fleet of one CTA
    (4099, 8, 64, None),           # a cluster of eight CTAs, the last one ragged
    (9000, 18, 33, None),          # a cluster of four
    (32768, 4, 1024, None),        # the longest list
    (3000, 4, 40, 2),              # ties: more equal keys than the gathered list holds, the lowest ranks win
    (20000, 4, 700, 2),            # the same over a cluster
])
def test_slowest_ranks(R, M, K, quant):
    """The top-k list beside the fleet baseline: single steps (a threshold left by the evaluation before; a fleet that
    turns round its order, so that it misses), then a block."""
    X, dirs = _rand_fleet(10, R, M, seed=R + K, quant=quant)
    X[5:] = X[5:, ::-1] * np.float32(0.5)
    run_both(X[:7], 3, 2, K, dirs, [1], capacity=4, min_signals=1)
    run_both(X, 5, 2, K, dirs, [5], capacity=5, min_signals=1)


@pytest.mark.parametrize("R,M,W", [
    (33, 3, 9),                  # rows of bytes that are not word aligned, a ragged last CTA of 32 ranks
    (9, 9, 40),                    # word-wide entries, eight ranks per CTA
    (2371, 9, 40),                 # 32 ranks per CTA
    (9477, 2, 70),                 # 128 ranks per CTA, rows not word aligned
    (40, 2, 33000),                # more exceedances of a rank than a thread's byte counter holds
])
def test_exceedance_counts(R, M, W):
    """k-of-W counts of whole windows, and sliding by a step and by eight, with ranks that exceed in every step."""
    T = W + 9
    rng = np.random.default_rng(R + W)
    X = (1.0 + 0.03 * rng.standard_normal((T, R, M), dtype=np.float32)).astype(np.float32)
    X[:, 5 % R] *= np.float32(2.0)
    X[:, R - 1] *= np.float32(1.5)
    run_both(X, W, W // 2 + 1, 4, [1] * M, [W, 1, 8], capacity=W + 16, min_signals=1)


@pytest.mark.parametrize("nodes,gpn,N,M", [
    (6145, 8, 32, 1),              # the last warp has few series left
    (2400, 7, 33, 3),              # by threads: one repetition in the last round
    (1031, 8, 200, 6),             # a warp per GPU
    (77, 130, 45, 5),              # more GPUs per node than a CTA has threads
    (400, 4, 256, 32),             # the most repetitions and metrics
    (340, 8, 100, 12),             # a warp per GPU, eight lanes of it idle
    (700, 8, 33, 12),              # fleet statistics by clusters of four, the cut beside them
    (600, 8, 20, 20),              # the same without room beside
])
def test_sweep_of_many_series(nodes, gpn, N, M):
    """Many series of repeated results: constant and two-valued series, denormal and huge values, and an outlier that
    makes the spread useless as a bracket; the verdicts follow from the same medians."""
    from paper_2605_17879_b200 import guard
    rng = np.random.default_rng(N + M)
    G = nodes * gpn
    S = (1.0 + 0.02 * rng.standard_normal((G, N, M), dtype=np.float32)).astype(np.float32)
    S[3::50] = S[3::50, :1]
    S[4::50] = np.where(S[4::50] > 1.0, np.float32(1.0), np.float32(0.5))
    S[5::50] *= np.float32(1e-39)
    S[6::50] *= np.float32(1e38) * np.sign(rng.standard_normal((1, N, 1))).astype(np.float32)
    S[7::50, 1] = np.float32(1e30)
    S[8::50, :, 0] *= np.float32(0.7)
    S[9::50] -= np.float32(1.0)
    S[11::50] = np.float32(0.0)
    S[12::50] = np.float32(-0.0)
    S[13::50] = np.copysign(np.float32(0.0), S[13::50] - 1.0)
    S[13::50, 0] = np.float32(0.0)
    S[14::50] = np.copysign(np.float32(0.0), S[14::50] - 1.0)
    S[14::50, 0] = np.float32(-0.0)
    S[10::50] = np.where(np.abs(S[10::50] - 1.0) < 0.01, np.copysign(np.float32(0.0), S[10::50] - 1.0), S[10::50] - 1.0)
    dirs = [-1] * M
    ref = go.sweep(S, nodes, gpn, dir=dirs)
    out = guard.sweep_qualify(torch.from_numpy(S).cuda(), nodes, gpn, dir=dirs)
    assert int(out["status"].cpu()[0]) == 0
    for key in ref:
        assert_bit_equal(to_np(out[key]), ref[key], key)


@pytest.mark.parametrize("R,M,W,B", [
    (61, 3, 7, 7),                 # a metric per CTA; a ring that the third block wraps
    (1024, 8, 64, 16),             # two metrics per CTA, eight values per thread
    (4096, 4, 128, 1),             # single rows; the most values of a window that stays on the caller's stream
    (4097, 4, 128, 1),             # the fewest that does not
    (2048, 6, 12, 12),             # sixteen values per thread: copied in front
])
def test_small_evaluations_in_line(R, M, W, B):
    """Blocks that the counting kernels put into the ring, evaluations on the caller's stream, and a change to deferred
    evaluations and back in between."""
    from paper_2605_17879_b200 import guard
    n = min(-(-W // B), 6) + 4
    X, dirs = _rand_fleet(n * B, R, M, seed=R + W)
    Xd = torch.from_numpy(X).cuda()
    g = guard.Guard(R, M, W, max(1, W // 2), dir=dirs, capacity=2 * W + 3, topk=5, min_signals=1)
    o = go.Oracle(R, M, W, max(1, W // 2), 5, dir=dirs, min_signals=1)
    for i in range(n):
        g.ingest(Xd[i * B:(i + 1) * B].contiguous())
        g.set_deferred(i % 4 >= 2)
        out = g.score()
        g.join()
        o.ingest(X[i * B:(i + 1) * B])
        assert g.sync_status() == 0
        compare_score(out, o.score(), "block %d" % i)
    g.close()


@pytest.mark.parametrize("R,M,W,quant", [
    (70, 3, 1, None),              # one step; a ragged last tile
    (64, 4, 64, None),             # every slot of eight warps of eight values in use
    (45, 5, 65, None),             # one step more: sixteen values per thread
    (40, 8, 129, None),            # 24 values per thread
    (33, 8, 256, None),            # 32 values per thread, all in use
    (24, 4, 257, None),            # sixteen warps
    (16, 4, 1024, None),           # the longest window held in registers
    (11, 3, 1025, None),           # read again in every pass
    (2100, 8, 40, None),           # a first evaluation wide enough for tiles
    (64, 4, 100, 12),              # ties: full bins of equal values, middle ranks in two bins
    (64, 4, 300, 2),               # a handful of distinct values
])
def test_window_tiles(R, M, W, quant):
    """Whole windows by tiles of 32 series: first evaluation, a second window just like it, a jump that leaves every
    range, and values whose differences overflow or are denormal (windowed medians and counts only: the reported score
    of a deviation of 3e38 is beyond float32, in which it is computed)."""
    from paper_2605_17879_b200 import guard
    T = 3 * W + 8
    X, dirs = _rand_fleet(T, R, M, seed=R + W, quant=quant)
    X[2 * W:] *= np.float32(2.5)
    X[:, 2 % R] = np.where(np.arange(T)[:, None] % 2 == 0, np.float32(3e38), np.float32(-3e38))
    X[:, 3 % R] = (np.arange(T)[:, None] * 7919 % 1000).astype(np.float32) * np.float32(1e-42)
    Xd = torch.from_numpy(X).cuda()
    g = guard.Guard(R, M, W, max(1, W // 2), dir=dirs, capacity=W, min_signals=1)
    g.set_sliding(False)
    o = go.Oracle(R, M, W, max(1, W // 2), 0, dir=dirs, min_signals=1)
    t = 0
    for B in (W, W, W, min(W, 8)):
        g.ingest(Xd[t:t + B].contiguous())
        o.ingest(X[t:t + B])
        t += B
        out, ref = g.score(), o.score()
        assert g.sync_status() == 0
        for key in ("wmed", "fleet_med", "fleet_mad", "counts", "mask", "flags", "tier"):
            assert_bit_equal(to_np(out[key]), ref[key], "t=%d %s" % (t, key))
    g.close()


@pytest.mark.parametrize("R,M,W", [
    (16385, 4, 32),                # two keys per lane where the interval misses; a CTA of four series
    (9001, 8, 101),
    (22000, 3, 256),               # the longest window of the path
])
def test_window_threads(R, M, W):
    """Many series, whole windows, a thread each from the second evaluation on: series about zero, with zeros of both
    signs at their middle, very small and very large ones, ties, and a fourth window that leaves every interval."""
    X, dirs = _rand_fleet(5 * W, R, M, seed=R + W)
    X[:, 1::40] -= np.float32(1.0)
    X[:, 2::40] = np.where(np.abs(X[:, 2::40] - 1.0) < 0.01, np.copysign(np.float32(0.0), X[:, 2::40] - 1.0), X[:, 2::40] - 1.0)
    X[:, 3::40] *= np.float32(1e-25)
    X[:, 4::40] *= np.float32(1e20)
    X[:, 5::40] = np.round(X[:, 5::40] * np.float32(40.0)) / np.float32(40.0)
    X[:, 6::40] = np.where(X[:, 6::40] > 1.0, X[:, 6::40], np.float32(1e-40))
    X[3 * W:] *= np.float32(1.5)
    run_both(X, W, max(1, W // 2), 8, dirs, [W], capacity=W)


@pytest.mark.parametrize("R,M,B,thr,deferred", [
    (4097, 8, 20, 3.5, False),     # exceedance rows that are not word aligned; a last strip of one rank
    (4611, 4, 33, 3.5, True),      # four metrics, odd rank count
    (12345, 8, 20, 3.5, True),     # a sample of every twelfth run
    (32767, 4, 20, 3.5, False),    # the widest fleet, odd
    (4096, 8, 20, 0.5, False),     # a threshold inside the MAD's band: every column is recomputed
    (8192, 8, 20, 1.3, False),     # a low threshold: many possible exceedances, lists of a warp overflow
    (36000, 8, 9, 3.5, False),     # wider than the path takes: a cluster per step
])
def test_one_pass_blocks(R, M, B, thr, deferred):
    """Blocks on the one-pass path: sampled estimates in the first, the previous block's in the second and third, a
    smaller block in between, heavy tails on some ranks."""
    from paper_2605_17879_b200 import guard
    X, dirs = _rand_fleet(3 * B + B // 2, R, M, seed=R + M + B)
    X[:, ::37, 0] *= np.float32(1.4)      # in every step: a block's statistics stay those of the block before
    X[:, 4::59] *= np.float32(0.2)
    Xd = torch.from_numpy(X).cuda()
    g = guard.Guard(R, M, B, max(1, B // 2), dir=dirs, capacity=2 * B, topk=8, thr=thr)
    g.set_deferred(deferred)
    o = go.Oracle(R, M, B, max(1, B // 2), 8, dir=dirs, thr=thr)
    t = 0
    for n in (B, B // 2, B, B):
        out = g.alloc_outputs()
        g.ingest(Xd[t:t + n].contiguous())
        g.score(out)
        g.join()
        assert g.sync_status() == 0
        o.ingest(X[t:t + n])
        compare_score(out, o.score(), "t=%d" % t)
        t += n
    if thr == 3.5 and R <= 32768:
        assert g.fallback_steps() == 0
    g.close()


@pytest.mark.parametrize("R,M,B,thr", [
    (8191, 8, 20, 3.5),            # a metric of a handful of values, recomputed by clusters
    (16384, 4, 40, 3.5),           # the most values per thread of a cluster
    (16385, 4, 18, 3.5),           # wider: sixteen values per thread, clusters only
    (32768, 8, 20, 0.5),           # every column, the widest
    (16384, 8, 45, 0.5),           # every column, a CTA each
])
def test_one_pass_columns_recomputed(R, M, B, thr):
    X, dirs = _rand_fleet(2 * B, R, M, seed=R + B)
    X[:, :, 1] = np.round(X[:, :, 1] * np.float32(20.0)) / np.float32(20.0)
    X[B + 3] *= np.float32(1.5)
    run_both(X, B, max(1, B // 2), 8, dirs, [B], capacity=2 * B, thr=thr)


@pytest.mark.parametrize("R,M,B", [
    (8191, 8, 12),                 # eight values per thread of a cluster's CTA
    (24000, 8, 10),                # sixteen
])
def test_one_pass_columns_recomputed_side_by_side(R, M, B):
    """Deferred blocks with nothing between them: both internal streams recompute columns (a metric of a handful of values,
    steps that jump) at the same step positions at the same time."""
    from paper_2605_17879_b200 import guard
    nblk = 8
    X, dirs = _rand_fleet(nblk * B, R, M, seed=R + B)
    X[:, :, 1] = np.round(X[:, :, 1] * np.float32(20.0)) / np.float32(20.0)
    for j in range(1, nblk):       # other steps jump in every block, some of them at the positions of the block before
        X[j * B + 2] *= np.float32(1.0 + 0.25 * (j % 3))
        X[j * B + (3 + j) % B] *= np.float32(1.5)
    Xd = torch.from_numpy(X).cuda()
    g = guard.Guard(R, M, B, max(1, B // 2), dir=dirs, capacity=nblk * B, topk=8)
    g.set_deferred(True)
    bufs = [g.alloc_outputs() for _ in range(nblk)]
    for j in range(nblk):
        g.ingest(Xd[j * B:(j + 1) * B])
        g.score(bufs[j])
    g.join()
    assert g.sync_status() == 0
    assert g.fallback_steps() > nblk
    g.close()
    o = go.Oracle(R, M, B, max(1, B // 2), 8, dir=dirs)
    for j in range(nblk):
        o.ingest(X[j * B:(j + 1) * B])
        compare_score(bufs[j], o.score(), "block %d" % j)


@pytest.mark.parametrize("nodes,gpn,N,M", [
    (37, 8, 5, 6),                 # the cut by CTAs of its own
    (2048, 8, 33, 5),              # by clusters of its own
    (600, 8, 20, 20),              # the cut after the median, in the same clusters
])
def test_sweep_with_unmeasured_metrics(nodes, gpn, N, M):
    """Metrics that were not measured on all, most or some of the GPUs (NaN): the status says non-finite and nothing else,
    with or without a status word, and the other metrics' results are what they are without them."""
    from paper_2605_17879_b200 import guard
    rng = np.random.default_rng(N + M)
    G = nodes * gpn
    S = (1.0 + 0.02 * rng.standard_normal((G, N, M), dtype=np.float32)).astype(np.float32)
    S[8::50, :, 0] *= np.float32(0.7)
    dirs = [-1] + [1] * (M - 1)
    ref = go.sweep(S, nodes, gpn, dir=dirs)
    X = S.copy()
    X[:, :, 1] = np.nan
    X[rng.random(G) < 0.6, :, 2] = np.nan
    X[rng.random(G) < 0.2, :, 3] = np.nan
    clean = [m for m in range(M) if m not in (1, 2, 3)]
    Xd = torch.from_numpy(X).cuda()
    out = guard.sweep_qualify(Xd, nodes, gpn, dir=dirs)
    bare = {k: torch.zeros_like(v) for k, v in out.items() if k != "status"}
    guard.sweep_qualify(Xd, nodes, gpn, dir=dirs, out=bare)
    assert int(out["status"].cpu()[0]) == 1
    for o in (out, bare):
        assert_bit_equal(to_np(o["gpu_med"])[:, clean], ref["gpu_med"][:, clean], "gpu_med")
        for key in ("fleet_med", "fleet_mad", "fleet_cut"):
            assert_bit_equal(to_np(o[key])[clean], ref[key][clean], key)
        assert_bit_equal(to_np(o["fail_mask"]) & ~np.uint32(14), ref["fail_mask"] & ~np.uint32(14), "fail_mask")
        for key in ("fleet_med", "fleet_mad", "fleet_cut"):   # NaN orders above all numbers
            assert np.isnan(to_np(o[key])[1]), key
        assert np.isnan(to_np(o["fleet_med"])[2]) and np.isnan(to_np(o["fleet_cut"])[3])
        assert np.isfinite(to_np(o["fleet_med"])[3])


@pytest.mark.parametrize("R,M,B,in_place", [(2, 3, 66000, False), (3, 2, 65536, True), (40, 1, 65535 * 2 + 1, False)])
def test_blocks_of_more_steps_than_a_grid_has_rows(R, M, B, in_place):
    X, dirs = _rand_fleet(B + 40, R, M, seed=R + M)
    run_both(X, 30, 10, 1, dirs, [B, 40], capacity=B + 40, in_place=in_place)


def test_small_block_the_kernels_do_not_read():
    """A small block in (pinned) host memory, handed to the C call: copied into the ring by the copy engine, as larger ones
    are; the counting kernels read only what is on their device."""
    import ctypes as C
    from paper_2605_17879_b200 import guard
    R, M, W = 64, 4, 20
    X, dirs = _rand_fleet(2 * W, R, M, seed=4)
    g = guard.Guard(R, M, W, 10, dir=dirs, capacity=2 * W, topk=8)
    o = go.Oracle(R, M, W, 10, 8, dir=dirs)
    host = torch.from_numpy(X).pin_memory()
    for t in (0, W):
        rc = guard.lib().guard_ingest(g._h, host[t:t + W].data_ptr(), W, None, None, guard._stream())
        assert rc == 0, guard.lib().guard_last_error(g._h)
        out = g.score()
        assert g.sync_status() == 0
        o.ingest(X[t:t + W])
        compare_score(out, o.score(), "t=%d" % t)
    g.close()


@pytest.mark.parametrize("R,M,W,B", [(64, 4, 50, 5), (3000, 8, 200, 20), (9000, 8, 50, 20), (20000, 8, 100, 1)])
def test_calls_under_stream_capture(R, M, W, B):
    """An ingest and an evaluation captured into a graph and launched give what the calls give."""
    from paper_2605_17879_b200 import guard
    X, dirs = _rand_fleet(W + 2 * B, R, M, seed=R + B)
    Xd = torch.from_numpy(X).cuda()
    got = []
    for capture in (False, True):
        g = guard.Guard(R, M, W, W // 2, dir=dirs, capacity=W + 4 * B, topk=8)
        out = g.alloc_outputs()
        g.ingest(Xd[:W])
        g.score(out)
        g.ingest(Xd[W:W + B])
        g.score(out)
        block = Xd[W + B:].clone()
        torch.cuda.synchronize()
        if capture:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                g.ingest(block)
                g.score(out)
            graph.replay()
        else:
            g.ingest(block)
            g.score(out)
        assert g.sync_status() == 0
        got.append({k: to_np(v) for k, v in out.items()})
        if capture:
            del graph
        g.close()
    for key in got[0]:
        assert_bit_equal(got[1][key], got[0][key], key)


@pytest.mark.parametrize("scale", [1e-26, 1e-17, 1.0, 1e20, 1e34])
def test_window_threads_serve_values_of_any_size(scale):
    """The thread-per-series path on values in other units (some about zero): equal to the oracle, and as few series left
    to the finishing kernel as in ordinary units."""
    from paper_2605_17879_b200 import guard
    R, M, W = 16400, 4, 40
    X, dirs = _rand_fleet(4 * W, R, M, seed=3)
    X[:, :, 2] -= np.float32(3.0)
    X = (X.astype(np.float64) * scale).astype(np.float32)
    Xd = torch.from_numpy(X).cuda()
    g = guard.Guard(R, M, W, W // 2, dir=dirs, capacity=W, topk=8)
    o = go.Oracle(R, M, W, W // 2, 8, dir=dirs)
    for t in range(0, 4 * W, W):
        g.ingest(Xd[t:t + W])
        out = g.score()
        assert g.sync_status() == 0
        o.ingest(X[t:t + W])
        compare_score(out, o.score(), "t=%d" % t)
    left = g.window_fallbacks()
    assert left["total"] < 3 * R * M // 20, left
    g.close()


@pytest.mark.parametrize("nodes,gpn,N,M", [
    (10923, 1, 33, 3),             # by threads and the finishing kernel: quarters of words; one series in the last
    (1300, 8, 64, 4),              # by a warp per GPU, which sorts every series
    (2500, 8, 40, 8),
])
def test_sweep_series_left_to_the_finishing_kernel(nodes, gpn, N, M):
    """Results that spread over decades: the mean says nothing about the median, and next to no series is served by it."""
    from paper_2605_17879_b200 import guard
    rng = np.random.default_rng(N + M)
    S = np.exp(6.0 * rng.standard_normal((nodes * gpn, N, M), dtype=np.float32)).astype(np.float32)
    dirs = [1 if m % 2 else -1 for m in range(M)]
    ref = go.sweep(S, nodes, gpn, dir=dirs)
    out = guard.sweep_qualify(torch.from_numpy(S).cuda(), nodes, gpn, dir=dirs)
    assert int(out["status"].cpu()[0]) == 0
    for key in ref:
        assert_bit_equal(to_np(out[key]), ref[key], key)


def test_selections_of_evaluations_in_flight_do_not_meet():
    """Fleets wider than the register paths: evaluations close together take the hinted selection on one internal stream,
    the others the full one on another, with the same scratch; deferred ones with nothing between them, then at once."""
    from paper_2605_17879_b200 import guard
    R, M, W, K = 33000, 2, 12, 1000
    gaps = [12, 1, 9, 1, 9, 9, 1, 2, 10, 1, 1, 9, 9, 3]
    X, dirs = _rand_fleet(sum(gaps), R, M, seed=8)
    Xd = torch.from_numpy(X).cuda()
    refs = []
    o = go.Oracle(R, M, W, 4, K, dir=dirs)
    t = 0
    for n in gaps:
        o.ingest(X[t:t + n])
        refs.append(o.score())
        t += n
    for defer in ([True] * len(gaps), [j % 2 == 0 for j in range(len(gaps))]):
        g = guard.Guard(R, M, W, 4, dir=dirs, capacity=sum(gaps), topk=K)
        bufs = [g.alloc_outputs() for _ in gaps]
        t = 0
        for j, n in enumerate(gaps):
            g.set_deferred(defer[j])
            g.ingest(Xd[t:t + n])
            g.score(bufs[j])
            t += n
        g.join()
        assert g.sync_status() == 0
        for j in range(len(gaps)):
            compare_score(bufs[j], refs[j], "evaluation %d" % j)
        g.close()


@pytest.mark.parametrize("R,M,B,quant", [
    (33001, 16, 6, None),
    (33001, 16, 6, 12),            # ties: lists overflow, CTAs give their step up while others of it start
    (33002, 32, 5, 30),
    (40001, 8, 20, 12),            # byte-wide exceedance entries
])
def test_wide_fleets_whose_steps_are_given_up(R, M, B, quant):
    """Fleets wider than the register paths, several CTAs per step: steps given up in the middle of a launch are redone."""
    X, dirs = _rand_fleet(2 * B, R, M, seed=R + M, quant=quant)
    run_both(X, B, max(1, B // 2), 8, dirs, [B], capacity=2 * B)


@pytest.mark.parametrize("R,M,W,deferred", [
    (4500, 8, 80, False), (4500, 8, 80, True),     # medians by tiles on an internal stream, by threads from the second evaluation on
    (33000, 2, 40, False), (33000, 2, 40, True),   # the selection on internal streams, too
    (64, 4, 20, True),                             # a small window
])
@pytest.mark.parametrize("gap", [1, 20])
def test_outputs_follow_what_the_caller_enqueued_before(R, M, W, deferred, gap):
    """The caller's stream still has work on the output buffers when an evaluation (a node verdict) is asked for: its
    results come after that work, not before it."""
    from paper_2605_17879_b200 import guard
    X, dirs = _rand_fleet(W + 3 * gap, R, M, seed=R + gap)
    Xd = torch.from_numpy(X).cuda()
    g = guard.Guard(R, M, W, W // 2, dir=dirs, capacity=W + 3 * gap, topk=8, ranks_per_node=4)
    g.set_deferred(deferred)
    o = go.Oracle(R, M, W, W // 2, 8, dir=dirs)
    out = g.alloc_outputs()
    N = R // 4
    nodes = {"node_flag": torch.empty(N, dtype=torch.uint8, device="cuda"), "node_tier": torch.empty(N, dtype=torch.uint8, device="cuda"),
             "node_stall": torch.empty(N, dtype=torch.uint16, device="cuda")}
    t = 0
    for n in (W, gap, gap, gap):
        g.ingest(Xd[t:t + n])
        o.ingest(X[t:t + n])
        t += n
        torch.cuda._sleep(2_000_000)
        for v in out.values():
            v.view(torch.uint8).fill_(7)
        g.score(out)
        torch.cuda._sleep(2_000_000)
        for v in nodes.values():
            v.view(torch.uint8).fill_(7)
        g.node_verdict(nodes)
        g.join()
        assert g.sync_status() == 0
        compare_score(out, o.score(), "t=%d" % t)
        want = o.node_verdict(4)
        for key in want:
            assert_bit_equal(to_np(nodes[key]), want[key], "t=%d %s" % (t, key))
    g.close()


@pytest.mark.parametrize("R,M,W,drift,quant", [
    (129, 1, 65, 0.02, None),     # the last CTA holds one series; two to four values per lane; medians that walk out of their intervals
    (77, 3, 128, 0.1, None),      # steps so large that the values about the old interval do not hold the new one
    (64, 8, 200, 0.01, None),
    (130, 2, 256, 0.02, 40),      # longest windows; ties at the ends of the values that are sorted
    (33, 4, 90, 0.0, 12),         # lists that fill up
])
def test_sliding_rebuilds(R, M, W, drift, quant):
    from paper_2605_17879_b200 import guard
    T = W + 70
    X, dirs = _rand_fleet(T, R, M, seed=R + W, quant=quant)
    X = (X * (1.0 + drift * np.arange(T) / 10.0)[:, None, None]).astype(np.float32)   # (every median moves the same way)
    X[:, 1, 0] = X[0, 1, 0]                                                         # ... but one, which stays the same number
    g = guard.Guard(R, M, W, W // 2, dir=dirs, capacity=W + 8, topk=8, min_signals=min(2, M))
    o = go.Oracle(R, M, W, W // 2, 8, dir=dirs, min_signals=min(2, M))
    Xd = torch.from_numpy(X).cuda()
    t = W
    g.ingest(Xd[:W])
    o.ingest(X[:W])
    for i in range(70):
        b = 1 + 2 * (i % 7 == 6)
        if t + b > T:
            break
        g.ingest(Xd[t:t + b])
        o.ingest(X[t:t + b])
        t += b
        out = g.score()
        assert g.sync_status() == 0
        compare_score(out, o.score(), "t=%d" % t)
    assert g.sliding_rebuilds() > R * M
    g.close()


@pytest.mark.parametrize("R,M,W,quant", [
    (41, 3, 96, None), (41, 3, 97, None),      # twelve and sixteen values per thread
    (21, 8, 160, None), (21, 8, 161, None),    # twenty and 24
    (33, 4, 192, None), (33, 4, 193, None),    # 24 and 28
    (40, 5, 224, None), (40, 5, 225, None),    # 28 and 32
    (30, 4, 128, 2),                           # more equal values in a thread than it notes
    (30, 4, 17, None), (30, 4, 47, None),      # windows too short for spread values of eight pairs
    (2100, 8, 17, None), (2100, 8, 130, 4),    # ... and first evaluations
])
def test_window_tiles_at_their_edges(R, M, W, quant):
    test_window_tiles(R, M, W, quant)


@pytest.mark.parametrize("nodes,gpn,N,M", [
    (6200, 1, 1, 1),               # one value per series (by a warp per series, as one and two metrics and the smaller ones below)
    (3100, 1, 64, 1), (3083, 1, 256, 2), (2049, 1, 96, 3),
    (1601, 1, 33, 4), (800, 1, 256, 4),                      # rows of eight: five of them, all 32
    (401, 2, 48, 5), (397, 2, 49, 5), (260, 1, 255, 5),      # a whole number of rows, one repetition more, the most
    (601, 1, 40, 6), (603, 1, 41, 6), (211, 1, 200, 6), (160, 1, 256, 6),
    (150, 2, 32, 8), (150, 2, 33, 8), (99, 1, 256, 8),
    (300, 1, 64, 7), (260, 1, 192, 9), (200, 1, 128, 13), (210, 1, 128, 16),   # other numbers of metrics
])
def test_sweep_gpu_by_warp(nodes, gpn, N, M):
    """A warp per GPU: ends of its rows of lanes; constant series, zeros of both signs, two values, many equal ones about the
    middle, an outlier that makes the spread useless, and values near the ends of the range of floats."""
    from paper_2605_17879_b200 import guard
    rng = np.random.default_rng(1000 * N + M)
    G = nodes * gpn
    S = (1.0 + 0.02 * rng.standard_normal((G, N, M), dtype=np.float32)).astype(np.float32)
    S[3::9] = S[3::9, :1]
    S[4::9] = np.where(S[4::9] > 1.0, np.float32(1.0), np.float32(0.5))
    S[5::9] = np.round(S[5::9] * np.float32(100.0)) / np.float32(100.0)
    S[6::27] *= np.float32(1e-39)
    S[7::27] *= np.float32(1e38) * np.sign(rng.standard_normal((1, N, 1))).astype(np.float32)
    S[8::27, N // 2] = np.float32(1e30)
    S[10::27] = np.copysign(np.float32(0.0), S[10::27] - 1.0)
    S[11::27] -= np.float32(1.0)
    S[12::27] = np.where(np.abs(S[12::27] - 1.0) < 0.01, np.copysign(np.float32(0.0), S[12::27] - 1.0), S[12::27] - 1.0)
    S[13::27] = np.exp(200.0 * (S[13::27] - 1.0))
    dirs = [-1 if m % 2 else 1 for m in range(M)]
    ref = go.sweep(S, nodes, gpn, dir=dirs)
    out = guard.sweep_qualify(torch.from_numpy(S).cuda(), nodes, gpn, dir=dirs)
    assert int(out["status"].cpu()[0]) == 0
    for key in ref:
        assert_bit_equal(to_np(out[key]), ref[key], key)
    S[G // 2, N - 1, M - 1] = np.float32("inf")
    out = guard.sweep_qualify(torch.from_numpy(S).cuda(), nodes, gpn, dir=dirs)
    assert int(out["status"].cpu()[0]) & 1


@pytest.mark.parametrize("nodes,gpn,N,M", [
    (3200, 1, 64, 3), (800, 1, 256, 3),                      # ten lanes per series: eight and 32 values each
    (2900, 1, 20, 4), (1800, 1, 33, 4), (240, 1, 256, 4),    # eight lanes: eight values, all 32
    (401, 3, 48, 5), (480, 2, 49, 5), (260, 1, 255, 5),      # a whole number of rows of six, one repetition more, the most
    (1001, 1, 40, 6), (1003, 1, 41, 6), (211, 1, 200, 6), (160, 1, 256, 6),
    (600, 1, 64, 7), (150, 1, 256, 7),                       # 28 lanes in use
    (1000, 1, 32, 8), (500, 2, 33, 8), (120, 1, 256, 8),
    (4200, 1, 16, 9), (360, 1, 192, 9), (500, 1, 128, 10),   # three lanes: sixteen values at least, all 64
    (860, 1, 64, 11), (1600, 1, 33, 12), (370, 1, 128, 13), (700, 1, 63, 14), (1300, 1, 31, 15), (1200, 1, 32, 16), (300, 1, 128, 16),
])
def test_sweep_gpu_by_warp_of_any_metrics(nodes, gpn, N, M):
    """... at the ends of the instances, and enough values that a warp per GPU is taken."""
    test_sweep_gpu_by_warp(nodes, gpn, N, M)


@pytest.mark.parametrize("nodes,gpn,N,M", [
    (10923, 1, 33, 3), (1000, 2, 33, 17),   # quarters of words
    (1500, 2, 64, 20),                      # halves
    (3000, 1, 100, 26),                     # whole words, up to 128 repetitions
    (9100, 1, 33, 18),                      # ... more of them than there are warps
])
def test_sweep_finishing_kernel(nodes, gpn, N, M):
    """Sweeps by threads, whose series a warp per GPU does not take."""
    test_sweep_series_left_to_the_finishing_kernel(nodes, gpn, N, M)


@pytest.mark.parametrize("nodes,gpn,N,M", [(2100, 1, 40, 20), (1100, 2, 200, 16)])   # more metrics or repetitions than a warp holds
def test_sweep_by_threads(nodes, gpn, N, M):
    test_sweep_of_many_series(nodes, gpn, N, M)
    test_sweep_series_left_to_the_finishing_kernel(nodes, gpn, N, M)


@pytest.mark.parametrize("R,M,B", [(16385, 18, 2), (17000, 9, 4), (32768, 20, 1)])
def test_widest_rows_of_four_cta_clusters(R, M, B):
    """More columns than clusters of eight find room for, and more ranks than four CTAs of 256 threads hold."""
    X, dirs = _rand_fleet(3 * B, R, M, seed=R + M)
    run_both(X, 2, 1, 4, dirs, [B], capacity=3 * B)
