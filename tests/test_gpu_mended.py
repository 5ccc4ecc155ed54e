"""Calls that earlier kernels or their host code answered wrongly, each against the oracle: counts
exact, sums to the parity tests' tolerances."""
import json
import os
import tempfile

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1708_00765_gb300 as cls  # noqa: E402
from paper_1708_00765_gb300 import workloads  # noqa: E402
from tests.test_gpu_small_and_grazing import COUNTS, assert_parity, ocase, run  # noqa: E402,F401


def test_a_batch_seed_counts_with_all_its_bits():
    """The captured graph holds the seed's round keys: a seed that differs in bit 63 alone is another seed."""
    params, n = workloads.batch_sweep(6, seed=3, nbins=10), 500
    for seeds in ((5, 5 | 1 << 63), (1 << 63, 0)):
        prob = cls.Problem(params, batch=True)
        for s in seeds:
            prob.run(n, s)
        for k in range(params.shape[0]):
            g = prob.raw_tallies(k)
            parts = [oracle.run(ocase(params[k]), s, i * n, n, case_id=k) for i, s in enumerate(seeds)]
            for key, ko in COUNTS.items():
                want = max(p[ko] for p in parts) if key == "max_events" else sum(p[ko] for p in parts)
                assert g[key] == want, (k, key)
            assert g["sum_t"] == pytest.approx(sum(p["sum_t"] for p in parts), rel=1e-12)
        prob.close()


THICK = [(1.0, 1.0, 1.0, 1.0, 0.5, 0.5, L, 1, 1) for L in (1e5, 1e6, 1e9, 1e12, 1e14, 1e16)] + [
    (1.0, 1.0, 1.0, 1.0, 0.5, 0.5, 1e16, 3, 3),
    (1e12, 1e-3, 1.0, 2.0, 0.0, 0.9, 10.0, 1, 4),       # one material a trillion times as thick as the other
    (0.1, 1e6, 1.0, 1e-9, 0.9, 0.0, 10.0, 11, 50),      # a chord of 1e-9 between ordinary ones
    (1e300, 1e300, 1.0, 1.0, 0.5, 0.5, 1e300, 1, 2),    # no fixed-point unit: every flight in FP64
    (0.5, 5.0, 2.0, 0.5, 0.5, 0.9, 10.0, 1, 4096)]      # the widest mesh


@pytest.mark.parametrize("schedule,n", [("history", 300), ("history", 40_000), ("event", 20_000)])
@pytest.mark.parametrize("params", THICK)
def test_flux_where_a_bin_is_very_many_flights_wide(params, schedule, n):
    """The flux bins hold what the flights deposit, whatever their length in bin widths."""
    assert_parity(run(params, n, 31, schedule=schedule), oracle.run(ocase(params), 31, 0, n))


@pytest.mark.parametrize("schedule,n", [("history", 300), ("history", 40_000), ("event", 20_000)])
@pytest.mark.parametrize("params", THICK)
def test_flux_of_a_thick_volume_source_is_the_track_length(params, schedule, n):
    """Histories born deep inside, where a coordinate does not resolve a flight: the bins sum to the
    track length all the same."""
    raw = run(params, n, 31, source="volume", schedule=schedule)
    o = oracle.run(ocase(params, 1), 31, 0, n)
    for k, ko in COUNTS.items():
        assert raw[k] == o[ko], k
    assert raw["sum_t"] == pytest.approx(o["sum_t"], rel=1e-12)
    assert raw["flux"].sum() == pytest.approx(raw["sum_t"], rel=1e-12)


@pytest.mark.parametrize("batch", [False, True])
def test_runs_of_one_handle_on_several_streams_follow_one_another(batch):
    """Long and short runs in turn on three streams, nothing waited for in between."""
    p = (1.0, 10.0, 0.5, 0.2, 0.999, 0.999, 8.0, 3, 60)
    params = np.array([p, workloads.ROD_L10, p]) if batch else np.array([p])
    streams = [torch.cuda.Stream() for _ in range(3)]
    sizes = [30_000, 500, 4_000, 4_000, 25_000, 100]
    prob = cls.Problem(params if batch else p, batch=batch)
    for i, n in enumerate(sizes):
        prob.run(n, 7, stream=streams[i % 3])
    for k in range(params.shape[0]):
        g = prob.raw_tallies(k)
        o = oracle.run(ocase(params[k]), 7, 0, sum(sizes), case_id=k)
        for key, ko in COUNTS.items():
            assert g[key] == o[ko], (k, key)
        assert g["sum_t"] == pytest.approx(o["sum_t"], rel=1e-12)
        np.testing.assert_allclose(g["flux"].sum(0), o["flux"].sum(0), rtol=1e-12)
    prob.close()


def launches(call):
    """(name, grid, block) of every kernel that `call` launches."""
    from torch.profiler import ProfilerActivity, profile
    for f in (lambda: torch.zeros(8, device="cuda").add_(1), call):  # the first session records nothing
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            f()
            torch.cuda.synchronize()
    with tempfile.TemporaryDirectory() as d:
        path = os.path.join(d, "trace.json")
        prof.export_chrome_trace(path)
        with open(path) as f:
            events = json.load(f)["traceEvents"]
    out = [(e["name"], e["args"]["grid"], e["args"]["block"]) for e in events if e.get("cat") == "kernel"]
    if not out:
        pytest.skip("the profiler records no kernels here")
    return out


@pytest.mark.parametrize("params,batch", [((*workloads.BOX_L10[:8], 37), False), (workloads.batch_sweep(2, seed=1, nbins=21), True)])
def test_autotuner_pilots_run_the_tracker(params, batch):
    """A pilot small enough for the narrow walk still times the tracker's launch shapes.  (These FP64
    boxes' histories are too short for a hand-over, so no other use of the narrow walk is expected.)"""
    prob = cls.Problem(params, batch=batch)
    names = [k for k, _, _ in launches(lambda: prob.autotune(2048 + 16 * batch, seed=12))]
    if batch:
        names += [k for k, _, _ in launches(lambda: prob.autotune_cases(2048, seed=12))]
    prob.close()
    assert any("history_kernel" in k for k in names) and any("event_kernel" in k for k in names)
    assert not any("narrow_kernel" in k for k in names)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_small_runs_keep_to_the_callers_launch_shape(precision):
    """The narrow walk takes no more blocks per SM and threads per block than asked for, says what it took,
    and walks the same histories."""
    p, n = (*workloads.ROD_L10[:8], 29), 900
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    prob = cls.Problem(p)
    prob.set_option("precision", precision)
    prob.run(n, 4)
    assert prob.get_option("blocks_per_sm") == 3  # of 128 threads
    prob.set_option("blocks_per_sm", 1)
    prob.set_option("block", 64)
    kernels = [k for k in launches(lambda: prob.run(n, 4)) if "narrow_kernel" in k[0]]
    assert len(kernels) == 1 and kernels[0][1][0] <= sms and kernels[0][2][0] <= 64, kernels
    assert prob.get_option("blocks_per_sm") == 1
    prob.set_option("blocks_per_sm", 0)
    prob.set_option("block", 32)
    prob.run(n, 4)
    assert prob.get_option("blocks_per_sm") == 12
    g = prob.raw_tallies()
    prob.close()
    assert g["n_histories"] == 3 * n
    if precision == "fp64":
        o = oracle.run(ocase(p), 4, 0, 3 * n)
        for k, ko in COUNTS.items():
            assert g[k] == o[ko], k
        np.testing.assert_allclose(g["flux"].sum(0), o["flux"].sum(0), rtol=1e-12)


@pytest.mark.parametrize("batch", [False, True])
def test_history_runs_wait_for_nothing_on_the_device(batch):
    """Runs that take their hand-over slots, and runs that outgrow them, return while the device is busy with
    other work."""
    params = np.array([workloads.ROD_L10[:8] + (20,)] * 3)
    prob, warm = (cls.Problem(params if batch else params[0], batch=batch) for _ in range(2))
    side, seeds, n = torch.cuda.Stream(), (3, 4, 5), 60_000

    def three(p, stream):
        p.set_option("blocks_per_sm", 1)
        p.run(n, seeds[0], stream)
        p.set_option("blocks_per_sm", 32)  # more warps, more slots
        p.run(n, seeds[1], stream)
        p.set_option("precision", "fp32")
        p.set_option("precision", "fp64")
        p.run(n, seeds[2], stream)

    own = torch.cuda.Stream()
    three(warm, own)  # kernels, streams and graphs are loaded and made at their first use
    torch.cuda.synchronize()
    done = torch.cuda.Event()
    with torch.cuda.stream(side):
        torch.cuda._sleep(2_000_000_000)  # about a second
        done.record()
    three(prob, own)
    assert not done.query()
    torch.cuda.synchronize()
    for k in range(3 if batch else 1):
        g = prob.raw_tallies(k)
        parts = [oracle.run(ocase(params[k]), s, i * n, n, case_id=k) for i, s in enumerate(seeds)]
        for key, ko in COUNTS.items():
            assert g[key] == (max if key == "max_events" else sum)(o[ko] for o in parts), key
        assert g["sum_t"] == pytest.approx(sum(o["sum_t"] for o in parts), rel=1e-12)
    prob.reset()
    prob.run(n, seeds[1], own)
    assert prob.raw_tallies()["nR"] == oracle.run(ocase(params[0]), seeds[1], 0, n)["nR"]
    prob.close()
    warm.close()


def test_a_replayed_graph_starts_from_fresh_counters_and_slots():
    """The second launch of one captured graph (the same size twice), for the tracker with hand-over and for
    the narrow walk: work counters, claimed pieces and hand-over slots are used again."""
    diffusive = (1.0, 10.0, 0.5, 0.2, 0.999, 0.999, 8.0, 3, 60)
    params = np.array([workloads.ROD_L10[:8] + (30,), diffusive, workloads.ROD_L10[:8] + (60,), diffusive])
    sizes = [14_000, 14_000, 600, 600, 14_000]
    prob = cls.Problem(params, batch=True)
    for n in sizes:
        prob.run(n, 9)
    for k in range(params.shape[0]):
        g = prob.raw_tallies(k)
        o = oracle.run(ocase(params[k]), 9, 0, sum(sizes), case_id=k)
        for key, ko in COUNTS.items():
            assert g[key] == o[ko], (k, key)
        for key in ("sum_t", "sum_t2"):
            assert g[key] == pytest.approx(o[key], rel=1e-12), (k, key)
        np.testing.assert_allclose(g["flux"].sum(0)[: int(params[k, 8])], o["flux"].sum(0), rtol=1e-12)
    prob.close()
