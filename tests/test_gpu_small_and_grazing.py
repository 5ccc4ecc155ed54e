"""Where the trackers change over: runs small enough for the narrow walk and just
beyond it, hand-overs of the last histories, pieces and statistics batches that do not divide
the run, a batch replayed with another size, and FP64 flights beyond the fixed-point bins.
Counts are exact against the oracle, sums to the parity tests' tolerances."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1708_00765_gb300 as cls  # noqa: E402
from paper_1708_00765_gb300 import workloads  # noqa: E402

COUNTS = {"nR": "nR", "nT": "nT", "nA": "nA", "n_coll": "n_coll", "n_interface": "n_int", "n_reflect": "n_refl",
          "n_events": "n_events", "max_events": "max_events", "n_capped": "n_capped"}


def ocase(p, source=0):
    return oracle.Case(*p[:7], int(p[7]), int(p[8]), source=source)


def assert_parity(g, o):
    for k, ko in COUNTS.items():
        assert g[k] == o[ko], k
    for k in ("sum_t", "sum_t2"):
        assert g[k] == pytest.approx(o[k], rel=1e-12), k
    fo, fg = o["flux"], g["flux"][: o["flux"].shape[0]]
    scale = max(np.abs(fo).max(), 1e-300)
    np.testing.assert_allclose(fg.sum(0), fo.sum(0), rtol=1e-12, atol=1e-14 * scale)
    np.testing.assert_allclose(fg, fo, rtol=1e-10, atol=1e-14 * scale)


def run(p, n, seed, **opts):
    prob = cls.Problem(p)
    for k, v in opts.items():
        prob.set_option(k, v)
    prob.run(n, seed)
    raw = prob.raw_tallies()
    prob.close()
    return raw


# one history, a warp's width and its neighbours, a statistics batch and its neighbours, the narrow walk's
# largest run on 152 SMs and one more (8 and 14 histories for each of 1824 warps)
SIZES = [1, 2, 31, 33, 1023, 1025, 14_592, 14_593, 25_536, 25_537]


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("params,source", [(workloads.ROD_L10, "incident"),
                                           (workloads.suite_case("1c", d=2, nbins=33), "volume"),
                                           (workloads.suite_case("2a", d=3, L=1.0, nbins=7), "incident"),
                                           (workloads.suite_case("3c", d=11, nbins=50), "volume")])
def test_sizes_where_the_walk_changes(params, source, n):
    raw = run(params, n, 17, source=source)
    assert_parity(raw, oracle.run(ocase(params, int(source == "volume")), 17, 0, n))


@pytest.mark.parametrize("schedule", ["history", "event"])
@pytest.mark.parametrize("n", [2_000, 30_000])
def test_long_histories_are_handed_over_exactly(schedule, n):
    """Long histories (c = 0.999): the narrow walk alone, and the last histories of every warp."""
    p = (1.0, 10.0, 0.5, 0.2, 0.999, 0.999, 8.0, 3, 60)
    assert_parity(run(p, n, 5, schedule=schedule), oracle.run(ocase(p), 5, 0, n))


@pytest.mark.parametrize("schedule", ["history", "event"])
def test_outcomes_and_counts_across_the_hand_over_in_fp32(schedule):
    """FP32: outcomes recorded across the hand-over are every history's, and the counters balance."""
    p, n = (1.0, 10.0, 0.5, 0.2, 0.999, 0.999, 8.0, 3, 60), 60_000
    codes = torch.full((n,), 255, dtype=torch.uint8, device="cuda")
    prob = cls.Problem(p)
    prob.set_option("precision", "fp32")
    prob.set_option("schedule", schedule)
    prob.record_outcomes(codes.data_ptr(), n)
    prob.run(n, 3)
    t = prob.raw_tallies()
    prob.close()
    got = torch.bincount(codes.long(), minlength=256).cpu().numpy()
    assert (got[0], got[1], got[2], got[3]) == (t["nR"], t["nT"], t["nA"], t["n_capped"]) and got[:4].sum() == n
    assert t["n_events"] == t["n_coll"] + t["n_interface"] + t["n_reflect"] + t["nR"] + t["nT"]
    assert t["flux"].sum() == pytest.approx(t["sum_t"], rel=1e-6)


@pytest.mark.parametrize("params", [(0.02, 0.02, 50.0, 80.0, 0.9, 0.9, 1.0, 11, 4096),   # grazing flights over many bins
                                    (1e-6, 1e-6, 1e6, 1e6, 1.0, 1.0, 1.0, 3, 4096),
                                    (0.5, 0.5, 1.0, 1.0, 0.5, 0.5, 1e-70, 1, 3),         # beyond FP32's range
                                    (1e-70, 0.0, 1e70, 1e70, 0.5, 0.5, 1e70, 11, 5)])
def test_grazing_flights_and_extreme_scales(params):
    """Flights of 2^9 bin widths and more leave the fixed-point bins; sizes whose FP32 bounds would
    over- or underflow take the exact comparison."""
    n = 20_000
    assert_parity(run(params, n, 29), oracle.run(ocase(params), 29, 0, n))


def test_batch_replayed_with_other_sizes_is_exact():
    """A batch run with several sizes: the captured graph belongs to one size only."""
    params = workloads.batch_sweep(24, seed=7, nbins=20)
    sizes = [2000, 1000, 5000, 64]
    prob = cls.Problem(params, batch=True)
    for n in sizes:
        prob.run(n, 9)
    for k in range(params.shape[0]):
        g = prob.raw_tallies(k)
        o = oracle.run(ocase(params[k]), 9, 0, sum(sizes), case_id=k)
        for key, ko in COUNTS.items():
            assert g[key] == o[ko], (k, key)
        assert g["sum_t"] == pytest.approx(o["sum_t"], rel=1e-12)
    prob.close()


@pytest.mark.parametrize("nbins,nbatch", [(1, 64), (33, 2), (100, 64), (4096, 1024)])
def test_tallies_equal_the_host_normalisation(nbins, nbatch):
    """cls_tallies (reduced on the device) against cls_finalize_raw of the raw tallies."""
    from paper_1708_00765_gb300 import _native
    p = (0.5, 5.0, 2.0, 0.5, 0.5, 0.9, 10.0, 1, nbins)
    prob = cls.Problem(p)
    prob.set_option("nbatch", nbatch)
    prob.run(30_000, 2)
    t = prob.tallies()
    ref = _native.finalize_raw(prob.raw_tallies(), 10.0)
    prob.close()
    for k in ("R", "T", "A", "total_flux", "sigma_total_flux", "track0"):
        assert t[k] == pytest.approx(ref[k], rel=1e-14), k
    np.testing.assert_allclose(t["flux"], ref["flux"], rtol=1e-13)
    np.testing.assert_allclose(t["flux_sigma"], ref["flux_sigma"], rtol=1e-11)


def test_histories_beyond_the_hand_over_buffer_are_walked_to_their_ends():
    """cls_run_noalloc keeps 4096 hand-over slots; every warp of this run ends with four long histories."""
    from paper_1708_00765_gb300 import _native
    p, n = (1.0, 10.0, 0.5, 0.2, 0.999, 0.999, 8.0, 3, 60), 30_000
    flux = torch.zeros((1, 8, 60), dtype=torch.float64, device="cuda")
    stats = torch.zeros((1, 4), dtype=torch.float64, device="cuda")
    counters = torch.zeros((1, 9), dtype=torch.int64, device="cuda")
    rc = _native.run_noalloc(np.array([p]), 0, n, 5, 8, 60, flux.data_ptr(), stats.data_ptr(), counters.data_ptr(),
                             torch.cuda.current_stream())
    assert rc == _native.CLS_OK, cls.strerror(rc)
    torch.cuda.synchronize()
    o = oracle.run(ocase(p), 5, 0, n)
    keys = ("nR", "nT", "nA", "n_coll", "n_int", "n_refl", "n_events", "n_capped", "max_events")
    assert [int(v) for v in counters[0].cpu()] == [int(o[k]) for k in keys]
    assert float(stats[0, 0]) == pytest.approx(o["sum_t"], rel=1e-12)
    np.testing.assert_allclose(flux[0].sum(0).cpu().numpy(), o["flux"].sum(0), rtol=1e-12)


@pytest.mark.parametrize("n", [1, 3])
def test_event_stragglers_keep_their_statistics_in_fp64(n):
    """The event tracker sums t^2 in FP64, in FP32 walks too: of one history it is the square of its track
    length, and of three no less than a third of the squared sum, to FP64 rounding, wherever they ended."""
    p = (1.0, 10.0, 0.5, 0.2, 0.999, 0.999, 8.0, 3, 60)
    for seed in range(8):
        t = run(p, n, seed, precision="fp32", schedule="event")
        assert t["sum_t"] == pytest.approx(sum(t["track"]), rel=1e-14)
        if n == 1:
            assert t["sum_t2"] == pytest.approx(t["sum_t"] ** 2, rel=1e-14)
        else:
            assert t["sum_t"] ** 2 / n * (1 - 1e-14) <= t["sum_t2"] <= t["sum_t"] ** 2 * (1 + 1e-14)
