"""Calls that earlier kernels or their host code answered wrongly, each against the oracle: counts
exact, sums to the parity tests' tolerances."""
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
