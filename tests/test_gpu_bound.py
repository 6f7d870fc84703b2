"""Bound passes of batch plans against the oracle: a lane per pair, a warp per pair, and batches that go without.

A bound below a pair's optimum would reject it, and one that only leaves the band reaches could not be met by the exact
pass, so the results must equal the oracle's whatever form the pass takes.  The counts lie on both sides of the lines
between the forms, the lengths from one base to the longest that 32 copies in a warp's shared memory allow and beyond.
"""
import numpy as np
import pytest

import gen
from devutil import assert_same, oracle_results
from test_gpu_batch import AFF, _batched

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("count,lo,hi,frac,band", [(1, 40, 40, 0.2, -1), (700, 1, 300, 0.2, -1), (130, 900, 2500, 0.1, -1),
                                                   (300, 100, 700, 0.15, 9), (26_000, 30, 260, 0.15, -1)])
def test_bound_pass_forms(oracle_lib, gen_lib, mode, count, lo, hi, frac, band):
    w = gen.Workload("bound_forms", 97, count, lo, hi, 0.0, frac, 0.1, "wfa", AFF, None, max_edits_frac=frac)
    p = gen.generate(w)
    me = gen.per_pair_max_edits(w, p)
    outs, _, _ = _batched(p, me, autotune=False, runs=1, bound=mode, band=band)
    idx = np.random.default_rng(3).choice(len(p), min(len(p), 500), replace=False)
    sub = gen.concat([gen.from_strings([p.read(i)], [p.target(i)]) for i in idx])
    lim = me[idx].astype(np.int64) * 8
    assert_same(outs[0], oracle_results(sub, AFF, lim, band=band), idx=idx, what=f"bound mode {mode}, {count} pairs")
