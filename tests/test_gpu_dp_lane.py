"""The one-pair-per-lane DP (dp_lane.cu) against the oracle: bands from 0 over the group-of-four and word edges to the
widest, ties between gap states (gap open 0, equal costs), reads shorter and longer than the band, batches around a
warp, thresholds that differ from pair to pair, and costs past its range (which the other kernel takes)."""
import numpy as np
import pytest

import gen
from devutil import assert_same, device_results, oracle_results
from test_gpu_ring import _mixed

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def aligner():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2208_01243_gb300 as aim
    al = aim.Aligner(0, 512 << 20)
    yield al
    al.close()


@pytest.mark.parametrize("band", [0, 1, 2, 3, 7, 8, 15, 16, 25, 31, 32, 47, 63, 64, 90, 127])
@pytest.mark.parametrize("algo,penalties", [("edit", (0, 1, 0, 1)), ("gotoh", (0, 4, 6, 2)), ("gotoh", (0, 1, 0, 1)),
                                            ("gotoh", (0, 3, 0, 2)), ("gotoh", (0, 2, 5, 1))])
def test_lane_dp_matches_oracle(aligner, algo, penalties, band):
    """(Batches under 27 pairs per SM take the other kernel: the pairs are repeated past that.)"""
    lengths = [1, 2, 15, 16, 17, 31, 33, 64, 100, 161]
    p = _mixed(lengths, 100 * band + len(penalties) + penalties[1])
    p = gen.concat([p, gen.from_strings([b"", b"ACGT", b"", b"A" * 70], [b"", b"", b"ACG", b"A" * 75])])
    rng = np.random.default_rng(band)
    most = 40
    per_pair = rng.integers(0, most + 1, len(p)).astype(np.int32)
    per_pair[::2] = most
    x, o, e = penalties[1:]
    lim = per_pair.astype(np.int64) * (1 if algo == "edit" else max(x, o + e))
    k = 8000 // len(p) + 1
    dev = device_results(gen.concat([p] * k), algo, penalties, most, per_pair=np.tile(per_pair, k), band=band,
                         aligner=aligner)
    want = oracle_results(p, penalties, lim, band=band)
    assert_same(dev, want, what=f"{algo} {penalties}, band {band}")
    assert np.array_equal(dev[0], np.tile(dev[0][:len(p)], k)) and np.array_equal(dev[3], np.tile(dev[3][:len(p)], k))


@pytest.mark.parametrize("count", [1, 33, 8000, 8001, 8031])
@pytest.mark.parametrize("algo,penalties", [("edit", (0, 1, 0, 1)), ("gotoh", (0, 4, 6, 2))])
def test_lane_dp_batches_and_rejections(aligner, algo, penalties, count):
    """Batches around a warp; most pairs unrelated, so lanes and whole warps stop early."""
    w = gen.Workload("lane_dp", 17, count, 80, 300, 0.02, 0.08, 0.6, algo, penalties, 12)
    p = gen.generate(w)
    unit = 1 if algo == "edit" else 8
    dev = device_results(p, algo, penalties, 12, band=20, aligner=aligner)
    assert_same(dev, oracle_results(p, penalties, np.full(len(p), 12 * unit, np.int64), band=20), what=algo)


def test_lane_dp_leaves_large_costs_to_the_other_kernel(aligner):
    p = _mixed([40, 150], 5)
    pen = (0, 1 << 20, 1 << 19, 1 << 20)
    lim = np.full(len(p), 1 << 24, np.int64)
    k = 8000 // len(p) + 1
    dev = device_results(gen.concat([p] * k), "gotoh", pen, -1, band=12, max_score=1 << 24, aligner=aligner)
    assert_same(dev, oracle_results(p, pen, lim, band=12), what="large costs")


@pytest.mark.parametrize("band", [0, 1, 3, 8, 15, 16, 25, 31, 32, 63, 64, 127])
@pytest.mark.parametrize("algo,penalties", [("edit", (0, 1, 0, 1)), ("gotoh", (0, 4, 6, 2)), ("gotoh", (0, 3, 0, 2))])
@pytest.mark.parametrize("long_share", [0.8, 0.05])
def test_lane_dp_by_evenness(aligner, algo, penalties, band, long_share):
    """The form is chosen by how even the reads are: batches of mostly long reads go to a pair per lane, whatever short,
    empty and one-base pairs are among them, and mostly short ones with a few long reads to a warp per pair."""
    rng = np.random.default_rng(band)
    short = gen.concat([_mixed([1, 2, 15, 16, 17, 31, 33, 64], 300 + band),
                        gen.from_strings([b"", b"ACGT", b"", b"A" * 70], [b"", b"", b"ACG", b"A" * 75])])
    long = _mixed([150, 159, 160, 161, 190], 500 + band)
    k_long = max(int(long_share / (1 - long_share) * len(short) / len(long) * 4), 1)
    p = gen.concat([short] * 4 + [long] * k_long)
    order = rng.permutation(len(p))
    p = gen.from_strings([p.read(i) for i in order], [p.target(i) for i in order])
    most = 40
    per_pair = rng.integers(0, most + 1, len(p)).astype(np.int32)
    per_pair[::2] = most
    x, o, e = penalties[1:]
    lim = per_pair.astype(np.int64) * (1 if algo == "edit" else max(x, o + e))
    k = 6000 // len(p) + 1
    dev = device_results(gen.concat([p] * k), algo, penalties, most, per_pair=np.tile(per_pair, k), band=band,
                         aligner=aligner)
    assert_same(dev, oracle_results(p, penalties, lim, band=band), what=f"{algo} {penalties}, band {band}")
    assert np.array_equal(dev[0], np.tile(dev[0][:len(p)], k)) and np.array_equal(dev[3], np.tile(dev[3][:len(p)], k))
