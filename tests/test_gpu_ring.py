"""The shared-memory wavefront form (wfa_ring.cu) against the oracle, for every number of lanes per pair: at lengths
around a packed word and around the 10-bit history's limit, at thresholds of one gap up to wide windows, with a band,
with thresholds that differ from pair to pair, and over end diagonals far from 0."""
import os
import subprocess
import sys

import numpy as np
import pytest

import gen
from devutil import assert_same, device_results, oracle_results

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def aligner():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2208_01243_gb300 as aim
    al = aim.Aligner(0, 256 << 20)
    yield al
    al.close()


def _mixed(lengths, seed):
    """Related pairs, unrelated pairs and pairs whose targets are cut short or run on, at each length."""
    rng = np.random.default_rng(seed)
    reads, targets = [], []
    for n in lengths:
        for rate in (0.0, 0.03, 0.1, 1.0):
            r = rng.integers(0, 4, n)
            t = []
            for b in r:
                u = rng.random()
                if u < rate / 3:
                    t += [(b + rng.integers(1, 4)) % 4]
                elif u < 2 * rate / 3:
                    t += [rng.integers(0, 4), b]
                elif u >= rate or rate == 0.0:
                    t += [b]
            for cut in (0, 1, 7):
                reads.append(bytes(b"ACGT"[x] for x in r))
                targets.append(bytes(b"ACGT"[x] for x in t[cut:]))
            reads.append(bytes(b"ACGT"[x] for x in r[: n - n // 8]))
            targets.append(bytes(b"ACGT"[x] for x in t))
    return gen.from_strings(reads, targets)


@pytest.mark.parametrize("lanes", [1, 2, 4, 8, 16, 32, 256])
@pytest.mark.parametrize("penalties,max_edits,band", [((0, 4, 6, 2), 6, -1), ((0, 3, 4, 1), 8, -1),
                                                      ((0, 4, 6, 2), 1, -1), ((0, 2, 3, 1), 12, 5),
                                                      ((0, 4, 4, 4), 9, 0), ((0, 4, 6, 2), 20, 15)])
def test_ring_matches_oracle(aligner, lanes, penalties, max_edits, band):
    import paper_2208_01243_gb300 as aim
    lengths = [1, 15, 16, 17, 31, 32, 33, 63, 64, 97, 150] if max_edits < 20 else [64, 250, 300]
    p = _mixed(lengths, 7 * lanes + max_edits)
    per_pair = np.random.default_rng(lanes).integers(0, max_edits + 1, len(p)).astype(np.int32)
    per_pair[::3] = max_edits
    x, o, e = penalties[1:]
    lim = per_pair.astype(np.int64) * max(x, o + e)
    aim.aim_set_wfa_group(aligner.ctx, lanes)
    try:
        dev = device_results(p, "wfa", penalties, max_edits, per_pair=per_pair, band=band, aligner=aligner)
    finally:
        aim.aim_set_wfa_group(aligner.ctx, 0)
    assert_same(dev, oracle_results(p, penalties, lim, band=band), what=f"ring, {lanes} lanes")


@pytest.mark.parametrize("lanes", [1, 4, 32, 256])
@pytest.mark.parametrize("length,edits", [(1000, 15), (1022, 15), (1023, 15), (1500, 60), (16382, 20), (16383, 20)])
def test_ring_history_forms(aligner, length, edits, lanes):
    """max_length up to 1,022 keeps 10-bit history fields, up to 16,382 source bits in 16-bit words, beyond in 32."""
    import paper_2208_01243_gb300 as aim
    rate = 0.7 * edits / length
    w = gen.Workload("ring_edge", 91, 40 if length < 2000 else 9, length, length, rate, rate, 0.2, "wfa", (0, 4, 6, 2),
                     edits)
    p = gen.generate(w)
    keep = p.target_len <= length
    p = gen.from_strings([p.read(i) for i in np.nonzero(keep)[0]], [p.target(i) for i in np.nonzero(keep)[0]])
    aim.aim_set_wfa_group(aligner.ctx, lanes)
    try:
        dev = device_results(p, "wfa", w.penalties, edits, max_length=length, aligner=aligner)
    finally:
        aim.aim_set_wfa_group(aligner.ctx, 0)
    assert_same(dev, oracle_results(p, w.penalties, np.full(len(p), 8 * edits, np.int64)),
                what=f"ring, {length} bp, {lanes} lanes")


@pytest.mark.parametrize("length,edits", [(9952, 690), (9921, 689), (9920, 690), (9953, 690), (2000, 752)])
def test_ring_shared_memory_around_48_kb(length, edits):
    """16 (W + ceil(length / 32) + 1) bytes of dynamic shared memory for a block per pair, W = 4 edits: 48 KB to the byte
    (beside which the kernel has a few static ones), a step below and a step above.  A process of its own for each: an
    earlier launch of the same kernel would already have asked for more."""
    code = f"""
import numpy as np
import __graft_entry__
__graft_entry__.build()
import gen
from devutil import assert_same, device_results, oracle_results
w = gen.Workload("ring_48k", 5, 3, {length} - 40, {length} - 40, 0.002, 0.002, 0.0, "wfa", (0, 4, 6, 2), 30)
p = gen.generate(w)
dev = device_results(p, "wfa", w.penalties, {edits}, max_length={length}, workspace=1 << 30)
assert_same(dev, oracle_results(p, w.penalties, np.full(len(p), 8 * {edits}, np.int64)), what="48 KB")
"""
    here = os.path.dirname(os.path.abspath(__file__))
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([here, os.path.dirname(here)]))
    r = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]


@pytest.mark.parametrize("length,edits,count,megabytes", [(300, 30, 200, 2), (1000, 50, 120, 8), (1000, 50, 120, 64),
                                                          (2500, 130, 30, 16), (2500, 130, 30, 400)])
def test_ring_short_of_scratch(length, edits, count, megabytes):
    """Workspaces that hold few pairs at once take more lanes for each, up to a block."""
    w = gen.Workload("ring_scratch", 41, count, length - 40, length - 40, 0.7 * edits / length, 0.7 * edits / length, 0.1,
                     "wfa", (0, 4, 6, 2), edits)
    p = gen.generate(w)
    dev = device_results(p, "wfa", w.penalties, edits, max_length=length, workspace=megabytes << 20)
    assert_same(dev, oracle_results(p, w.penalties, np.full(len(p), 8 * edits, np.int64)), what=f"ring, {megabytes} MB")
