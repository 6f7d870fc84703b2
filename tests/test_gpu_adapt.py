"""WFA-adaptive with its state in shared memory (wfa_adapt.cu) against the oracle: batches past its line, at the paper's
costs and others, pruning from tight to none, a band, pairs that outgrow it (aligned again by the other kernel), and
thresholds that differ from pair to pair."""
import numpy as np
import pytest

import gen
import oracle
from devutil import assert_same, device_results

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def aligner():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2208_01243_gb300 as aim
    al = aim.Aligner(0, 2 << 30)
    yield al
    al.close()


@pytest.mark.parametrize("params", [(10, 50), (4, 5), (2, 1), (10, 4000)])
@pytest.mark.parametrize("penalties", [(0, 3, 4, 1), (0, 4, 6, 2), (0, 1, 1, 1)])
@pytest.mark.parametrize("length,count,copies", [(900, 300, 80), (2500, 80, 40)])
def test_adaptive_in_shared_memory(aligner, length, count, copies, penalties, params):
    import paper_2208_01243_gb300 as aim
    w = gen.Workload("adapt_ring", 5, count, length // 4, length, 0.01, 0.08, 0.05, "wfa_adaptive", penalties, None, 0.08)
    p = gen.generate(w)
    me = gen.per_pair_max_edits(w, p)
    lim = np.array([oracle.limit_for(penalties, int(k)) for k in me], np.int64)
    s, f, off, cig, lens = oracle.wfa_adaptive_batch(p, penalties, lim, min_len=params[0], max_dist=params[1])
    want = (s, f, [cig[off[i]:off[i] + lens[i]].astype(np.uint32) for i in range(len(p))])
    # the kernel takes batches that fill the device: the pairs repeated, results the same for every copy
    aim.aim_set_wfa_adaptive(aligner.ctx, *params)
    try:
        dev = device_results(gen.concat([p] * copies), "wfa_adaptive", penalties, int(me.max()),
                             per_pair=np.tile(me, copies), aligner=aligner)
    finally:
        aim.aim_set_wfa_adaptive(aligner.ctx, 10, 50)
    assert_same(dev, want, what=f"adaptive {length} bp {penalties} {params}")
    assert np.array_equal(dev[0], np.tile(dev[0][:len(p)], copies))
    assert np.array_equal(dev[3], np.tile(dev[3][:len(p)], copies))


@pytest.mark.parametrize("megabytes", [40, 80, 200, 1000])
@pytest.mark.parametrize("length,count,copies", [(1000, 300, 80), (2600, 80, 40)])
def test_adaptive_places(length, count, copies, megabytes):
    """Workspaces that hold from one pair's history per group to many: groups that end take their next pair while others of
    the warp go on, around histories that still await their traceback.  Pairs end at scores far apart, some are rejected, and
    some end on their first row."""
    import paper_2208_01243_gb300 as aim
    pen = (0, 3, 4, 1)
    w = gen.Workload("adapt_places", 15, count, 40, length, 0.0, 0.08, 0.1, "wfa_adaptive", pen, None, 0.08)
    p = gen.generate(w)
    me = gen.per_pair_max_edits(w, p)
    lim = np.array([oracle.limit_for(pen, int(k)) for k in me], np.int64)
    s, f, off, cig, lens = oracle.wfa_adaptive_batch(p, pen, lim, min_len=10, max_dist=50)
    want = (s, f, [cig[off[i]:off[i] + lens[i]].astype(np.uint32) for i in range(len(p))])
    al = aim.Aligner(0, megabytes << 20)
    dev = device_results(gen.concat([p] * copies), "wfa_adaptive", pen, int(me.max()), per_pair=np.tile(me, copies),
                         max_length=length + 40, aligner=al)
    al.close()
    assert_same(dev, want, what=f"adaptive {length} bp, {megabytes} MB")
    assert np.array_equal(dev[0], np.tile(dev[0][:len(p)], copies))
    assert np.array_equal(dev[3], np.tile(dev[3][:len(p)], copies))


@pytest.mark.parametrize("lanes", [8, 32])
@pytest.mark.parametrize("params", [(10, 50), (4, 5), (2, 1), (10, 4000)])
@pytest.mark.parametrize("penalties", [(0, 3, 4, 1), (0, 4, 6, 2), (0, 1, 1, 1)])
def test_adaptive_lanes(aligner, penalties, params, lanes):
    """The shared-memory kernel by name, whatever the rule for when it is the faster one."""
    import paper_2208_01243_gb300 as aim
    w = gen.Workload("adapt_lanes", 25, 250, 30, 900, 0.0, 0.08, 0.08, "wfa_adaptive", penalties, None, 0.08)
    p = gen.generate(w)
    me = gen.per_pair_max_edits(w, p)
    lim = np.array([oracle.limit_for(penalties, int(k)) for k in me], np.int64)
    s, f, off, cig, lens = oracle.wfa_adaptive_batch(p, penalties, lim, min_len=params[0], max_dist=params[1])
    want = (s, f, [cig[off[i]:off[i] + lens[i]].astype(np.uint32) for i in range(len(p))])
    aim.aim_set_wfa_adaptive(aligner.ctx, *params)
    aim.aim_set_wfa_group(aligner.ctx, lanes)
    try:
        dev = device_results(gen.concat([p] * 80), "wfa_adaptive", penalties, int(me.max()), per_pair=np.tile(me, 80),
                             aligner=aligner)
    finally:
        aim.aim_set_wfa_adaptive(aligner.ctx, 10, 50)
        aim.aim_set_wfa_group(aligner.ctx, 0)
    assert_same(dev, want, what=f"adaptive {lanes} lanes {penalties} {params}")
    assert np.array_equal(dev[0], np.tile(dev[0][:len(p)], 80))
    assert np.array_equal(dev[3], np.tile(dev[3][:len(p)], 80))
