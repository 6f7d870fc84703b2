"""The general wavefront kernels (wfa.cu), which serve costs that the shared-memory forms do not take: a gap opening of more
than four scaled units, none at all, or a gap extension that is not the unit.  Every lanes-per-pair value, the compact
histories, bands, batch plans with and without trials and bound passes, and the server, against the oracle."""
import numpy as np
import pytest

import gen
from devutil import assert_same, device_results, oracle_results
from test_gpu_ring import _mixed

pytestmark = pytest.mark.gpu

COSTS = [(0, 4, 6, 1), (0, 1, 0, 1), (0, 3, 5, 2)]


@pytest.fixture(scope="module")
def aligner():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2208_01243_gb300 as aim
    al = aim.Aligner(0, 2 << 30)
    yield al
    al.close()


def _limits(pen, me):
    return np.asarray(me, np.int64) * max(pen[1], pen[2] + pen[3])


@pytest.mark.parametrize("lanes", [0, 1, 2, 4, 8, 16, 32, 256])
@pytest.mark.parametrize("pen", COSTS)
@pytest.mark.parametrize("max_edits,band", [(1, -1), (9, -1), (12, 4)])
def test_every_group_size(aligner, lanes, pen, max_edits, band):
    import paper_2208_01243_gb300 as aim
    p = _mixed([1, 15, 16, 31, 32, 33, 64, 97, 150], 11 * lanes + max_edits)
    me = np.random.default_rng(lanes).integers(0, max_edits + 1, len(p)).astype(np.int32)
    me[::3] = max_edits
    aim.aim_set_wfa_group(aligner.ctx, lanes)
    try:
        dev = device_results(p, "wfa", pen, max_edits, per_pair=me, band=band, aligner=aligner)
    finally:
        aim.aim_set_wfa_group(aligner.ctx, 0)
    assert_same(dev, oracle_results(p, pen, _limits(pen, me), band=band), what=f"wfa {pen}, {lanes} lanes")


@pytest.mark.parametrize("max_length", [2048, 2049, 16_382, 16_383, 32_001])   # 8-byte, 16-bit and 32-bit histories
@pytest.mark.parametrize("lanes", [32, 256])
@pytest.mark.parametrize("pen", COSTS[:2])
@pytest.mark.parametrize("band", [-1, 12])
def test_compact_histories(aligner, max_length, lanes, pen, band):
    import paper_2208_01243_gb300 as aim
    w = gen.Workload("general_compact", 61, 300, 100, 700, 0.0, 0.08, 0.1, "wfa", pen, 40)
    p = gen.generate(w)
    me = np.random.default_rng(2).integers(10, 41, len(p)).astype(np.int32)
    aim.aim_set_wfa_group(aligner.ctx, lanes)
    try:
        dev = device_results(p, "wfa", pen, 40, per_pair=me, band=band, max_length=max_length, aligner=aligner)
    finally:
        aim.aim_set_wfa_group(aligner.ctx, 0)
    assert_same(dev, oracle_results(p, pen, _limits(pen, me), band=band), what=f"compact {max_length} {pen}")


@pytest.mark.parametrize("autotune", [False, True])
@pytest.mark.parametrize("bound", [0, 1, 2])
@pytest.mark.parametrize("pen", COSTS)
def test_batch_plans(aligner, pen, bound, autotune):
    import torch
    import paper_2208_01243_gb300 as aim
    w = gen.Workload("general_batch", 71, 1500, 60, 900, 0.0, 0.1, 0.1, "wfa", pen, None, max_edits_frac=0.1)
    p = gen.generate(w)
    me = gen.per_pair_max_edits(w, p)
    n = len(p)
    cap = p.read_len.astype(np.int64) + p.target_len.astype(np.int64) + 1
    coff = np.zeros(n + 1, np.int64); coff[1:] = np.cumsum(cap)
    reads, targets, ro, to, rl, tl, cd, pp = aim.upload(p.reads, p.targets, p.read_off, p.target_off, p.read_len,
                                                        p.target_len, coff, me.astype(np.int32))
    al = aim.Aligner(0, 256 << 20)
    aim.aim_set_batch_bound(al.ctx, bound)
    out = al.outputs(n, cigar_capacity=torch.from_numpy(cap))
    plan = aim.aim_batch_plan(al.ctx, reads, targets, ro, to, rl, tl, int(max(p.read_len.max(), p.target_len.max())),
                              aim.penalties(*pen[1:]), int(me.max()), pp, out["scores"], out["cigars"], cd,
                              out["cigar_lens"], out["flags"], scratch_bytes=1 << 30, autotune=autotune)
    lanes, n_bound = aim.aim_batch_bound_passes(plan)
    assert set(lanes) <= {0, 4, 8, 16, 32} and (n_bound > 0 if bound == 1 else n_bound == 0 if bound == 2 else True)
    aim.aim_batch_run(plan); aim.aim_batch_run(plan); torch.cuda.synchronize()
    s, f = out["scores"].cpu().numpy(), out["flags"].cpu().numpy()
    ln, cg = out["cigar_lens"].cpu().numpy(), out["cigars"].cpu().numpy().view(np.uint32)
    aim.aim_batch_destroy(plan)
    al.close()
    idx = np.random.default_rng(1).choice(n, 300, replace=False)
    sub = gen.concat([gen.from_strings([p.read(i)], [p.target(i)]) for i in idx])
    assert_same((s, f, [cg[coff[i]:coff[i] + ln[i]] for i in range(n)]), oracle_results(sub, pen, _limits(pen, me[idx])),
                idx=idx, what=f"batch {pen}, bound {bound}")
    plain = device_results(p, "wfa", pen, int(me.max()), per_pair=me, aligner=aligner)
    assert np.array_equal(s, plain[0]) and np.array_equal(f, plain[1]) and np.array_equal(ln, plain[3].view(np.int32))


@pytest.mark.parametrize("pen", COSTS[:2])
def test_server(aligner, pen):
    import paper_2208_01243_gb300 as aim
    from test_gpu_serve import _runs, _submit
    w = gen.Workload("general_serve", 81, 260, 60, 1600, 0.0, 0.1, 0.1, "wfa", pen, None, max_edits_frac=0.1)
    pool = gen.generate(w)
    me = gen.per_pair_max_edits(w, pool)
    ctx = aim.aim_create(0, 64 << 20)
    srv = aim.aim_server_create(ctx, aim.penalties(*pen[1:]), 256 << 20, 256 << 20)
    subs = [_submit(aim, srv, pool, idx, me[idx]) for idx in np.split(np.arange(len(pool)), [1, 4, 60, 200])]
    for t, _ in subs:
        aim.aim_server_wait(srv, t)
    aim.aim_server_destroy(srv)
    aim.aim_destroy(ctx)
    for _, o in subs:
        plain = device_results(o["pairs"], "wfa", pen, int(o["me"].max()), per_pair=o["me"], aligner=aligner)
        assert np.array_equal(o["scores"], plain[0]) and np.array_equal(o["flags"], plain[1])
        assert all(np.array_equal(a, b) for a, b in zip(_runs(o), plain[2]))


def test_cross_check_with_the_oracle_on_uneven_pairs(aligner):
    pen = (0, 4, 6, 1)
    w = gen.Workload("general_plain", 91, 400, 60, 1600, 0.0, 0.1, 0.1, "wfa", pen, None, max_edits_frac=0.1)
    p = gen.generate(w)
    me = gen.per_pair_max_edits(w, p)
    dev = device_results(p, "wfa", pen, int(me.max()), per_pair=me, aligner=aligner)
    assert_same(dev, oracle_results(p, pen, _limits(pen, me)), what="uneven pairs")
