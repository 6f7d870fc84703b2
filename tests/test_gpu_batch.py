"""Batched form (bucketed queues, autotuned lanes per pair, CUDA-graph replay) against the plain form and the oracle."""
import numpy as np
import pytest

import gen
import oracle
from devutil import assert_same, device_results, oracle_results

pytestmark = pytest.mark.gpu

AFF = (0, 4, 6, 2)


def _mixed(n_uneven=2_500, n_short=2_003):
    pu = gen.generate(gen.WFA_UNEVEN, n_uneven)
    ps = gen.generate(gen.WFA_150BP, n_short)
    p = gen.concat([pu, ps])
    me = np.concatenate([gen.per_pair_max_edits(gen.WFA_UNEVEN, pu), np.full(n_short, 6, np.int32)])
    return p, me


def _batched(p, me, autotune, runs=2, scratch=0, compact=0, passes=None, bound=0, bounds=None, band=-1):
    import torch
    import paper_2208_01243_gb300 as aim
    n = len(p)
    cap = p.read_len.astype(np.int64) + p.target_len.astype(np.int64) + 1
    coff = np.zeros(n + 1, np.int64); coff[1:] = np.cumsum(cap)
    reads, targets, ro, to, rl, tl, cd, pp = aim.upload(p.reads, p.targets, p.read_off, p.target_off, p.read_len,
                                                        p.target_len, coff, me.astype(np.int32))
    al = aim.Aligner(0, 1 << 30)
    aim.aim_set_batch_compact(al.ctx, compact)
    aim.aim_set_batch_bound(al.ctx, bound)
    dev = rl.device
    scores = torch.full((n,), -7, dtype=torch.int32, device=dev)
    flags = torch.full((n,), 255, dtype=torch.uint8, device=dev)
    lens = torch.zeros(n, dtype=torch.int32, device=dev)
    cig = torch.zeros(int(coff[-1]), dtype=torch.int32, device=dev)
    ml = int(max(p.read_len.max(), p.target_len.max()))
    plan = aim.aim_batch_plan(al.ctx, reads, targets, ro, to, rl, tl, ml, aim.penalties(4, 6, 2, band=band),
                              int(me.max()), pp, scores, cig, cd, lens, flags, scratch_bytes=scratch,
                              autotune=autotune)
    groups, counts = aim.aim_batch_info(plan)
    if passes is not None:
        passes.append(aim.aim_batch_passes(plan))
    if bounds is not None:
        bounds.append(aim.aim_batch_bound_passes(plan))
    outs = []
    for _ in range(runs):
        scores.fill_(-7); flags.fill_(255)
        aim.aim_batch_run(plan)
        torch.cuda.synchronize()
        s = scores.cpu().numpy(); f = flags.cpu().numpy(); ln = lens.cpu().numpy().view(np.uint32)
        cg = cig.cpu().numpy().view(np.uint32)
        outs.append((s, f, [cg[coff[i]:coff[i] + ln[i]] for i in range(n)], ln))
    aim.aim_batch_destroy(plan)
    al.close()
    return outs, groups, counts


@pytest.mark.parametrize("autotune", [False, True])
def test_batched_equals_plain_and_oracle(oracle_lib, gen_lib, autotune):
    import __graft_entry__
    __graft_entry__.build()
    p, me = _mixed()
    outs, groups, counts = _batched(p, me, autotune)
    assert sum(counts) == len(p)
    assert all(g in (1, 2, 4, 8, 16, 32, 256) for g in groups)
    plain = device_results(p, "wfa", AFF, int(me.max()), per_pair=me)
    for o in outs:                       # every replay gives the plain form's results, bit for bit
        assert np.array_equal(o[0], plain[0]) and np.array_equal(o[1], plain[1])
        assert all(np.array_equal(x, y) for x, y in zip(o[2], plain[2]))
    idx = np.random.default_rng(4).choice(len(p), 400, replace=False)
    sub = gen.concat([gen.from_strings([p.read(i)], [p.target(i)]) for i in idx])
    lim = np.array([oracle.limit_for(AFF, int(me[i])) for i in idx], np.int64)
    assert_same(outs[-1], oracle_results(sub, AFF, lim), idx=idx, what="batched vs oracle")


@pytest.mark.parametrize("autotune", [False, True])
def test_compact_first_pass_gives_the_plain_results(oracle_lib, gen_lib, autotune):
    """Compact first passes forced on every bucket that allows one, with the fewest lanes that fit (so many pairs
    outgrow them): the second pass re-aligns exactly those, and every replay equals the plain form bit for bit."""
    import __graft_entry__
    __graft_entry__.build()
    p, me = _mixed(6_000, 2_003)
    passes = []
    outs, groups, counts = _batched(p, me, autotune, compact=1, passes=passes, scratch=4 << 30)
    first, full, n_compact = passes[0]
    assert n_compact > 0 and any(f and f < g for f, g in zip(first, full))
    plain = device_results(p, "wfa", AFF, int(me.max()), per_pair=me)
    for o in outs:
        assert (o[1] & 8).sum() == 0                 # no pair left flagged after the full pass
        assert np.array_equal(o[0], plain[0]) and np.array_equal(o[1], plain[1])
        assert all(np.array_equal(x, y) for x, y in zip(o[2], plain[2]))
    # never: one pass, the same results
    passes = []
    outs2, _, _ = _batched(p, me, autotune, runs=1, compact=2, passes=passes, scratch=4 << 30)
    assert passes[0][2] == 0
    assert np.array_equal(outs2[0][0], plain[0]) and np.array_equal(outs2[0][1], plain[1])


@pytest.mark.parametrize("autotune", [False, True])
@pytest.mark.parametrize("band", [-1, 25])
def test_bound_pass_gives_the_plain_results(oracle_lib, gen_lib, autotune, band):
    """Bound passes forced on every bucket: each exact pass runs with min(limit, bound) as its pairs' limit, and
    every replay equals the plain form (no bound pass) bit for bit, rejected pairs included (a tenth of the
    150 bp pairs are unrelated and exceed their limit); a sample also equals the oracle."""
    import __graft_entry__
    __graft_entry__.build()
    p, me = _mixed(3_000, 2_003)
    if band >= 0:
        keep = np.flatnonzero(np.abs(p.target_len.astype(np.int64) - p.read_len.astype(np.int64)) <= band)
        p = gen.concat([gen.from_strings([p.read(i)], [p.target(i)]) for i in keep])
        me = me[keep]
    bounds = []
    outs, groups, counts = _batched(p, me, autotune, bound=1, bounds=bounds, scratch=4 << 30, band=band)
    lanes, n_bound = bounds[0]
    assert n_bound >= 1 and all(g in (0, 4) for g in lanes)
    assert all(lanes[k] == 4 for k in range(32) if counts[k])
    plain = device_results(p, "wfa", AFF, int(me.max()), per_pair=me, band=band)
    assert (plain[1] & 1).sum() > 0                  # some pairs are rejected at their limit
    for o in outs:
        assert np.array_equal(o[0], plain[0]) and np.array_equal(o[1], plain[1])
        assert np.array_equal(o[3], plain[3])
        assert all(np.array_equal(x, y) for x, y in zip(o[2], plain[2]))
    idx = np.random.default_rng(9).choice(len(p), 300, replace=False)
    sub = gen.concat([gen.from_strings([p.read(i)], [p.target(i)]) for i in idx])
    lim = np.array([oracle.limit_for(AFF, int(me[i])) for i in idx], np.int64)
    assert_same(outs[-1], oracle_results(sub, AFF, lim, band=band), idx=idx, what="bound pass vs oracle")
    # never: no bound pass, the same results
    bounds = []
    outs2, _, _ = _batched(p, me, autotune, runs=1, bound=2, bounds=bounds, scratch=4 << 30, band=band)
    assert bounds[0][1] == 0
    assert np.array_equal(outs2[0][0], plain[0]) and np.array_equal(outs2[0][1], plain[1])


def test_tune_choices_export_and_import(gen_lib):
    """A plan made with autotune off in a context that imported another context's exported choices uses the same
    lanes, compact and bound passes per bucket, and gives the same results; a malformed text imports nothing."""
    import torch
    import paper_2208_01243_gb300 as aim
    p, me = _mixed(4_000, 1_003)
    n = len(p)
    cap = p.read_len.astype(np.int64) + p.target_len.astype(np.int64) + 1
    coff = np.zeros(n + 1, np.int64); coff[1:] = np.cumsum(cap)
    reads, targets, ro, to, rl, tl, cd, pp = aim.upload(p.reads, p.targets, p.read_off, p.target_off, p.read_len,
                                                        p.target_len, coff, me.astype(np.int32))
    ml = int(max(p.read_len.max(), p.target_len.max()))
    runs = []
    text = None
    for autotune in (True, False):
        al = aim.Aligner(0, 1 << 30)
        if text is not None:
            with pytest.raises(aim.AimError):
                aim.aim_tune_import(al.ctx, "4 6 2 -1 3 200 32 0\n")        # a field short
            assert aim.aim_tune_export(al.ctx) == ""
            aim.aim_tune_import(al.ctx, text)
            assert aim.aim_tune_export(al.ctx) == text
        out = al.outputs(n, cigar_capacity=torch.from_numpy(cap))
        out["cigars"].zero_()   # entries past a pair's runs are not written: compare whole buffers from zero
        plan = aim.aim_batch_plan(al.ctx, reads, targets, ro, to, rl, tl, ml, aim.penalties(4, 6, 2), int(me.max()),
                                  pp, out["scores"], out["cigars"], out["cigar_offsets"], out["cigar_lens"],
                                  out["flags"], autotune=autotune)
        aim.aim_batch_run(plan); torch.cuda.synchronize()
        runs.append((aim.aim_batch_info(plan)[0], aim.aim_batch_passes(plan)[:2], aim.aim_batch_bound_passes(plan)[0],
                     out["scores"].cpu().numpy().copy(), out["flags"].cpu().numpy().copy(),
                     out["cigars"].cpu().numpy().copy()))
        if autotune:
            text = aim.aim_tune_export(al.ctx)
            assert len(text.splitlines()) >= sum(1 for c in aim.aim_batch_info(plan)[1] if c)
        aim.aim_batch_destroy(plan)
        al.close()
    a, b = runs
    assert a[0] == b[0] and a[1] == b[1] and a[2] == b[2]
    assert all(np.array_equal(x, y) for x, y in zip(a[3:], b[3:]))


def test_batched_replay_sees_new_contents(gen_lib):
    """The plan binds buffers, not data: a replay after the inputs change aligns the new pairs."""
    import torch
    import paper_2208_01243_gb300 as aim
    p1 = gen.generate(gen.WFA_150BP, 3000)
    p2 = gen.generate(gen.WFA_150BP, 3000, first=3000)
    # same shapes: every read 150 bp, targets of varying length -> pad both batches into fixed slots
    slot = 160
    def slots(p):
        buf = np.full(2 * len(p) * slot, ord("A"), np.uint8)
        for i in range(len(p)):
            r, t = p.read(i), p.target(i)
            buf[2 * i * slot:2 * i * slot + len(r)] = np.frombuffer(r, np.uint8)
            buf[(2 * i + 1) * slot:(2 * i + 1) * slot + len(t)] = np.frombuffer(t, np.uint8)
        return buf
    n = len(p1)
    ro = np.arange(n, dtype=np.int64) * 2 * slot; to = ro + slot
    buf, ro_d, to_d = aim.upload(slots(p1), ro, to)
    rl, tl = aim.upload(p1.read_len, p1.target_len)
    al = aim.Aligner(0, 1 << 30)
    out = al.outputs(n)
    plan = aim.aim_batch_plan(al.ctx, buf, buf, ro_d, to_d, rl, tl, slot, aim.penalties(4, 6, 2), 6, None,
                              out["scores"], None, None, out["cigar_lens"], out["flags"], autotune=False)
    aim.aim_batch_run(plan); torch.cuda.synchronize()
    a = out["scores"].cpu().numpy().copy()
    buf.copy_(torch.from_numpy(slots(p2)).cuda()); tl.copy_(torch.from_numpy(p2.target_len.view(np.int32)).cuda())
    aim.aim_batch_run(plan); torch.cuda.synchronize()
    b = out["scores"].cpu().numpy().copy()
    aim.aim_batch_destroy(plan); al.close()
    assert np.array_equal(a, device_results(p1, "wfa", AFF, 6)[0])
    assert np.array_equal(b, device_results(p2, "wfa", AFF, 6)[0])


def _plan_of(al, p, me, autotune, ml=None, pen=(4, 6, 2)):
    """A plan over the pairs: (lanes, first-pass lanes, bound-pass lanes) per bucket and the pairs' scores and flags."""
    import torch
    import paper_2208_01243_gb300 as aim
    reads, targets, ro, to, rl, tl, pp = aim.upload(p.reads, p.targets, p.read_off, p.target_off, p.read_len,
                                                    p.target_len, me.astype(np.int32))
    out = al.outputs(len(p))
    ml = int(ml or max(p.read_len.max(), p.target_len.max()))
    plan = aim.aim_batch_plan(al.ctx, reads, targets, ro, to, rl, tl, ml, aim.penalties(*pen), int(me.max()), pp,
                              out["scores"], None, None, out["cigar_lens"], out["flags"], autotune=autotune)
    aim.aim_batch_run(plan); torch.cuda.synchronize()
    first, full, _ = aim.aim_batch_passes(plan)
    res = ((full, first, aim.aim_batch_bound_passes(plan)[0]),
           (out["scores"].cpu().numpy().copy(), out["flags"].cpu().numpy().copy()))
    aim.aim_batch_destroy(plan)
    return res


def test_choices_of_one_batch_do_not_reach_another(gen_lib):
    """A context that tuned a small batch, and one that imported its choices, plan a large batch of the same costs and
    thresholds as a fresh context does."""
    import paper_2208_01243_gb300 as aim
    p, me = _mixed(20_000, 0)
    small = gen.concat([gen.from_strings([p.read(i)], [p.target(i)]) for i in range(60)])
    few = me[:60].copy(); few[0] = me.max()
    al = aim.Aligner(0, 1 << 30)
    fresh, want = _plan_of(al, p, me, autotune=False)
    al.close()
    al = aim.Aligner(0, 1 << 30)
    tuned, _ = _plan_of(al, small, few, autotune=True)
    assert tuned[0] != fresh[0]                      # the small batch takes other lanes
    text = aim.aim_tune_export(al.ctx)
    assert text
    again, got = _plan_of(al, p, me, autotune=False)
    al.close()
    assert again == fresh and all(np.array_equal(a, b) for a, b in zip(got, want))
    al = aim.Aligner(0, 1 << 30)
    aim.aim_tune_import(al.ctx, text)
    assert _plan_of(al, p, me, autotune=False)[0] == fresh
    al.close()


def test_cached_choices_for_longer_reads(oracle_lib, gen_lib):
    """Choices tuned on short reads, or imported, for costs of the general kernels (a gap opening of 6 scaled units): a plan
    whose reads may pass 32,000 bp keeps to groups of 32 lanes and up without a bound pass, and bound lanes of 1 become 4
    where the form in registers does not take the costs."""
    import paper_2208_01243_gb300 as aim
    pen = (0, 4, 6, 1)
    w = gen.Workload("tuned", 12, 600, 100, 260, 0.0, 0.06, 0.1, "wfa", pen, 12)
    p = gen.generate(w)
    me = np.full(len(p), 12, np.int32)
    lim = np.full(len(p), 12 * 7, np.int64)
    want = oracle_results(p, pen, lim)
    al = aim.Aligner(0, 1 << 30)
    (full, first, bound), res = _plan_of(al, p, me, autotune=True, pen=pen[1:])
    text = aim.aim_tune_export(al.ctx)
    lines = [[int(v) for v in line.split()] for line in text.splitlines()]
    assert lines
    for change in (lambda v: v, lambda v: v[:6] + [4, 4, 1], lambda v: v[:6] + [8, 0, 1]):
        aim.aim_tune_import(al.ctx, "".join(" ".join(map(str, change(v))) + "\n" for v in lines))
        (full, first, bound), res = _plan_of(al, p, me, autotune=False, ml=33_000, pen=pen[1:])
        assert min(full) >= 32 and set(first) <= {0, 32, 256} and not any(bound)
        assert np.array_equal(res[0], want[0]) and np.array_equal(res[1], want[1])
    (full, first, bound), res = _plan_of(al, p, me, autotune=False, pen=pen[1:])
    assert 4 in bound and set(bound) <= {0, 4} and 8 in full
    assert np.array_equal(res[0], want[0]) and np.array_equal(res[1], want[1])
    al.close()


@pytest.mark.parametrize("scratch_mb,compact", [(48, 0), (48, 1), (48, 2), (32, 0)])
def test_plans_short_of_scratch(oracle_lib, gen_lib, scratch_mb, compact):
    """Scratch too small for classes of limits: buckets tuned by trials, each on the kernels that then run it.  The bound
    pass of these costs has one form, reported as 1 lane; results are the plain form's."""
    p = gen.generate(gen.Workload("scratch", 31, 500, 300, 2600, 0.01, 0.15, 0.1, "wfa", AFF, None, max_edits_frac=0.2))
    me = gen.per_pair_max_edits(gen.Workload("scratch", 31, 500, 300, 2600, 0.01, 0.15, 0.1, "wfa", AFF, None,
                                             max_edits_frac=0.2), p)
    bounds, passes = [], []
    outs, groups, counts = _batched(p, me, True, scratch=scratch_mb << 20, compact=compact, passes=passes, bounds=bounds)
    assert [k for k in range(32) if counts[k]] == [0, 4, 8]   # work and width classes
    assert set(bounds[0][0]) <= {0, 1}
    assert bounds[0][1] or (scratch_mb, compact) != (48, 0)   # (it saves far more than the few per cent it has to)
    plain = device_results(p, "wfa", AFF, int(me.max()), per_pair=me)
    for o in outs:
        assert np.array_equal(o[0], plain[0]) and np.array_equal(o[1], plain[1])
        assert all(np.array_equal(x, y) for x, y in zip(o[2], plain[2]))


@pytest.mark.parametrize("autotune", [False, True])
def test_replay_moves_pairs_between_classes(oracle_lib, gen_lib, autotune):
    """A plan of classes of limits, made on short reads with few errors, replayed over longer and noisier ones and over other
    thresholds, which put its pairs into classes that were empty or merged at planning, and back."""
    import torch
    import paper_2208_01243_gb300 as aim
    slot, n = 700, 2500
    rng = np.random.default_rng(8)

    def content(lo, hi, r0, r1, unrelated, seed):
        p = gen.generate(gen.Workload("classes", seed, n, lo, hi, r0, r1, unrelated, "wfa", AFF, 60))
        buf = np.full(2 * n * slot, ord("A"), np.uint8)
        for i in range(n):
            r, t = p.read(i), p.target(i)
            buf[2 * i * slot:2 * i * slot + len(r)] = np.frombuffer(r, np.uint8)
            buf[(2 * i + 1) * slot:(2 * i + 1) * slot + len(t)] = np.frombuffer(t, np.uint8)
        return p, buf
    easy, mixed, hard = (content(80, 200, 0.0, 0.01, 0.0, 3), content(80, 600, 0.0, 0.1, 0.1, 4),
                         content(500, 600, 0.08, 0.1, 0.2, 5))
    steps = [(easy, np.full(n, 60)), (hard, np.full(n, 60)), (mixed, rng.integers(0, 61, n)), (easy, rng.integers(0, 8, n)),
             (hard, np.where(rng.random(n) < 0.5, 60, 5)), (easy, np.full(n, 60))]
    ro = np.arange(n, dtype=np.int64) * 2 * slot
    buf, ro_d, to_d, rl, tl, pp = aim.upload(easy[1], ro, ro + slot, easy[0].read_len, easy[0].target_len,
                                             np.full(n, 60, np.int32))
    al = aim.Aligner(0, 1 << 30)
    cap = np.full(n, 260, np.int64)
    out = al.outputs(n, cigar_capacity=torch.from_numpy(cap))
    coff = np.concatenate([[0], np.cumsum(cap)])
    plan = aim.aim_batch_plan(al.ctx, buf, buf, ro_d, to_d, rl, tl, slot, aim.penalties(4, 6, 2), 60, pp, out["scores"],
                              out["cigars"], out["cigar_offsets"], out["cigar_lens"], out["flags"], autotune=autotune)
    for step, ((p, text), me) in enumerate(steps):
        me = me.astype(np.int32)
        buf.copy_(torch.from_numpy(text)); pp.copy_(torch.from_numpy(me))
        rl.copy_(torch.from_numpy(p.read_len.view(np.int32))); tl.copy_(torch.from_numpy(p.target_len.view(np.int32)))
        aim.aim_batch_run(plan); torch.cuda.synchronize()
        s, f = out["scores"].cpu().numpy(), out["flags"].cpu().numpy()
        ln, cg = out["cigar_lens"].cpu().numpy(), out["cigars"].cpu().numpy().view(np.uint32)
        plain = device_results(p, "wfa", AFF, 60, per_pair=me)
        assert np.array_equal(s, plain[0]) and np.array_equal(f, plain[1]), step
        assert all(np.array_equal(cg[coff[i]:coff[i] + ln[i]], plain[2][i]) for i in range(n)), step
        idx = rng.choice(n, 60, replace=False)
        sub = gen.concat([gen.from_strings([p.read(i)], [p.target(i)]) for i in idx])
        assert_same((s, f, [cg[coff[i]:coff[i] + ln[i]] for i in range(n)]),
                    oracle_results(sub, AFF, me[idx].astype(np.int64) * 8), idx=idx, what=f"replay {step}")
    aim.aim_batch_destroy(plan)
    al.close()
