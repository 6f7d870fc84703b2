"""GenASM windows whose distance lies at the edge of what a 32-bit band of the columns holds.

A window needing at most 14 edits is traced back from 32 bits a column, one
needing more from whole words.  Pairs here have 12 to 18 edits of one kind
within one window, at either end of it or spread out, so that the paths run
along the band's edges; limits on both sides of 14 take both kernels.
"""
import numpy as np
import pytest

import gen
import oracle
from devutil import assert_same, device_results

pytestmark = pytest.mark.gpu


def pairs():
    rnd = np.random.default_rng(7)
    acgt = np.frombuffer(b"ACGT", np.uint8)
    reads, targets = [], []
    for length in (64, 90, 200):
        for edits in range(12, 19):
            r = rnd.choice(acgt, length)
            extra = rnd.choice(acgt, edits)
            for at in (0, 20, 64 - edits):
                reads += [r, r, r]
                changed = r.copy()
                changed[at:at + edits] = rnd.choice(acgt, edits)
                targets += [np.concatenate([r[:at], extra, r[at:]]), np.concatenate([r[:at], r[at + edits:]]), changed]
            spread = np.sort(rnd.choice(60, edits, replace=False))
            reads += [r, r]
            targets += [np.delete(r, spread), np.insert(r, spread, extra)]
            # all insertions, then as many deletions: off the diagonal and back within one window
            reads.append(r)
            half = edits // 2
            targets.append(np.concatenate([r[:10], extra[:half], r[10:40], r[40 + half:]]))
    return gen.from_strings([x.tobytes() for x in reads], [x.tobytes() for x in targets])


@pytest.mark.parametrize("limit", [13, 14, 15, 18, 200, -1])
def test_windows_at_the_band_edge(oracle_lib, limit):
    import paper_2208_01243_gb300 as aim
    p = pairs()
    with_limit = np.full(len(p), (1 << 62) if limit < 0 else limit, np.int64)
    s, f, off, cig, lens = oracle.genasm_batch(p, with_limit, W=oracle.GENASM_W, O=oracle.GENASM_O)
    want = s, f, [cig[off[i]:off[i] + lens[i]].astype(np.uint32) for i in range(len(p))]
    a = aim.Aligner(0, 1 << 30)
    dev = device_results(p, "genasm", oracle.UNIT, limit, aligner=a)
    a.close()
    assert_same(dev, want, what=f"genasm limit {limit}")


def test_pairs_without_a_threshold_of_their_own(oracle_lib):
    """A negative entry takes the call's largest threshold: at 14 the call's windows are kept as 32-bit bands alone."""
    import paper_2208_01243_gb300 as aim
    p = pairs()
    per_pair = np.full(len(p), 14, np.int32)
    per_pair[1::2] = -1
    per_pair[::5] = 9
    s, f, off, cig, lens = oracle.genasm_batch(p, np.where(per_pair < 0, 14, per_pair).astype(np.int64),
                                               W=oracle.GENASM_W, O=oracle.GENASM_O)
    want = s, f, [cig[off[i]:off[i] + lens[i]].astype(np.uint32) for i in range(len(p))]
    a = aim.Aligner(0, 1 << 30)
    dev = device_results(p, "genasm", oracle.UNIT, 14, per_pair=per_pair, aligner=a)
    a.close()
    assert_same(dev, want, what="genasm, negative entries")
