"""aim_pack_2bit over lists of uneven sequences: every byte alignment, lengths around a chunk and a word, empty
sequences, gaps in the output, batches from one sequence to many, and bytes that are no base (written as code 0)."""
import numpy as np
import pytest

from oracle import pack

pytestmark = pytest.mark.gpu

LENGTHS = [0, 1, 3, 15, 16, 17, 31, 32, 33, 47, 48, 63, 64, 65, 100, 151, 992, 1023, 2500]


@pytest.mark.parametrize("count", [1, 2, 31, 32, 33, 700, 100_000])
@pytest.mark.parametrize("bad_share", [0.0, 0.2])
def test_pack_lists(count, bad_share):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2208_01243_gb300 as aim
    rng = np.random.default_rng(count)
    lens = rng.choice(LENGTHS if count < 10_000 else LENGTHS[:15], count).astype(np.int64)
    if count == 1:
        lens[0] = 2500
    off = np.cumsum(np.concatenate([[3], lens + rng.integers(0, 3, count)]))[:-1]
    nw = (lens + 31) // 32
    woff = np.cumsum(np.concatenate([[1], nw + rng.integers(0, 2, count)]))[:-1]
    text = np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, int(off[-1] + lens[-1]) + 1)].copy()
    want_bad = np.zeros(count, bool)
    for i in np.nonzero((rng.random(count) < bad_share) & (lens > 0))[0]:
        text[off[i] + rng.integers(0, lens[i])] = rng.choice(np.frombuffer(b"Nacgt-\x00\xffU", np.uint8))
        want_bad[i] = True
    al = aim.Aligner(0, 1 << 20)
    a, o, l, w = aim.upload(text, off.astype(np.uint64), lens.astype(np.uint32), woff.astype(np.uint64))
    words = torch.full((int(woff[-1] + nw[-1]) + 1,), -7, dtype=torch.int64, device=a.device)
    flags = torch.full((count,), 9, dtype=torch.uint8, device=a.device)
    aim.aim_pack_2bit(al.ctx, a, o, l, words, w, flags)
    torch.cuda.synchronize()
    al.close()
    words, flags = words.cpu().numpy(), flags.cpu().numpy()
    assert np.array_equal(flags, want_bad.astype(np.uint8))
    clean = np.where(np.isin(text, np.frombuffer(b"ACGT", np.uint8)), text, ord("A")).astype(np.uint8)
    written = np.zeros(len(words), bool)
    for i in range(count) if count < 10_000 else rng.choice(count, 3000, replace=False):
        got = words[woff[i]:woff[i] + nw[i]].view(np.uint64)
        assert np.array_equal(got, np.array(pack.pack_one(clean[off[i]:off[i] + lens[i]].tobytes()), np.uint64)), i
    for i in range(count):
        written[woff[i]:woff[i] + nw[i]] = True
    assert np.all(words[~written] == -7), "words outside the sequences' own were written"


@pytest.mark.parametrize("count", [1, 3, 151, 153, 1215, 1217])
@pytest.mark.parametrize("flags_wanted", [True, False])
def test_pack_shared_sequences(count, flags_wanted):
    """Few sequences, each taken by several warps: a byte that is no base is seen by whichever warp has its word, the flags
    of the others stay 0, and the words are the same with and without flags."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2208_01243_gb300 as aim
    rng = np.random.default_rng(count)
    lens = rng.integers(1, 20_000 if count < 10 else 3000, count).astype(np.int64)
    lens[0] = 17_000
    off = np.cumsum(np.concatenate([[1], lens]))[:-1]
    nw = (lens + 31) // 32
    woff = np.cumsum(np.concatenate([[0], nw]))[:-1]
    text = np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, int(off[-1] + lens[-1]))].copy()
    want_bad = (np.arange(count) % 3 == 0).astype(np.uint8)
    for i in np.nonzero(want_bad)[0]:
        text[off[i] + (lens[i] - 1 if i % 2 else rng.integers(0, lens[i]))] = ord("N")
    al = aim.Aligner(0, 1 << 20)
    a, o, l, w = aim.upload(text, off.astype(np.uint64), lens.astype(np.uint32), woff.astype(np.uint64))
    words = torch.full((int(nw.sum()),), -7, dtype=torch.int64, device=a.device)
    flags = torch.full((count,), 9, dtype=torch.uint8, device=a.device)
    aim.aim_pack_2bit(al.ctx, a, o, l, words, w, flags if flags_wanted else None)
    torch.cuda.synchronize()
    al.close()
    if flags_wanted:
        assert np.array_equal(flags.cpu().numpy(), want_bad)
    words = words.cpu().numpy().view(np.uint64)
    clean = np.where(text == ord("N"), ord("A"), text).astype(np.uint8)
    for i in range(0, count, max(count // 40, 1)):
        want = np.array(pack.pack_one(clean[off[i]:off[i] + lens[i]].tobytes()), np.uint64)
        assert np.array_equal(words[woff[i]:woff[i] + nw[i]], want), i
