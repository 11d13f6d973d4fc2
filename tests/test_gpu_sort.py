"""The record sort at the edges of its tiles (1,024 and 2,048 records) and of
its two ways (262,144 records): every pair of two one-word banks is a hit at
the lowest S1, in an order that stage 2's threads leave, so the hit count is
chosen exactly; and a plan whose list is sized for one way or the other and
holds fewer records, against the oracle bit for bit."""
import numpy as np
import pytest

import oracle
from conftest import bank_from

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    torch = pytest.importorskip("torch")
    from paper_0804_3643_gb300 import binding, build

    assert torch.cuda.is_available(), "CUDA device required for -m gpu tests"
    build.build()
    return binding


def both(B, seqs):
    codes, off = bank_from(seqs)
    d = B.DeviceBank.from_host(codes, off)
    return B.plast_index_bank(d.codes, d.seq_off), oracle.make_bank(codes, off)


def one_word_bank(rng, n):
    """n sequences with the word AQAA once each, other residues W, at any place."""
    seqs = []
    for _ in range(n):
        s = np.full(int(rng.integers(4, 40)), 17, np.int8)  # W
        p = int(rng.integers(0, len(s) - 3))
        s[p:p + 4] = [0, 5, 0, 0]
        s[p + 4:] = 18  # Y: no second word of this bank's
        seqs.append(s)
    return seqs


@pytest.mark.parametrize("n1,n2", [(1, 1), (1, 2), (31, 33), (1, 1024), (25, 41), (1, 2047), (2, 1024), (3, 1024), (7, 439),
                                   (32, 1000), (511, 513), (512, 512), (5, 52429), (513, 512), (640, 900)])
def test_hit_counts(B, n1, n2):
    rng = np.random.default_rng(1000 * n1 + n2)
    (g1, o1), (g2, o2) = (both(B, one_word_bank(rng, n)) for n in (n1, n2))
    key = oracle.seed_key([0, 5, 0, 0])
    want = oracle.ungapped(o1, o2, oracle.Params(s1=-30000), key_lo=key, key_hi=key + 1, threads=4)
    assert len(want) == n1 * n2
    got = B.hits_numpy(B.plast_ungapped_ex(g1, g2, B.plast_default_params(s1=-30000), keys=[key]))
    assert got.shape == want.shape and np.array_equal(got.view(np.uint8), want.view(np.uint8))


@pytest.mark.parametrize("room", [5000, 262144, 262145, 700000])
def test_plan_with_room_to_spare(B, room):
    rng = np.random.default_rng(room)
    base = [rng.integers(0, 20, 200).astype(np.int8) for _ in range(60)]
    (g1, o1), (g2, o2) = both(B, base[:40]), both(B, [np.roll(s, 3) for s in base] * 3)
    want = oracle.search(o1, o2)
    assert 1000 < len(want) < 5000 * 5
    room = max(room, len(want))
    plan = B.Plan(g1, g2, max_hits=4 * room, max_records=room)
    for _ in range(2):
        plan.run()
        records, _ = plan.result()
        got = B.gapped_numpy(records)
        assert got.shape == want.shape and np.array_equal(got.view(np.uint8), want.view(np.uint8))


@pytest.mark.parametrize("n", [1448, 1449])
def test_scan_of_few_and_many_tiles(B, n):
    # stage 3.1 of n * n given hits: 1,024 tiles of 2,048 flags and more
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(n)
    (g1, o1), (g2, o2) = (both(B, one_word_bank(rng, n)) for _ in range(2))
    key = oracle.seed_key([0, 5, 0, 0])
    hits = oracle.ungapped(o1, o2, oracle.Params(s1=-30000), key_lo=key, key_hi=key + 1, threads=8)
    assert len(hits) == n * n
    prm = dict(s2=25)
    want = oracle.small_gapped(o1, o2, hits, oracle.Params(**prm), threads=8)
    assert n < len(want) < len(hits)
    got = B.gapped_numpy(B.plast_small_gapped(g1, g2, B.hits_from_numpy(hits), B.plast_default_params(**prm)))
    assert got.shape == want.shape and np.array_equal(got.view(np.uint8), want.view(np.uint8))
