"""Room for stage 2's survivors: sized from the last like search, and never the
reason for a search to fail that fits without.  Every pair of one key passes
the lowest threshold; a default search of the same banks has to fit in what it
needs itself.  A search whose own last rate asks for a tenth more than there is
falls back to the first guess and the exact count."""
import numpy as np
import pytest

import oracle
from paper_0804_3643_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    torch = pytest.importorskip("torch")
    from paper_0804_3643_gb300 import binding, build

    assert torch.cuda.is_available(), "CUDA device required for -m gpu tests"
    build.build()
    return binding


def both(B, b):
    d = B.DeviceBank.from_host(b.codes, b.seq_off)
    return B.plast_index_bank(d.codes, d.seq_off), oracle.make_bank(b.codes, b.seq_off)


def most_pairs_key(o1, o2):
    return int(np.argmax(np.diff(np.asarray(o1.idx.key_off, dtype=np.int64)) *
                         np.diff(np.asarray(o2.idx.key_off, dtype=np.int64))))


def same(a, b):
    return a.shape == b.shape and np.array_equal(a.view(np.uint8), b.view(np.uint8))


def test_rate_of_one_key_is_not_the_banks(B):
    b1, b2 = synth.workload("plastp_plain", seed=4, scale=1.0)
    (g1, o1), (g2, o2) = both(B, b1), both(B, b2)
    pairs = B.plast_pair_count(g1, g2)
    key = most_pairs_key(o1, o2)
    # between the first guess (8-byte keys) and every pair
    limit = 8 * (pairs // 128 + (1 << 20)) + (8 << 20)
    assert limit < 8 * pairs
    want = oracle.ungapped(o1, o2, threads=16)
    every = B.plast_ungapped_ex(g1, g2, B.plast_default_params(s1=-30000), keys=[key])
    assert len(every) > 1000
    try:
        B.plast_set_alloc_limit(limit)
        got = B.hits_numpy(B.plast_ungapped(g1, g2))
        assert same(got, want)
        # nor another threshold's rate
        low = B.plast_ungapped_ex(g1, g2, B.plast_default_params(s1=-30000), keys=[key])
        assert len(low) == len(every)
        recs, n = B.plast_search_ex(g1, g2, B.plast_default_params(s1=40))
        assert n == int((want["score"] >= 40).sum())
    finally:
        B.plast_set_alloc_limit(0)


def test_rate_with_too_little_room(B):
    b1, b2 = synth.workload("plastp_plain", seed=5, scale=1.0)
    (g1, _), (g2, _) = both(B, b1), both(B, b2)
    prm = B.plast_default_params(s1=-30000)
    first = B.plast_ungapped(g1, g2, prm)
    n = len(first)
    assert n == B.plast_pair_count(g1, g2)
    limit = 8 * n + (1 << 20)  # the exact count's keys, no tenth more
    assert limit < 8 * (11 * n // 10 + (1 << 20))
    try:
        B.plast_set_alloc_limit(limit)
        again = B.plast_ungapped(g1, g2, prm)
    finally:
        B.plast_set_alloc_limit(0)
    assert len(again) == n and bool((again == first).all())
