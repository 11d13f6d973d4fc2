"""The upper bound that stage 2's tensor kernel drops pairs by, and the kernel
at the edges of its tiles.

CPU: the bound, restated over the oracle's matrix, never lies below the
oracle's ungapped score (the seed's sum is its largest prefix; windows with
stops, and windows that run off their sequences).  GPU: wide tiles only, banks
that give one key a chosen number of bank-1 rows and bank-2 windows (around
the 32-row and 128-window steps), thresholds on both sides of the lowest one
that takes the tensor kernel, against the oracle bit for bit."""
import numpy as np
import pytest

import oracle
from conftest import bank_from

E2M1 = np.array([0, 1, 2, 3, 4, 6, 8, 12])  # times 2
STOP, WILD = 20, 17
SEGMENTS = ([7, 6, 9], [6, 6, 10])  # right (after the seed), left


def up(v):
    """The smallest e2m1 value (times 2) at or above v."""
    g = np.concatenate([-E2M1[::-1], E2M1])
    return int(g[g >= max(v, -12)].min())


def tables():
    s = np.array([[oracle.score(a, b) for b in range(21)] for a in range(21)])
    bound = np.full((22, 22), -12)  # 21: the sentinel
    bound[:21, :20] = s[:, :20]
    bound[:21, WILD] = np.maximum(s[:, WILD], s[:, STOP])
    bound[21, :20] = -12
    bound[:, 20] = bound[:, 21] = bound[:, WILD]
    pos = np.vectorize(up)(np.maximum(bound, 0))
    return bound, pos, np.vectorize(up)(bound)


def window(seq, p):
    pad = np.concatenate([np.full(30, 21), seq, np.full(30, 21)]).astype(int)
    q = p + 30
    return np.concatenate([pad[q:q + 26], pad[q - 22:q][::-1]])


def bound_of(a, b, t):
    bound, pos, seed = t
    s, p = bound[a, b], pos[a, b]
    best = []
    # the seed's cells 1 and 2 rounded up in the first segment, exact after it
    exact = s[:4].sum()
    for side, (first, segs) in enumerate(((4, SEGMENTS[0]), (26, SEGMENTS[1]))):
        q = s[0] + seed[a[1], b[1]] + seed[a[2], b[2]] + s[3] if side == 0 else 0
        v = []
        for i, n in enumerate(segs):
            v.append(q + p[first:first + n].sum())
            q = (exact if side == 0 and i == 0 else q) + s[first:first + n].sum()
            first += n
        best.append(max(v))
    return sum(best)


def test_seed_sum_is_its_largest_prefix():
    m = np.array([[oracle.score(a, b) for b in range(20)] for a in range(20)])
    for a in range(20):
        for b in range(20):
            if oracle.seed_class(1, a) == oracle.seed_class(1, b):
                for c in range(20):
                    for d in range(20):
                        if oracle.seed_class(2, c) == oracle.seed_class(2, d):
                            low = m.diagonal().min()
                            run = np.cumsum([low, m[a, b], m[c, d], low])
                            assert run[3] >= run.max() and run[3] >= 0


def test_bound_never_below_the_score():
    rng = np.random.default_rng(17)
    t = tables()
    # every positive score and its rounding's correction are e2m1 values
    assert set(np.unique(t[0][:, :20] - t[1][:, :20])) <= set(-E2M1)
    tight = 0
    for k in range(3000):
        n = int(rng.integers(4, 70))
        p = int(rng.integers(0, n - 3))
        x = rng.integers(0, 21 if k % 3 == 0 else 20, n)
        y = np.where(rng.random(n) < rng.uniform(0.1, 0.9), x, rng.integers(0, 21 if k % 3 == 0 else 20, n))
        word = rng.integers(0, 20, 4)
        x[p:p + 4] = y[p:p + 4] = word
        lo, hi = int(rng.integers(0, p + 1)), int(rng.integers(p + 4, n + 1))
        x, y = x.astype(np.int8), y[lo:hi].astype(np.int8)
        score = oracle.ungapped_pair(x, p, y, p - lo)[0]
        b = bound_of(window(x, p), window(y, p - lo), t)
        assert b >= score
        tight += b == score
    assert tight > 30  # (it is a bound that is met, not a loose one)


# ---------------------------------------------------------------------------
# GPU
# ---------------------------------------------------------------------------
def one_key_bank(rng, n, stops):
    """n sequences that hold the word AQAA once, at any place, ends included."""
    seqs = []
    for _ in range(n):
        s = rng.integers(0, 21 if stops else 20, int(rng.integers(4, 60))).astype(np.int8)
        p = int(rng.integers(0, len(s) - 3))
        s[p:p + 4] = [0, 5, 0, 0]
        seqs.append(s)
    return bank_from(seqs)


@pytest.mark.gpu
@pytest.mark.parametrize("n1,n2", [(1, 1), (31, 127), (32, 128), (33, 129), (64, 257), (65, 1000), (96, 130), (97, 5),
                                   (127, 300), (128, 384), (129, 1), (300, 700)])
def test_tile_edges(n1, n2):
    torch = pytest.importorskip("torch")
    from paper_0804_3643_gb300 import binding as B, build

    assert torch.cuda.is_available(), "CUDA device required for -m gpu tests"
    build.build()
    rng = np.random.default_rng(1000 * n1 + n2)
    banks = []
    for n in (n1, n2):
        codes, off = one_key_bank(rng, n, stops=n % 2 == 1)
        d = B.DeviceBank.from_host(codes, off)
        banks.append((B.plast_index_bank(d.codes, d.seq_off), oracle.make_bank(codes, off)))
    (g1, o1), (g2, o2) = banks
    B.plast_set_tile_shape(1)
    try:
        for s1 in (31, 32, 38, 60):
            want = oracle.ungapped(o1, o2, oracle.Params(s1=s1), threads=4)
            got = B.hits_numpy(B.plast_ungapped(g1, g2, B.plast_default_params(s1=s1)))
            assert got.shape == want.shape and np.array_equal(got.view(np.uint8), want.view(np.uint8)), s1
    finally:
        B.plast_set_tile_shape(0)
