"""Stage 0 at the edges of its chunks (8192 padded positions), of its groups of
chunks and of the fill's 2048-word batches: the lists against the oracle's,
and the windows through stage 2's hits, bit for bit."""
import numpy as np
import pytest

import oracle
from conftest import bank_from

pytestmark = pytest.mark.gpu
CHUNK, GAP = 8192, 80


@pytest.fixture(scope="module")
def B():
    torch = pytest.importorskip("torch")
    from paper_0804_3643_gb300 import binding, build

    assert torch.cuda.is_available(), "CUDA device required for -m gpu tests"
    build.build()
    return binding


def cut(codes, n_seqs, rng):
    """codes as n_seqs sequences, empty ones included."""
    off = np.sort(rng.integers(0, len(codes) + 1, n_seqs - 1)) if n_seqs > 1 else np.empty(0, np.int64)
    return codes, np.concatenate([[0], off, [len(codes)]]).astype(np.int64)


def random_bank(rng, n_pad, n_seqs, kind):
    n = n_pad - GAP * (n_seqs + 1)
    codes = rng.integers(0, 21 if kind == "stops" else 20, n).astype(np.int8)
    if kind == "runs":  # one key, and keys of one bucket, thousands of times in a row
        codes[n // 8:n // 2] = 0
        codes[n // 2:n * 3 // 4] = np.tile([0, 1], n)[:n * 3 // 4 - n // 2]
    return cut(codes, n_seqs, rng)


def both(B, codes, off):
    d = B.DeviceBank.from_host(codes, off)
    return B.plast_index_bank(d.codes, d.seq_off), oracle.make_bank(codes, off)


@pytest.mark.parametrize("n_pad,n_seqs,kind", [
    (161, 1, "plain"), (164, 1, "plain"), (CHUNK - 1, 3, "plain"), (CHUNK, 1, "stops"), (CHUNK + 1, 5, "plain"),
    (CHUNK + 3, 1, "plain"), (4 * CHUNK, 7, "runs"), (36 * CHUNK - 2, 900, "stops"), (37 * CHUNK + 5, 1, "runs"),
    (55 * CHUNK + 16, 300, "plain"), (1216 * CHUNK + 7, 20000, "plain"), (4865 * CHUNK + 1, 60000, "runs")])
def test_lists_and_windows(B, n_pad, n_seqs, kind):
    rng = np.random.default_rng(n_pad + n_seqs)
    g, o = both(B, *random_bank(rng, n_pad, n_seqs, kind))
    key_off, pos = B.plast_bank_export_index(g)
    assert np.array_equal(key_off.cpu().numpy(), o.idx.key_off)
    assert np.array_equal(pos.cpu().numpy(), o.idx.pos)
    if n_pad > 60 * CHUNK:
        return
    q, qo = both(B, *bank_from([rng.integers(0, 20, 90).astype(np.int8) for _ in range(30)]))
    for s1 in (20, 38):
        for (x, xo), (y, yo) in (((q, qo), (g, o)), ((g, o), (q, qo))):
            want = oracle.ungapped(xo, yo, oracle.Params(s1=s1), threads=4)
            got = B.hits_numpy(B.plast_ungapped(x, y, B.plast_default_params(s1=s1)))
            assert got.shape == want.shape and np.array_equal(got.view(np.uint8), want.view(np.uint8)), s1


def test_empty_banks(B):
    for codes, off in ((np.empty(0, np.int8), [0]), (np.empty(0, np.int8), [0, 0, 0]), (np.zeros(3, np.int8), [0, 3])):
        g, o = both(B, codes, np.asarray(off, np.int64))
        key_off, pos = B.plast_bank_export_index(g)
        assert not key_off.cpu().numpy().any() and len(pos) == 0
