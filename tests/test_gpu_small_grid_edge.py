"""Stage 3.1 where the best path leaves through the last column of the grid
(j = 64 in rows 57 to 64): alignments that run on past 64 residues on both
sides of every seed, on the diagonal and up to eight residues off it, with gap
costs down to none, against the oracle bit for bit."""
import numpy as np
import pytest

import oracle
from conftest import bank_from

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("go,ge", [(0, 0), (0, 1), (1, 0), (2, 1), (11, 1), (1000, 0), (3, 400)])
def test_paths_off_the_grid(go, ge):
    torch = pytest.importorskip("torch")
    from paper_0804_3643_gb300 import binding as B, build

    assert torch.cuda.is_available(), "CUDA device required for -m gpu tests"
    build.build()
    rng = np.random.default_rng(64)
    q, t = [], []
    for shift in range(9):
        a = rng.integers(0, 20, 240).astype(np.int8)
        ins = [rng.integers(0, 20, shift).astype(np.int8) for _ in range(2)]
        q.append(a)
        t.append(np.concatenate([a[:95], ins[0], a[95:140], ins[1], a[140:]]))  # path above the diagonal, then back on it
        q.append(np.concatenate([a[:95], ins[0], a[95:]]))                      # and below it
        t.append(a[:200 - shift])
    banks = []
    for seqs in (q, t):
        codes, off = bank_from(seqs)
        d = B.DeviceBank.from_host(codes, off)
        banks.append((B.plast_index_bank(d.codes, d.seq_off), oracle.make_bank(codes, off)))
    (g1, o1), (g2, o2) = banks
    prm = dict(s1=30, s2=30, gap_open=go, gap_extend=ge)
    want_h = oracle.ungapped(o1, o2, oracle.Params(**prm))
    want = oracle.small_gapped(o1, o2, want_h, oracle.Params(**prm))
    assert len(want) > 500
    recs, n = B.plast_search_ex(g1, g2, B.plast_default_params(**prm))
    got = B.gapped_numpy(recs)
    assert n == len(want_h) and got.shape == want.shape
    assert np.array_equal(got.view(np.uint8), want.view(np.uint8))
