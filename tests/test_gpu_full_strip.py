"""Stage 3.2 where a row changes between the register strip (64 columns) and
the chunks of the row buffer: drop-offs, gap costs and sequence lengths that
put the live window, the sequence end or a long gap at the strip's edges,
against the oracle bit for bit."""
import numpy as np
import pytest

import oracle
from conftest import bank_from

pytestmark = pytest.mark.gpu


def pair_bank(rng, n, length, gap):
    """n pairs: a sequence and its copy with substitutions and one indel of `gap` residues."""
    one, two = [], []
    for k in range(n):
        s = rng.integers(0, 20, length).astype(np.int8)
        t = np.where(rng.random(length) < 0.25, rng.integers(0, 20, length), s).astype(np.int8)
        t[:4] = s[:4]
        cut = int(rng.integers(4, length - 4))
        if k % 2:
            t = np.concatenate([t[:cut], t[min(cut + gap, length):]])
        else:
            t = np.concatenate([t[:cut], rng.integers(0, 20, gap).astype(np.int8), t[cut:]])
        one.append(s)
        two.append(t)
    return bank_from(one), bank_from(two)


@pytest.mark.parametrize("length,gap", [(30, 3), (62, 1), (63, 8), (64, 2), (65, 20), (130, 30), (400, 60)])
@pytest.mark.parametrize("xdrop,go,ge", [(0, 11, 1), (20, 11, 1), (38, 11, 1), (44, 11, 1), (60, 11, 1), (38, 9, 2),
                                         (38, 0, 1), (38, 11, 0), (500, 11, 1)])
def test_strip_edges(length, gap, xdrop, go, ge):
    torch = pytest.importorskip("torch")
    from paper_0804_3643_gb300 import binding as B, build

    assert torch.cuda.is_available(), "CUDA device required for -m gpu tests"
    build.build()
    rng = np.random.default_rng(100 * length + xdrop + go + 7 * ge)
    (c1, f1), (c2, f2) = pair_bank(rng, 12, length, gap)
    o1, o2 = oracle.make_bank(c1, f1), oracle.make_bank(c2, f2)
    prm = dict(gap_open=go, gap_extend=ge, s1=30, s2=30)
    d1, d2 = B.DeviceBank.from_host(c1, f1), B.DeviceBank.from_host(c2, f2)
    g1, g2 = B.plast_index_bank(d1.codes, d1.seq_off), B.plast_index_bank(d2.codes, d2.seq_off)
    records = B.plast_search(g1, g2, B.plast_default_params(**prm))
    want_g = oracle.small_gapped(o1, o2, oracle.ungapped(o1, o2, oracle.Params(**prm)), oracle.Params(**prm))
    assert len(want_g) > 0 and np.array_equal(B.gapped_numpy(records).view(np.uint8), want_g.view(np.uint8))
    want, want_ext = oracle.full_gapped(o1, o2, want_g, oracle.Params(**prm), x=xdrop, s3=30, return_extended=True)
    got, ext = B.plast_full_gapped(g1, g2, records, B.plast_default_params(**prm), xdrop=xdrop, s3=30)
    got = B.alignments_numpy(got)
    assert ext == want_ext and got.shape == want.shape
    assert np.array_equal(got.view(np.uint8), want.view(np.uint8))
