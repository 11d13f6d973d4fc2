"""Six-frame translation where its 16-residue chunks meet contig ends, word
boundaries of a nucleotide array that starts anywhere, and the array's own
ends; and a bad code found wherever it stands."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def B():
    from paper_0804_3643_gb300 import binding, build

    assert torch.cuda.is_available(), "CUDA device required for -m gpu tests"
    build.build()
    return binding


@pytest.mark.parametrize("shift", [0, 1, 2, 3, 5, 15])
@pytest.mark.parametrize("lens", [[48], [51, 2, 0, 49], [144, 145, 146], [47, 50, 4096, 3, 1000], [30001]])
def test_chunks(B, shift, lens):
    rng = np.random.default_rng(shift + sum(lens))
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    dna = rng.integers(0, 4, off[-1]).astype(np.uint8)
    held = torch.full((shift + len(dna),), 3, dtype=torch.uint8, device="cuda")
    held[shift:] = torch.from_numpy(dna).cuda()
    aa, so, meta = B.plast_translate6(held[shift:], torch.from_numpy(off).cuda())
    w_aa, w_so, w_meta = oracle.translate6(dna, off)
    assert np.array_equal(aa.cpu().numpy(), w_aa) and np.array_equal(so.cpu().numpy(), w_so)
    assert np.array_equal(meta.cpu().numpy(), w_meta)


@pytest.mark.parametrize("shift", [0, 1, 15])
@pytest.mark.parametrize("n", [1, 14, 16, 17, 100])
def test_bad_code_anywhere(B, shift, n):
    off = torch.tensor([0, n], dtype=torch.int64, device="cuda")
    for at in {0, n // 2, n - 1}:
        held = torch.zeros(shift + n + 20, dtype=torch.uint8, device="cuda")
        held[:shift] = 255  # around the array, not in it
        held[shift + n:] = 255
        B.plast_translate6(held[shift:shift + n], off)
        held[shift + at] = 4 if at % 2 else 255
        with pytest.raises(B.PlastError):
            B.plast_translate6(held[shift:shift + n], off)
