"""An indexing that runs out of memory after its first kernels are queued (on a
stream that the default stream does not wait for) gives its arrays back only
when these have ended: banks indexed right behind it, in the memory it gave
back, have the oracle's lists."""
import numpy as np
import pytest

import oracle
from paper_0804_3643_gb300 import synth

pytestmark = pytest.mark.gpu


def test_arrays_outlive_the_queued_kernels():
    torch = pytest.importorskip("torch")
    from paper_0804_3643_gb300 import binding as B
    from paper_0804_3643_gb300 import build

    assert torch.cuda.is_available(), "CUDA device required for -m gpu tests"
    build.build()
    big = synth.random_protein_bank(np.random.default_rng(1), 20000)
    small = synth.random_protein_bank(np.random.default_rng(2), 2000)
    db = B.DeviceBank.from_host(big.codes, big.seq_off)
    ds = B.DeviceBank.from_host(small.codes, small.seq_off)
    want = oracle.make_bank(small.codes, small.seq_off)
    # the padded bank fits, the 4 bytes a residue of the sorted positions do not
    limit = 3 * len(big.codes)
    assert len(big.codes) + 80 * (big.n_seqs + 1) < limit
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(10):
        try:
            B.plast_set_alloc_limit(limit)
            with pytest.raises(B.PlastError) as e:
                B.plast_index_bank(db.codes, db.seq_off, stream=side)
            assert e.value.code == B.PLAST_E_OOM
        finally:
            B.plast_set_alloc_limit(0)
        g = B.plast_index_bank(ds.codes, ds.seq_off)
        key_off, pos = B.plast_bank_export_index(g)
        assert np.array_equal(key_off.cpu().numpy(), want.idx.key_off)
        assert np.array_equal(pos.cpu().numpy(), want.idx.pos)
        g.free()
