"""Stage 2 key by key (plast_set_schedule(1)) around the list length from which
a key's wide tiles take the tensor kernel, with full and partial wide tiles,
at thresholds on both sides of 32, against the oracle bit for bit."""
import numpy as np
import pytest

import oracle
from test_tensor_bound import one_key_bank

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n1,n2", [(1, 1024), (128, 1023), (128, 1024), (129, 1025), (200, 1100), (260, 95), (127, 3000)])
def test_list_lengths(n1, n2):
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
    B.plast_set_schedule(1)
    try:
        for shape in (0, 1):
            B.plast_set_tile_shape(shape)
            for s1 in (31, 32, 38):
                want = oracle.ungapped(o1, o2, oracle.Params(s1=s1), threads=4)
                got = B.hits_numpy(B.plast_ungapped(g1, g2, B.plast_default_params(s1=s1)))
                assert got.shape == want.shape and np.array_equal(got.view(np.uint8), want.view(np.uint8)), (shape, s1)
    finally:
        B.plast_set_schedule(0)
        B.plast_set_tile_shape(0)
