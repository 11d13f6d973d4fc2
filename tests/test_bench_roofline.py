"""The bench's rating of stage 2: only pairs of wide tiles count as tensor work,
and the pace against the direct form is no share of a bound."""
import numpy as np

import bench


def test_only_tensor_pairs_count():
    # (key, first row, rows, shape, first and end window): two wide, one narrow
    t = np.array([[0, 0, 128, 0, 0, 2000], [1, 128, 40, 0, 128, 640], [2, 168, 16, 4, 0, 9000]], dtype=np.int32)
    pairs = 128 * 2000 + 40 * 512 + 16 * 9000
    wide = 128 * 2000 + 40 * 512
    r = bench.stage2_roofline(t, pairs, 0.001, True, None)
    assert r["tensor_pairs"] == wide and r["other_pairs"] == pairs - wide and r["bound"] == "tensor"
    assert np.isclose(r["achieved"], wide * 27 * 128 / 1e-6 / 1e15) and np.isclose(r["frac"], r["achieved"] / 13.5)
    # key by key, lists of fewer than 1,024 windows are not on the tensor cores
    assert bench.stage2_roofline(t, pairs, 0.001, False, None)["tensor_pairs"] == 128 * 2000
    d = bench.direct_form(pairs, 0.001, 152, 2070.0)
    assert "frac" not in d and np.isclose(d["cells_per_s"], pairs * 48 / 1e-6)
