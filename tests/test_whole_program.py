"""The files compiled as whole programs (build.WHOLE) do not see the library's
constant-memory tables: linked relocatably those are one set, in a whole program
they would be zero-filled copies that nothing uploads."""
import os
import subprocess

import pytest

from paper_0804_3643_gb300 import build


@pytest.mark.parametrize("name", sorted(build.WHOLE))
def test_no_shared_tables(name):
    src = os.path.join(build.CSRC, name)
    r = subprocess.run([build.nvcc(), *build._flags(False, src), "-E", src], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    assert "build_tables" in r.stdout  # (the shared header is in)
    for table in ("c_score", "c_cls2", "c_cls3", "seed_key"):
        assert table not in r.stdout, table
