"""The bounded waits of stage 2's tensor kernel: with a limit that no wait
meets, a call, a plan and the calibration report PLAST_E_TIMEOUT, and the next
call with the usual limit gives the oracle's hits (the device is as before);
with limits in between, which end the work at some later wait or at none, a
call either says so or gives the oracle's hits."""
import numpy as np
import pytest

import oracle
from paper_0804_3643_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def setup():
    torch = pytest.importorskip("torch")
    from paper_0804_3643_gb300 import binding as B
    from paper_0804_3643_gb300 import build

    assert torch.cuda.is_available(), "CUDA device required for -m gpu tests"
    build.build()
    b1, b2 = synth.workload("plastp_plain", seed=6, scale=1.0)
    gs, os_ = [], []
    for b in (b1, b2):
        d = B.DeviceBank.from_host(b.codes, b.seq_off)
        gs.append(B.plast_index_bank(d.codes, d.seq_off))
        os_.append(oracle.make_bank(b.codes, b.seq_off))
    want = oracle.ungapped(*os_, threads=16)
    B.plast_set_tile_shape(1)  # every tile on the tensor kernel
    yield B, gs[0], gs[1], want, oracle.small_gapped(*os_, want, threads=16)
    B.plast_set_wait_limit(0)
    B.plast_set_tile_shape(0)


def hits_of(B, g1, g2):
    return B.hits_numpy(B.plast_ungapped(g1, g2))


def same(a, b):
    return a.shape == b.shape and np.array_equal(a.view(np.uint8), b.view(np.uint8))


def timed_out(B, call):
    with pytest.raises(B.PlastError) as e:
        call()
    assert e.value.code == B.PLAST_E_TIMEOUT


def test_no_wait_met(setup):
    B, g1, g2, want, _ = setup
    B.plast_set_wait_limit(1)
    try:
        timed_out(B, lambda: B.plast_ungapped(g1, g2))
        timed_out(B, lambda: B.plast_search(g1, g2))
    finally:
        B.plast_set_wait_limit(0)
    assert same(hits_of(B, g1, g2), want)
    with pytest.raises(B.PlastError):
        B.plast_set_wait_limit(-1)


def test_plan(setup):
    import torch

    B, g1, g2, want, want_r = setup
    st = torch.cuda.Stream()
    plan = B.Plan(g1, g2, max_hits=2 * len(want), max_records=2 * len(want_r) + 64, stream=st)
    B.plast_set_wait_limit(1)
    try:
        plan.run(st)
        timed_out(B, lambda: plan.result(st))
    finally:
        B.plast_set_wait_limit(0)
    for _ in range(2):
        plan.run(st)
        recs, hits = plan.result(st)
        assert hits == len(want) and same(B.gapped_numpy(recs), want_r)


def test_calibration(setup):
    B, g1, g2, want, _ = setup
    costs = B.plast_get_tile_costs()
    B.plast_set_wait_limit(1)
    try:
        timed_out(B, B.plast_autotune)
    finally:
        B.plast_set_wait_limit(0)
    assert B.plast_get_tile_costs() == costs
    assert same(hits_of(B, g1, g2), want)


@pytest.mark.parametrize("clocks", [300, 1000, 3000, 10000, 30000, 100000, 1000000])
def test_some_waits_met(setup, clocks):
    B, g1, g2, want, _ = setup
    B.plast_set_wait_limit(clocks)
    try:
        got = hits_of(B, g1, g2)
    except B.PlastError as e:
        assert e.code == B.PLAST_E_TIMEOUT
    else:
        assert same(got, want)
    finally:
        B.plast_set_wait_limit(0)
    assert same(hits_of(B, g1, g2), want)
