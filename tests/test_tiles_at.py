"""The stage-2 work list that a search at a threshold runs (host logic, no
GPU).  On the tensor cores (S1 of 32 and more) a wide tile of r rows is charged
(r rounded up to 32, plus 83) / 211 of a full one, and without any full wide
tile the keys' remainders become wide ones only if together they save
30 SM-microseconds per SM; every list covers each key once, and long ones are
cut into whole passes, partial wide tiles too."""
import numpy as np
import pytest

from paper_0804_3643_gb300 import binding as B
from test_tiles import (NARROW, NARROW16, NK, ROWS, T1, WIDE, check_cover, costs, offsets, random_counts,  # noqa: F401
                        round_up, tail_cover, tile_cost)

WIDE_LAUNCH = 30000.0


def tensor_cost(c, rows, n2):
    """A wide tile's cost on the tensor cores."""
    full = c["wide_slot"] * 128 * round_up(n2, 128)
    return full * ((round_up(rows, 32) + 83) / 211 if rows < T1 else 1.0) + c["wide_tile"]


def narrow_cover(c, rem, n2, known={}):
    at = (rem, round_up(n2, 512))  # (one set of costs in this file)
    if at not in known:
        known[at] = _narrow_cover(c, *at)
    return known[at]


def _narrow_cover(c, rem, n2):
    bulk = NARROW16 if tile_cost(c, NARROW16, n2) <= 2 * tile_cost(c, NARROW, n2) else NARROW
    return rem // ROWS[bulk] * tile_cost(c, bulk, n2) + tail_cover(c, rem % ROWS[bulk], n2)


def by_row_range(tiles):
    """{(key, first row): (rows, shape)}, pieces of a cut list together."""
    return {(int(k), int(f)): (int(r), int(s)) for k, f, r, s, _, _ in tiles}


@pytest.mark.parametrize("s1", [32, 38, 30000])
@pytest.mark.parametrize("n_sms", [0, 152])
def test_remainders_by_cost(costs, s1, n_sms):  # noqa: F811
    # a mix with full wide tiles: each remainder by its own cost
    n1, n2 = random_counts(np.random.default_rng(15))
    k1, k2 = offsets(n1), offsets(n2)
    tiles = B.plast_stage2_tiles(k1, k2, n_sms=n_sms, s1=s1)
    by_key = check_cover(tiles, k1, n1, n2)
    wide_rests = narrow_rests = plain_differs = 0
    for k, t in by_key.items():
        t = sorted(t)
        full, rem = divmod(int(n1[k]), T1)
        assert all(s == WIDE and r == T1 for _, r, s in t[:full])
        if not rem:
            continue
        narrow, wide = narrow_cover(costs, rem, n2[k]), tensor_cost(costs, rem, n2[k])
        if narrow < wide:
            assert all(s != WIDE for _, _, s in t[full:])
            narrow_rests += 1
        else:
            assert t[full:] == [(t[full][0], rem, WIDE)]
            wide_rests += 1
            plain_differs += narrow < tile_cost(costs, WIDE, n2[k])
    assert wide_rests > 100 and narrow_rests > 100 and plain_differs > 10
    wide = tiles[:, 3] == WIDE
    assert wide[:int(wide.sum())].all()


def test_rests_pay_the_launch(costs):  # noqa: F811
    # no key fills a wide tile: the remainders go wide together or not at all
    n1, n2, n_sms = np.zeros(NK, np.int64), np.zeros(NK, np.int64), 152
    gain = narrow_cover(costs, 100, 600) - tensor_cost(costs, 100, 600)
    assert gain > 0
    need = int(np.ceil(WIDE_LAUNCH * n_sms / gain))
    assert 10 < need < NK - 2
    for keys, wide in ((need - 1, False), (need, True)):
        n1[:], n2[:] = 0, 0
        n1[:keys], n2[:keys] = 100, 600
        n1[NK - 2], n2[NK - 2] = 3, 700  # narrow either way
        k1, k2 = offsets(n1), offsets(n2)
        tiles = B.plast_stage2_tiles(k1, k2, n_sms=n_sms, s1=38)
        check_cover(tiles, k1, n1, n2)
        got = by_row_range(tiles)
        assert all((s == WIDE) == wide for (k, _), (_, s) in got.items() if k < keys)
        assert all(s != WIDE for (k, _), (_, s) in got.items() if k == NK - 2)
        # without an SM count each goes by its own cost
        assert (B.plast_stage2_tiles(k1, k2, s1=38)[:keys, 3] == WIDE).all()
        # and one full wide tile anywhere pays the launch for all
        n1[NK - 1], n2[NK - 1] = 128, 100
        got = by_row_range(B.plast_stage2_tiles(offsets(n1), offsets(n2), n_sms=n_sms, s1=38))
        assert all(s == WIDE for (k, _), (_, s) in got.items() if k < keys)


def test_partial_wide_tiles_cut(costs):  # noqa: F811
    # few partial wide tiles against long lists: cut into whole passes, no
    # piece above twice the target, costliest first by their own charge
    rng = np.random.default_rng(18)
    n1, n2 = np.zeros(NK, np.int64), rng.integers(1000, 200000, size=NK).astype(np.int64)
    picked = rng.choice(NK, 200, replace=False)
    n1[picked] = rng.choice([5, 33, 64, 97, 127, 128], size=200)
    k1, k2 = offsets(n1), offsets(n2)
    B.plast_set_tile_shape(1)
    whole, cut = B.plast_stage2_tiles(k1, k2, s1=38), B.plast_stage2_tiles(k1, k2, n_sms=152, s1=38)
    assert len(whole) == 200 and len(cut) > 2 * 152 and (cut[:, 3] == WIDE).all()
    check_cover(cut, k1, n1, n2)
    cost = [tensor_cost(costs, r, hi - lo) for _, _, r, _, lo, hi in cut]
    assert all(a >= b for a, b in zip(cost, cost[1:]))
    target = sum(tensor_cost(costs, r, hi - lo) for _, _, r, _, lo, hi in whole) / (4 * 152)
    assert max(cost) <= 2 * target + tensor_cost(costs, 128, 128)


@pytest.mark.parametrize("s1", [-30000, 0, 31, 32, 38])
def test_cover_at_every_threshold(costs, s1):  # noqa: F811
    n1, n2 = random_counts(np.random.default_rng(16))
    k1, k2 = offsets(n1), offsets(n2)
    for schedule in (0, 1):
        B.plast_set_schedule(schedule)
        tiles = B.plast_stage2_tiles(k1, k2, n_sms=152, s1=s1)
        check_cover(tiles, k1, n1, n2)
        if schedule:
            assert (np.diff(tiles[:, 0]) >= 0).all()


def test_bad_offsets_at(costs):  # noqa: F811
    k = offsets(np.ones(NK, dtype=np.int64))
    bad = k.copy()
    bad[10] = bad[11] + 1
    with pytest.raises(B.PlastError):
        B.plast_stage2_tiles(bad, k, s1=38)


@pytest.mark.parametrize("s1,windows", [(31, 96), (-30000, 96), (32, 128)])
def test_wide_pieces_are_whole_passes(costs, s1, windows):  # noqa: F811
    # the plain wide kernel scores 96 windows a pass, the tensor kernel 128
    rng = np.random.default_rng(19)
    n1, n2 = np.zeros(NK, np.int64), rng.integers(1000, 200000, size=NK).astype(np.int64)
    n1[rng.choice(NK, 200, replace=False)] = 128
    B.plast_set_tile_shape(1)
    tiles = B.plast_stage2_tiles(offsets(n1), offsets(n2), n_sms=152, s1=s1)
    last = tiles[:, 5] == n2[tiles[:, 0]]
    assert (tiles[:, 3] == WIDE).all() and (~last).sum() > 200
    assert ((tiles[~last, 5] - tiles[~last, 4]) % windows == 0).all()
    # costliest first: by passes
    passes = -(-(tiles[:, 5] - tiles[:, 4]) // windows)
    assert (np.diff(passes) <= 0).all()
    # each row range's pieces partition its list
    for k in np.unique(tiles[:, 0]):
        v = sorted((int(a), int(b)) for a, b in tiles[tiles[:, 0] == k][:, 4:])
        assert v[0][0] == 0 and v[-1][1] == n2[k] and all(a[1] == b[0] for a, b in zip(v, v[1:]))


@pytest.mark.parametrize("s1", [31, 38])
def test_narrow_order(costs, s1):  # noqa: F811
    n1, n2 = random_counts(np.random.default_rng(20))
    n2 += np.arange(NK) % 700 * (n2 > 0)  # list lengths at every step of both passes
    tiles = B.plast_stage2_tiles(offsets(n1), offsets(n2), s1=s1)
    narrow = tiles[tiles[:, 3] != WIDE]
    cost = [tile_cost(costs, s, hi - lo) for _, _, _, s, lo, hi in narrow]
    assert len(narrow) > 1000 and all(a >= b for a, b in zip(cost, cost[1:]))


@pytest.mark.parametrize("slot,tile", [(1.0, 1.0), (0.25, 1.0), (4.0, 1.0), (1.0, 12.0), (0.6, 3.0)])
def test_callers_wide_costs_below_32(costs, slot, tile):  # noqa: F811
    # the plain wide kernel's costs, 0.317 and 2,960 beside the tensor kernel's
    # 0.140 and 3,660, scale with the wide costs that a caller sets
    c = dict(costs, wide_slot=0.140 * slot, wide_tile=3660.0 * tile)
    B.plast_set_tile_costs(c)
    n1, n2 = random_counts(np.random.default_rng(21))
    k1, k2 = offsets(n1), offsets(n2)
    by_key = check_cover(B.plast_stage2_tiles(k1, k2, s1=31), k1, n1, n2)
    wide_rests = narrow_rests = 0
    for k, t in by_key.items():
        t = sorted(t)
        full, rem = divmod(int(n1[k]), T1)
        if not rem:
            continue
        wide = 0.317 * slot * 128 * round_up(n2[k], 96) + 2960.0 * tile
        goes_wide = narrow_cover(costs, rem, n2[k]) >= wide
        assert ([s for _, _, s in t[full:]] == [WIDE]) == goes_wide
        wide_rests += goes_wide
        narrow_rests += not goes_wide
    assert wide_rests > 50 and narrow_rests > 50


@pytest.mark.parametrize("s1", [31, 38])
def test_key_by_key(costs, s1):  # noqa: F811
    # one launch per key: a remainder beside full wide tiles is one more of
    # them; without any, by the plain wide kernel's costs
    c = dict(costs, wide_slot=0.140, wide_tile=3660.0)
    B.plast_set_tile_costs(c)
    B.plast_set_schedule(1)
    n1, n2 = random_counts(np.random.default_rng(22))
    k1, k2 = offsets(n1), offsets(n2)
    tiles = B.plast_stage2_tiles(k1, k2, n_sms=152, s1=s1)
    by_key = check_cover(tiles, k1, n1, n2)
    assert (tiles[:, 4] == 0).all() and (tiles[:, 5] == n2[tiles[:, 0]]).all()
    wide_rests = narrow_rests = 0
    for k, t in by_key.items():
        t = sorted(t)
        if n1[k] >= T1:
            assert [r for _, r, _ in t[:-1]] == [T1] * (len(t) - 1) and all(s == WIDE for _, _, s in t)
            continue
        wide = 0.317 * 128 * round_up(n2[k], 96) + 2960.0
        goes_wide = narrow_cover(costs, int(n1[k]), n2[k]) >= wide
        assert ([s for _, _, s in t] == [WIDE]) == goes_wide
        wide_rests += goes_wide
        narrow_rests += not goes_wide
    assert wide_rests > 50 and narrow_rests > 50
