"""Integer detection at the edges of its tiles (31 regions of 32 samples a
warp, 7712 positions a CTA) against the oracle, bit for bit."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

WARP, TILE = 31 * 32, 7712


@pytest.mark.parametrize("nsamp", [1, 2, 31, 255, 256, 257, WARP - 1, WARP, WARP + 1, WARP + 225,
                                   7 * WARP + 1, TILE - 1, TILE, TILE + 1, TILE + 257,
                                   2 * TILE + WARP, 1 << 21])
@pytest.mark.parametrize("offset,nlevels", [(0, 9), (1, 9), (0, 6), (3, 5)])
def test_integer_tile_edges(built_lib, oracle_lib, nsamp, offset, nlevels):
    """The whole range of values, the last samples, plateaus across every
    boundary, rows that end short of the widest boxcar; rows on and off 16
    bytes."""
    rng = np.random.default_rng(nsamp + offset)
    plane = rng.integers(0, 1 << 20, size=(4, nsamp)).astype(np.float64)
    plane[1] = 0.0                                # all ties: the first time
    plane[2] = 2097151.0                          # the largest sums
    plane[3, -1:] = 2097151.0                     # highest at the row's end
    for edge in (WARP, TILE, TILE + WARP):
        plane[0, max(0, edge - 100):edge + 100] += 900000.0
    buf = torch.full((4 * nsamp + 64 + offset,), 1e9, dtype=torch.float32, device="cuda")
    pitch = nsamp + 3 if offset else (nsamp + 3) // 4 * 4
    x = torch.as_strided(buf, (4, nsamp), (pitch, 1), offset)
    x.copy_(torch.from_numpy(plane.astype(np.float32)))
    got = built_lib.detect(x, nsamp=nsamp, nlevels=nlevels, integer_valued=True)
    for g, w in zip(got, oracle_lib.detect(plane, nlevels, True)):
        assert np.array_equal(g.cpu().numpy(), w)


@pytest.mark.parametrize("value", [-1.0, -0.5, 0.25, 2097152.0, 1e30, float("inf"),
                                   float("-inf"), float("nan")])
@pytest.mark.parametrize("at", [0, WARP, TILE - 1, TILE, 15499])
def test_integer_rows_of_other_values(built_lib, value, at):
    x = torch.full((3, 15500), 1000.0, dtype=torch.float32, device="cuda")
    x[1, at] = value
    mean, std, snr, tpk = [r.cpu().numpy()
                           for r in built_lib.detect(x, nsamp=15500, nlevels=9,
                                                     integer_valued=True)]
    assert np.isnan(mean).tolist() == [False, True, False]
    assert np.isnan(std[1]) and np.all(np.isnan(snr[1])) and np.all(tpk[1] == -1)
    assert np.all(mean[[0, 2]] == 1000.0) and np.all(tpk[[0, 2]] == 0)


FTILE = 7680  # positions of a CTA, FP32 planes


@pytest.mark.parametrize("nsamp", [1, 2, 255, 256, WARP - 1, WARP + 1, WARP + 225, FTILE - 1, FTILE,
                                   FTILE + 1, FTILE + 257, 2 * FTILE + WARP])
@pytest.mark.parametrize("offset,nlevels", [(0, 9), (1, 9), (0, 6), (3, 5)])
def test_float_tile_edges(built_lib, oracle_lib, nsamp, offset, nlevels):
    """FP32 planes of small multiples of 1/4: every boxcar and row sum is exact,
    so the search equals the oracle's bit for bit; values of both signs, rows
    of negative values only (windows past the end must not count), zeros."""
    rng = np.random.default_rng(nsamp + offset)
    plane = rng.integers(-1000, 1000, size=(5, nsamp)) / 4.0
    plane[1] = 0.0
    plane[2] = -7.25
    plane[3] = -np.abs(plane[3]) - 1.0
    plane[4, -1:] = 900.5
    buf = torch.full((5 * nsamp + 64 + offset,), 1e9, dtype=torch.float32, device="cuda")
    pitch = nsamp + 3 if offset else (nsamp + 3) // 4 * 4
    x = torch.as_strided(buf, (5, nsamp), (pitch, 1), offset)
    x.copy_(torch.from_numpy(plane.astype(np.float32)))
    got = built_lib.detect(x, nsamp=nsamp, nlevels=nlevels, integer_valued=False)
    for g, w in zip(got, oracle_lib.detect(plane, nlevels, False)):
        assert np.array_equal(g.cpu().numpy(), w)


@pytest.mark.parametrize("value", [1e35, float("inf"), 1e-20])
@pytest.mark.parametrize("at", [0, WARP, FTILE - 1, FTILE, 15499])
def test_float_tiles_of_extreme_values(built_lib, value, at):
    """A huge or infinite value tops every window that holds it (all equal: the
    first counts); a row whose only value is tiny keeps it in its sums."""
    nsamp = 15500
    x = torch.zeros((2, nsamp), dtype=torch.float32, device="cuda")
    x[1, at] = value
    mean, std, snr, tpk = [r.cpu().numpy()
                           for r in built_lib.detect(x, nsamp=nsamp, nlevels=9,
                                                     integer_valued=False)]
    first = [min(max(0, at - (1 << i) + 1), nsamp - (1 << i)) for i in range(9)]
    assert tpk[1].tolist() == first and np.all(tpk[0] == 0)
    assert mean[0] == 0.0 and std[0] == 0.0
    v = float(np.float32(value))
    assert mean[1] == v / nsamp
    if np.isfinite(v):
        assert abs(std[1] - np.sqrt(v * v / nsamp - (v / nsamp) ** 2)) <= 1e-12 * std[1]
