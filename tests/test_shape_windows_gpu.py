"""Executions on wide windows (coarse DM steps, low frequencies), where rings of
fewer stages and shapes with several time warps come in: every cell against the
oracle, and never slower than the tile of few DMs that fits with the most
stages, set by hand."""
import numpy as np
import pytest
import torch

import filterbank as fb

pytestmark = pytest.mark.gpu

LOW = (150.0, 30.0, 327.68e-6)
LBAND = (1500.0, 300.0, 64e-6)
# Tiles of 12 (FP16), 24 (FP32) and 48 (uint8) DMs, and of half as many each
# time, with ever smaller stages.
BY_HAND = {
    "f16": [(1, 12, 1, c, 8) for c in (16, 8, 4)] + [(1, 6, 3, c, 8) for c in (16, 8, 4)],
    "f32": [(2, 12, 1, c, 8) for c in (16, 8, 4)] + [(2, 6, 2, c, 8) for c in (16, 8, 4)],
    "u8": [(4, 12, 1, c, 8) for c in (8, 4)] + [(4, 6, 2, c, 8) for c in (8, 4)],
}


def _plan(dd, band, nchan, ndm, step):
    f, width, tsamp = band
    return dd.Plan(nchan, f, -width / nchan, tsamp, (step * np.arange(ndm)).astype(np.float32))


@pytest.mark.parametrize("kind", ["u8", "f16", "f32"])
@pytest.mark.parametrize("band,nchan,ndm,step,ns", [
    (LBAND, 75, 97, 3.0, 8191),
    (LBAND, 67, 50, 9.0, 4100),
    (LOW, 66, 25, 3.0, 2050),
    (LOW, 49, 13, 12.0, 1025),
])
def test_wide_windows_match_the_oracle(built_lib, oracle_lib, kind, band, nchan, ndm, step, ns):
    rng = np.random.default_rng(nchan)
    plan = _plan(built_lib, band, nchan, ndm, step)
    nin = ns + plan.maxshift
    data = fb.random_filterbank(rng, nchan, nin, kind if kind == "u8" else kind + "-frac",
                                pitch=(nin + 15) // 16 * 16)
    out = torch.full((ndm, (ns + 7) // 4 * 4), -7.0, device="cuda")
    plan.execute(torch.from_numpy(data).cuda(), out, nsamp_in=nin, nsamp_out=ns)
    plan.sync(torch.cuda.current_stream())
    got = out.cpu().numpy()
    assert np.all(got[:, ns:] == -7.0)
    dms = (step * np.arange(ndm)).astype(np.float32)
    want = oracle_lib.dedisperse(np.ascontiguousarray(data[:, :nin]), plan.dmshift(), dms, ns)
    if kind == "u8":
        assert np.array_equal(got[:, :ns], want)
    else:
        mag = oracle_lib.dedisperse(np.ascontiguousarray(np.abs(data[:, :nin])), plan.dmshift(),
                                    dms, ns)
        # Blocks of at most 48 channels in FP32, their sums in FP32 or wider.
        assert np.all(np.abs(got[:, :ns].astype(np.float64) - want)
                      <= (50 + nchan / 48) * 2.0 ** -24 * mag)


def _time(plan, x, out, nin, ns):
    best = 1e9
    for _ in range(8):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        plan.execute(x, out, nsamp_in=nin, nsamp_out=ns)
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("kind", ["u8", "f16", "f32"])
@pytest.mark.parametrize("band,nchan,ndm,step,ns", [
    (LOW, 1024, 200, 0.3, 16384),
    (LBAND, 512, 480, 5.0, 16384),
    (LBAND, 512, 200, 8.0, 16384),
])
def test_wide_windows_are_not_slower_than_small_tiles(built_lib, kind, band, nchan, ndm, step, ns):
    plan = _plan(built_lib, band, nchan, ndm, step)
    nin = ns + plan.maxshift
    x = torch.zeros((nchan, (nin + 15) // 16 * 16), device="cuda",
                    dtype={"u8": torch.uint8, "f16": torch.float16, "f32": torch.float32}[kind])
    out = torch.empty((ndm, ns), device="cuda")
    own = _time(plan, x, out, nin, ns)
    for tiles in BY_HAND[kind]:
        try:
            plan.set_tiles(kind, *tiles)
        except built_lib.DDError:
            continue
        by_hand = _time(plan, x, out, nin, ns)
        print(kind, tiles, own, by_hand)
        assert own <= 1.05 * by_hand, (tiles, own, by_hand)
        break
