"""The channeliser's thread groups, rounds and code paths at their edges."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _run(dd, volts, M, T, h, **kw):
    out = dd.channelise(volts, M, T, h, **kw)
    torch.cuda.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("M", [16, 32, 64, 128, 256])
@pytest.mark.parametrize("T", [1, 8, 12])
def test_spectra_do_not_depend_on_the_split(built_lib, M, T):
    """Spectra at the edges of segments, rounds and CTAs: a short row (one
    round per CTA) and the long row that it is cut from give equal bits."""
    rng = np.random.default_rng(M + T)
    per = 128 // min(M, 128) * (16 if T > 8 else 8)  # spectra of a CTA's round
    nspec = 33 * per * 5 + 3
    v = torch.from_numpy(rng.integers(-128, 128, size=(8, (nspec + T - 1) * M, 4), dtype=np.int8)).cuda()
    h = torch.from_numpy(rng.normal(size=M * T).astype(np.float32)).cuda()
    long = _run(built_lib, v, M, T, h, kind="cf32")
    for n0, n in ((0, 1), (per - 1, 2), (7, per), (31 * per - 3, 2 * per + 5), (nspec - 9, 9)):
        short = _run(built_lib, v[3:4, n0 * M:(n0 + n + T - 1) * M].contiguous(), M, T, h,
                     kind="cf32")
        assert np.array_equal(short[:, :n], long[3 * M:4 * M, n0:n0 + n])


@pytest.mark.parametrize("M,T", [(16, 8), (32, 4), (64, 12), (256, 2)])
@pytest.mark.parametrize("scale", [2.0 ** -9, 0.25, 777.0, 1e6, 3e30])
def test_codes_are_the_rounded_values(built_lib, M, T, scale):
    """Every code equals clamp(rint(v * scale)) of the FP32 value: products in
    and out of the range that the integer clamp takes, ties among them."""
    rng = np.random.default_rng(M)
    v = torch.from_numpy(rng.integers(-128, 128, size=(2, M * 300, 4), dtype=np.int8)).cuda()
    h = rng.integers(-4, 5, size=M * T).astype(np.float32) / 4  # ties at small scales
    h = torch.from_numpy(h).cuda()
    x = _run(built_lib, v, M, T, h, kind="cf32").astype(np.float64)
    q = _run(built_lib, v, M, T, h, kind="ci8", scale=scale)[:, :x.shape[1]]
    want = np.clip(np.rint(x * float(np.float32(scale))), -127, 127).astype(np.int8)
    assert np.array_equal(q, want)


def test_codes_of_values_that_are_not_numbers(built_lib):
    v = torch.ones((1, 16 * 64, 4), dtype=torch.int8, device="cuda")
    h = torch.ones(16 * 4, device="cuda")
    h[5] = float("nan")
    assert np.all(_run(built_lib, v, 16, 4, h)[:, :61] == -127)
