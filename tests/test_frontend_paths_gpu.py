"""Every load path of the front end (16-byte words of several samples or of
part of one, 4-byte words for rows off 16 bytes) at the ends of words and of
groups of 32 samples, with extreme voltages, against the oracle bit for bit."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nint", [1, 2, 4, 8, 16, 32, 64])
@pytest.mark.parametrize("n", [1, 3, 31, 33, 511, 16387, 33000])
@pytest.mark.parametrize("offset", [0, 4, 12])
def test_load_paths(built_lib, oracle_lib, nint, n, offset):
    rng = np.random.default_rng(nint * 100000 + n)
    nraw = n * nint + int(rng.integers(0, nint))
    volts = rng.integers(-128, 128, size=(3, nraw, 4)).astype(np.int8)
    volts[1] = -128                          # the largest power, constant
    volts[2, :nraw // 2] //= 16              # most samples clipped away in the end
    pitch = (4 * nraw + 15) // 16 * 16
    buf = torch.zeros(3 * pitch + offset, dtype=torch.int8, device="cuda")
    rows = buf[offset:].view(3, pitch)
    rows[:, :4 * nraw] = torch.from_numpy(volts.reshape(3, -1)).cuda()
    for k, niter in ((3.0, 1), (1.0, 4)):
        out = torch.full((3, (n + 31) // 16 * 16), 0xA7, dtype=torch.uint8, device="cuda")
        got = built_lib.frontend(rows[:, :4 * nraw].unflatten(1, (nraw, 4)), nint, k, niter,
                                 out=out)
        want = oracle_lib.frontend(volts, nint, k, niter)
        assert np.array_equal(got[0].cpu().numpy()[:, :n], want[0])
        assert torch.all(out[:, n:] == 0xA7)
        assert np.array_equal(got[1].cpu().numpy(), want[1])
        assert np.array_equal(got[2].cpu().numpy(), want[2])
