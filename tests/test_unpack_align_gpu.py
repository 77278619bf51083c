"""The corner turn for spectra on 16, 8, 4 or fewer bytes and channel counts
that leave part of a tile, against numpy."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nbits,nchan", [(8, 8), (8, 16), (8, 124), (8, 136), (8, 1000), (8, 260),
                                         (4, 8), (4, 16), (4, 264), (4, 1016), (2, 16), (2, 272),
                                         (2, 1000), (1, 32), (1, 160), (1, 992), (1, 1000)])
@pytest.mark.parametrize("nsamp", [1, 255, 256, 1029])
@pytest.mark.parametrize("offset", [0, 8, 4, 1])
def test_alignments(built_lib, nbits, nchan, nsamp, offset):
    rng = np.random.default_rng(nchan * nsamp + nbits)
    want = rng.integers(0, 1 << nbits, size=(nsamp, nchan), dtype=np.uint8)
    per = 8 // nbits
    packed = np.zeros((nsamp, nchan // per), dtype=np.uint8)
    for i in range(per):
        packed |= want[:, i::per] << (i * nbits)
    buf = torch.full((packed.size + offset + 64,), 0xFF, dtype=torch.uint8, device="cuda")
    src = buf[offset:offset + packed.size]
    src.copy_(torch.from_numpy(packed.reshape(-1)))
    out = torch.full((nchan + 1, (nsamp + 31) // 16 * 16), 0xA7, dtype=torch.uint8, device="cuda")
    built_lib.unpack(src, nbits, nchan, nsamp, out=out[:nchan])
    torch.cuda.synchronize()
    host = out.cpu().numpy()
    assert np.array_equal(host[:nchan, :nsamp], want.T)
    assert np.all(host[:nchan, nsamp:] == 0xA7) and np.all(host[nchan] == 0xA7)
