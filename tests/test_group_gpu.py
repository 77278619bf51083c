"""Channel-group execution of uint8 beams: beams long enough and shifts fine
enough that dd_execute takes it, at the sizes where it can go wrong.  Every
cell equals the oracle's sum (integers, exact)."""
import numpy as np
import pytest
import torch

import filterbank as fb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dd(built_lib):
    return built_lib


def _case(oracle_lib, nchan, band, dms, nsamp_out, seed=0, fill=None):
    rng = np.random.default_rng(1000 * nchan + seed)
    table = oracle_lib.dmshift(nchan, *band)
    nin = nsamp_out + oracle_lib.maxshift(table, dms)
    pitch = (nin + 15) // 16 * 16
    data = fb.random_filterbank(rng, nchan, nin, "u8", pitch=pitch)
    if fill is not None:
        data[:] = fill
    want = oracle_lib.dedisperse(np.ascontiguousarray(data[:, :nin]), table, dms, nsamp_out,
                                 threads=True)
    return data, nin, want


def _run(dd, plan, data, nin, nsamp_out):
    x = torch.from_numpy(data).cuda()
    out = torch.full((plan.ndm, (nsamp_out + 7) // 4 * 4), -7.0, dtype=torch.float32,
                     device="cuda")
    plan.execute(x, out, nsamp_in=nin, nsamp_out=nsamp_out)
    plan.sync(torch.cuda.current_stream())
    got = out.cpu().numpy()
    assert np.all(got[:, nsamp_out:] == -7.0)  # nothing written past the row's end
    return got[:, :nsamp_out]


L = (1500.0, 64e-6)


@pytest.mark.parametrize("nchan,width,ndm,lo,step,nsamp_out", [
    (64, -8.0, 130, 0.0, 0.5, 61440),     # whole groups, whole tiles
    (65, -8.0, 130, 0.0, 0.5, 61441),     # one channel left, one sample left, odd groups
    (66, -8.0, 129, 3.0, 0.5, 61439),     # two channels left, one DM in the last tile
    (67, -8.0, 192, 0.0, 0.4, 60417),     # three channels left, whole DM tiles
    (260, -20.0, 130, 50.0, 0.5, 61000),  # one group past the 256-channel widening
    (261, 20.0, 130, 50.0, 0.5, 61003),   # ascending band
    (1025, -300.0, 130, 0.0, 0.2, 60500),  # several widenings
])
def test_group_edges(dd, oracle_lib, nchan, width, ndm, lo, step, nsamp_out):
    band = (L[0], width / nchan, L[1])
    dms = (lo + step * np.arange(ndm)).astype(np.float32)
    dms = np.random.default_rng(ndm).permutation(dms)
    data, nin, want = _case(oracle_lib, nchan, band, dms, nsamp_out)
    plan = dd.Plan(nchan, *band, dms)
    assert np.array_equal(_run(dd, plan, data, nin, nsamp_out), want)


def test_group_of_three_channels(dd, oracle_lib):
    """Wide DM tiles, whose arrays do not fit for four channels."""
    band = (150.0, -30.0 / 1024, 327.68e-6)
    dms = (40.0 + 0.1 * np.arange(130)).astype(np.float32)
    data, nin, want = _case(oracle_lib, 1024, band, dms, 61000)
    plan = dd.Plan(1024, *band, dms)
    assert np.array_equal(_run(dd, plan, data, nin, 61000), want)


def test_group_largest_sums(dd, oracle_lib):
    """Every sample 255: the 16-bit lanes are full at each widening."""
    band = (L[0], -60.0 / 515, L[1])
    dms = np.repeat(np.float32([0.0, 0.3]), 65)  # repeated DMs, one pattern for zeros
    plan = dd.Plan(515, *band, dms)
    nin = 61440 + plan.maxshift
    data = np.full((515, (nin + 15) // 16 * 16), 255, dtype=np.uint8)
    assert np.all(_run(dd, plan, data, nin, 61440) == 515 * 255)


def test_group_in_a_captured_graph(dd, oracle_lib):
    """Its table is built outside the capture of the caller's stream."""
    band = (L[0], -20.0 / 260, L[1])
    dms = (0.5 * np.arange(130)).astype(np.float32)
    data, nin, want = _case(oracle_lib, 260, band, dms, 61000)
    plan = dd.Plan(260, *band, dms)
    _run(dd, plan, data[:, :1024].copy(), 200 + plan.maxshift, 200)  # short: the direct kernel
    x = torch.from_numpy(data).cuda()
    out = torch.zeros((130, 61000), dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        plan.execute(x, out, nsamp_in=nin)
    graph.replay()
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy(), want)
