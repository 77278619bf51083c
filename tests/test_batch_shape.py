"""The tile shape that FP16/FP32 batches and servers choose for their beams: by
the launches they would make (no GPU), and on the GPU against the oracle and
against tiles of 12 (FP16) and 24 (FP32) DMs set by hand."""
import ctypes

import numpy as np
import pytest

import filterbank as fb
from tests import hostrt

FEW_DMS = {"f16": (1, 12, 1, 16, 8), "f32": (2, 12, 1, 16, 8)}
BATCHES = [  # beams, channels, DMs, samples
    (4, 512, 8, 32768), (4, 512, 12, 32768), (8, 1024, 24, 16384), (1, 512, 24, 65536),
    (64, 256, 16, 8192), (2, 128, 1, 16384), (16, 512, 48, 32768), (16, 512, 200, 8192),
]


@pytest.fixture(scope="module")
def host():
    return hostrt.Host()


def _band(nchan):
    return nchan, 1500.0, -300.0 / nchan, 64e-6


@pytest.mark.parametrize("kind", ["f16", "f32"])
@pytest.mark.parametrize("beams,nchan,ndm,ns", BATCHES)
def test_few_dms_do_not_take_the_48_dm_tiles(host, kind, beams, nchan, ndm, ns):
    plans = [host.plan(*_band(nchan), np.arange(ndm)) for _ in range(beams)]
    batch = host.batch(plans, kind, [ns] * beams)
    host.reset()
    assert host.batch_execute(batch) == 0
    launch = host.records(hostrt.DIRECT)[0]
    assert ndm > 24 or launch.dm_per_thread * launch.dm_warps < 48
    tiles = (ctypes.c_int * 5)()
    assert host.lib.dd_batch_get_tiles(batch, tiles) == 0
    assert tuple(tiles) == launch.shape


def test_shape_set_by_the_caller_stays(host):
    plan = host.plan(*_band(64), np.arange(8))
    batch = host.batch([plan], "f16", [8192])
    shape = (ctypes.c_int * 5)(4, 8, 1, 12, 8)
    assert host.lib.dd_batch_set_tiles(batch, shape) == 0
    host.reset()
    assert host.batch_execute(batch) == 0
    assert host.records(hostrt.DIRECT)[0].shape == (4, 8, 1, 12, 8)


def test_a_longer_binding_chooses_anew(host):
    """64 channels x 64 DMs: 8192 samples want small tiles, 2^20 the preferred ones."""
    plan = host.plan(*_band(64), np.arange(96))
    batch = host.batch([plan], "f32", [8192])
    host.reset()
    assert host.batch_execute(batch) == 0
    pin, nin, pout, nout = host.sizes(plan, 1 << 20)
    assert host.lib.dd_batch_set_io(batch, 0, ctypes.c_void_p(host.IN), pin, nin,
                                    ctypes.c_void_p(host.OUT), pout, nout) == 0
    assert host.batch_execute(batch) == 0
    short, long = [r.dm_per_thread * r.dm_warps for r in host.records(hostrt.DIRECT)][::2]
    assert short < long == 48


def _beam(dd, torch, kind, nchan, ndm, ns, rng):
    plan = dd.Plan(*_band(nchan), np.arange(ndm, dtype=np.float32))
    nin = ns + plan.maxshift
    data = fb.random_filterbank(rng, nchan, nin, kind, pitch=(nin + 15) // 16 * 16)
    out = torch.zeros((ndm, (ns + 3) // 4 * 4), device="cuda")
    return plan, data, torch.from_numpy(data).cuda(), out, nin


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["f16", "f32"])
def test_uneven_batch_matches_the_oracle(built_lib, oracle_lib, kind):
    """Integer values: exact in every type and shape."""
    import torch
    rng = np.random.default_rng(3)
    sizes = [(70, 5, 1023), (33, 12, 4097), (129, 25, 700)]
    beams = [_beam(built_lib, torch, kind, n, d, ns, rng) for n, d, ns in sizes]
    batch = built_lib.Batch([b[0] for b in beams], kind)
    for i, ((plan, _, x, out, nin), (_, _, ns)) in enumerate(zip(beams, sizes)):
        batch.set_io(i, x, out, nsamp_in=nin, nsamp_out=ns)
    for _ in range(2):
        batch.execute()
    batch.sync(torch.cuda.current_stream())
    for (plan, data, _, out, nin), (_, ndm, ns) in zip(beams, sizes):
        want = oracle_lib.dedisperse(np.ascontiguousarray(data[:, :nin]), plan.dmshift(),
                                     np.arange(ndm, dtype=np.float32), ns)
        assert np.array_equal(out.cpu().numpy()[:, :ns], want)


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["f16", "f32"])
@pytest.mark.parametrize("beams,nchan,ndm,ns", BATCHES[:6])
def test_few_dms_are_not_slower_than_small_tiles(built_lib, kind, beams, nchan, ndm, ns):
    import torch
    rng = np.random.default_rng(5)
    plan, _, x, out, nin = _beam(built_lib, torch, kind, nchan, ndm, ns, rng)
    batch = built_lib.Batch([plan] * beams, kind)
    outs = [torch.zeros_like(out) for _ in range(beams)]
    for i in range(beams):
        batch.set_io(i, x, outs[i], nsamp_in=nin, nsamp_out=ns)

    def best():
        times = []
        for _ in range(9):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            batch.execute()
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        return min(times[2:])

    own = best()
    batch.set_tiles(*FEW_DMS[kind])
    by_hand = best()
    assert own <= 1.05 * by_hand + 0.002
