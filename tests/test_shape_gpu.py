"""Executions that choose their own tile shape: sizes on both sides of the
lines where the choice changes (each listed shape of a data type is taken by
at least one of them on 152 SMs), against the oracle."""
import numpy as np
import pytest
import torch

import filterbank as fb

pytestmark = pytest.mark.gpu

# Blocks of at most 64 channels in FP32, block sums in FP32 or wider: the error
# of a cell is below (64 + nchan / 60 + 2) * 2^-24 of the sum of magnitudes.
CASES = [(kind, nchan, ndm, ns) for kind, sizes in {
    "u8": [(16, 1, 34), (16, 9, 39153), (16, 17, 40575), (16, 27, 40299), (150, 28, 39813),
           (16, 1, 82655), (16, 18, 78521), (16, 28, 80311), (16, 33, 86271), (16, 41, 81080),
           (16, 49, 80815), (64, 64, 8192)],
    "f16": [(16, 1, 34), (16, 1, 47785), (16, 9, 39094), (16, 17, 41720), (64, 17, 26146),
            (16, 18, 26651), (16, 33, 41344), (37, 34, 38969)],
    "f32": [(16, 1, 34), (16, 1, 20035), (16, 1, 42069), (16, 9, 20253), (16, 17, 20690),
            (150, 17, 20494), (16, 33, 20261), (16, 49, 26473), (16, 134, 25848)],
}.items() for nchan, ndm, ns in sizes]


@pytest.mark.parametrize("kind,nchan,ndm,ns", CASES)
def test_chosen_shape_matches_oracle(built_lib, oracle_lib, kind, nchan, ndm, ns):
    rng = np.random.default_rng(nchan * ndm + ns)
    band = (1400.0, -300.0 / nchan, 1e-4)
    dms = rng.uniform(0.0, 60.0, size=ndm).astype(np.float32)
    table = oracle_lib.dmshift(nchan, *band)
    nin = ns + oracle_lib.maxshift(table, dms)
    data = fb.random_filterbank(rng, nchan, nin, kind if kind == "u8" else kind + "-frac",
                                pitch=(nin + 15) // 16 * 16)
    plan = built_lib.Plan(nchan, *band, dms)
    before = plan.get_tiles(kind)
    x = torch.from_numpy(data).cuda()
    out = torch.full((ndm, (ns + 7) // 4 * 4), -7.0, dtype=torch.float32, device="cuda")
    plan.execute(x, out, nsamp_in=nin, nsamp_out=ns)
    plan.sync(torch.cuda.current_stream())
    assert plan.get_tiles(kind) == before  # the plan's own shape is not replaced
    got = out.cpu().numpy()
    assert np.all(got[:, ns:] == -7.0)
    want = oracle_lib.dedisperse(np.ascontiguousarray(data[:, :nin]), table, dms, ns,
                                 threads=True)
    if kind == "u8":
        assert np.array_equal(got[:, :ns], want)
    else:
        mag = oracle_lib.dedisperse(np.ascontiguousarray(np.abs(data[:, :nin])), table, dms, ns,
                                    threads=True)
        bound = (66 + nchan / 60) * 2.0 ** -24 * mag
        assert np.all(np.abs(got[:, :ns].astype(np.float64) - want) <= bound)


@pytest.mark.parametrize("kind,nchan,ndm,ns", [("u8", 96, 40, 57345), ("u8", 33, 301, 115000),
                                               ("f32", 64, 20, 90001)])
def test_host_blocks_equal_one_execution(built_lib, kind, nchan, ndm, ns):
    """Several host blocks of whole tile rounds give what one launch gives
    (integer values: exact in every type and shape)."""
    rng = np.random.default_rng(ns)
    plan = built_lib.Plan(nchan, 1400.0, -300.0 / nchan, 1e-4,
                          rng.uniform(0.0, 60.0, size=ndm).astype(np.float32))
    nin = ns + plan.maxshift
    data = fb.random_filterbank(rng, nchan, nin, kind, pitch=(nin + 15) // 16 * 16)
    x = torch.from_numpy(data).cuda()
    out = torch.empty((ndm, (ns + 3) // 4 * 4), dtype=torch.float32, device="cuda")
    plan.execute(x, out, nsamp_in=nin, nsamp_out=ns)
    host = np.full((ndm, ns + 5), -7.0, dtype=np.float32)
    plan.execute_host(data, host, nsamp_in=nin, nsamp_out=ns)
    assert np.array_equal(host[:, :ns], out.cpu().numpy()[:, :ns])
    assert np.all(host[:, ns:] == -7.0)


def test_autotuner_times_the_shapes_themselves(built_lib):
    """On a beam that the channel-group kernel takes, only the default shape
    stands for it: 8-DM tiles, a sixth of its rate, are timed as such."""
    dms = np.arange(260, dtype=np.float32) * 0.5
    plan = built_lib.Plan(512, 1500.0, -30.0 / 512, 64e-6, dms)
    ns = 61440
    nin = (ns + plan.maxshift + 15) // 16 * 16
    x = torch.zeros((512, nin), dtype=torch.uint8, device="cuda")
    out = torch.empty((260, ns), dtype=torch.float32, device="cuda")
    plan.execute(x, out, nsamp_in=nin, nsamp_out=ns)   # builds the table first
    ms = {tuple(t): m for t, m in plan.autotune(x, out, nsamp_in=nin, nsamp_out=ns)}
    assert ms[(1, 8, 1, 16, 4)] > 2.0 * ms[(4, 12, 1, 8, 8)] > 0.0
    assert plan.get_tiles("u8") == min((m, t) for t, m in ms.items() if m >= 0)[1]
