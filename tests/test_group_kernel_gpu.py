"""The channel-group kernel itself: each case asserts that it ran there, and is
compared with the oracle cell by cell, at the sizes where it can go wrong (left
over channels, odd group counts, widenings, ragged rows and DM tiles, groups of
three channels, first use inside a capture)."""
import numpy as np
import pytest

import filterbank as fb
from tests import hostrt

TSAMP = 64e-6
# channels, highest frequency, channel width, DMs, lowest DM, DM step, samples, channels a group
CASES = [
    (256, 1500.0, -0.0625, 128, 0.0, 0.5, 77824, 4),    # whole groups, tiles and widening
    (257, 1500.0, -0.0625, 192, 0.0, 0.5, 50175, 4),    # one channel left, odd groups
    (262, 1500.0, -0.03125, 62, 10.0, 0.5, 155000, 4),  # two left, a DM tile not full
    (263, 1500.0, 0.0625, 128, 50.0, 0.5, 77000, 4),    # three left, ascending band
    (517, 1500.0, -0.039, 130, 0.0, 0.5, 38001, 4),     # widenings, two DMs in the last tile
    (511, 1500.0, -0.293, 128, 0.0, 1.5, 77001, 3),     # one left, odd groups of three
    (515, 1500.0, -0.293, 128, 0.0, 1.2, 76999, 3),     # two left
    (514, 1500.0, -0.293, 64, 0.0, 1.2, 155001, 3),     # one left, even groups
]


# A batch: channels, DMs, samples of its beams, and their bands.
SIZES = [(257, 192, 50175), (262, 128, 61441), (263, 128, 60417), (512, 130, 61440),
         (64, 40, 5001)]
BANDS = [(n, 1500.0, -16.0 / n if n > 64 else -4.0, TSAMP) for n, _, _ in SIZES]


def _dms(ndm, lo, step):
    return np.random.default_rng(ndm).permutation((lo + step * np.arange(ndm)).astype(np.float32))


@pytest.mark.parametrize("nchan,top,width,ndm,lo,step,ns,G", CASES)
def test_the_cases_take_the_group_kernel(nchan, top, width, ndm, lo, step, ns, G):
    """By the rules, on 152 SMs (no GPU)."""
    host = hostrt.Host()
    plan = host.plan(nchan, top, width, TSAMP, _dms(ndm, lo, step))
    host.reset()
    for _ in range(2):
        assert host.execute(plan, "u8", ns) == 0
    assert [r.beams for r in host.records(hostrt.TABLE)] == [G]
    assert host.records(hostrt.DIRECT, hostrt.GROUPED)[-1].kind == hostrt.GROUPED


def _execute(torch, plan, x, nin, ns):
    """Twice: the first may run in the direct kernel, its table built behind it."""
    out = torch.full((plan.ndm, (ns + 7) // 4 * 4), -7.0, device="cuda")
    plan.execute(x, out, nsamp_in=nin, nsamp_out=ns)
    torch.cuda.synchronize()
    first = out.clone()
    out.fill_(-7.0)
    plan.execute(x, out, nsamp_in=nin, nsamp_out=ns)
    plan.sync(torch.cuda.current_stream())
    assert torch.equal(first, out)
    return out.cpu().numpy()


@pytest.mark.gpu
@pytest.mark.parametrize("fill", [None, 255])
@pytest.mark.parametrize("nchan,top,width,ndm,lo,step,ns,G", CASES)
def test_group_kernel_matches_the_oracle(built_lib, oracle_lib, nchan, top, width, ndm, lo, step,
                                         ns, G, fill):
    import torch
    dms = _dms(ndm, lo, step)
    plan = built_lib.Plan(nchan, top, width, TSAMP, dms)
    nin = ns + plan.maxshift
    pitch = (nin + 15) // 16 * 16
    if fill is None:
        data = fb.random_filterbank(np.random.default_rng(nchan), nchan, nin, "u8", pitch=pitch)
        want = oracle_lib.dedisperse(np.ascontiguousarray(data[:, :nin]), plan.dmshift(), dms, ns,
                                     threads=True)
    else:  # the 16-bit lanes are full at each widening
        data = np.full((nchan, pitch), fill, dtype=np.uint8)
        want = np.full((ndm, ns), float(nchan * fill), dtype=np.float32)
    got = _execute(torch, plan, torch.from_numpy(data).cuda(), nin, ns)
    assert plan.groups(ns) == G
    assert np.all(got[:, ns:] == -7.0)
    assert np.array_equal(got[:, :ns], want)


@pytest.mark.gpu
def test_first_use_inside_a_capture(built_lib, oracle_lib):
    """The capture waits for the table; the graph holds the group kernel."""
    import torch
    nchan, top, width, ndm, lo, step, ns, G = CASES[1]
    dms = _dms(ndm, lo, step)
    plan = built_lib.Plan(nchan, top, width, TSAMP, dms)
    nin = ns + plan.maxshift
    data = fb.random_filterbank(np.random.default_rng(1), nchan, nin, "u8",
                                pitch=(nin + 15) // 16 * 16)
    x = torch.from_numpy(data).cuda()
    out = torch.zeros((ndm, (ns + 3) // 4 * 4), device="cuda")
    plan.execute(x, out, nsamp_in=200 + plan.maxshift, nsamp_out=200)  # the plan's own tables
    assert plan.groups(ns) == 0
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        plan.execute(x, out, nsamp_in=nin, nsamp_out=ns)
    assert plan.groups(ns) == G
    for _ in range(2):
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        want = oracle_lib.dedisperse(np.ascontiguousarray(data[:, :nin]), plan.dmshift(), dms, ns,
                                     threads=True)
        assert np.array_equal(out.cpu().numpy()[:, :ns], want)


@pytest.mark.gpu
def test_a_plan_destroyed_behind_its_first_execution(built_lib):
    """Its table may still be under way."""
    import torch
    nchan, top, width, ndm, lo, step, ns, _ = CASES[0]
    for _ in range(5):
        plan = built_lib.Plan(nchan, top, width, TSAMP, _dms(ndm, lo, step))
        nin = ns + plan.maxshift
        x = torch.ones((nchan, (nin + 15) // 16 * 16), dtype=torch.uint8, device="cuda")
        out = torch.zeros((ndm, ns), device="cuda")
        plan.execute(x, out, nsamp_in=nin, nsamp_out=ns)
        plan.close()
        torch.cuda.synchronize()
        assert bool((out == nchan).all())


@pytest.mark.gpu
def test_batch_beams_in_the_group_kernel(built_lib, oracle_lib):
    """Beams of every remainder of channels in one grouped launch, beside one in
    the direct kernel."""
    import torch
    rng = np.random.default_rng(8)
    beams = []
    for (nchan, ndm, ns), band in zip(SIZES, BANDS):
        dms = _dms(ndm, 0.0, 0.5)
        plan = built_lib.Plan(*band, dms)
        nin = ns + plan.maxshift
        data = fb.random_filterbank(rng, nchan, nin, "u8", pitch=(nin + 15) // 16 * 16)
        out = torch.full((ndm, (ns + 7) // 4 * 4), -7.0, device="cuda")
        beams.append((plan, dms, data, torch.from_numpy(data).cuda(), out, nin, ns))
    batch = built_lib.Batch([b[0] for b in beams], "u8")
    for i, (_, _, _, x, out, nin, ns) in enumerate(beams):
        batch.set_io(i, x, out, nsamp_in=nin, nsamp_out=ns)
    wants = [oracle_lib.dedisperse(np.ascontiguousarray(data[:, :nin]), plan.dmshift(), dms, ns,
                                   threads=True)
             for plan, dms, data, _, _, nin, ns in beams]
    for _ in range(4):  # directly, then grouped, then the graph
        for b in beams:
            b[4].fill_(-7.0)
        batch.execute()
        batch.sync(torch.cuda.current_stream())
        for (_, _, _, _, out, _, ns), want in zip(beams, wants):
            got = out.cpu().numpy()
            assert np.array_equal(got[:, :ns], want) and np.all(got[:, ns:] == -7.0)


def test_that_batch_takes_the_group_kernel():
    """By the rules, on 152 SMs (no GPU): four beams grouped, one direct."""
    host = hostrt.Host()
    plans = [host.plan(*band, _dms(ndm, 0.0, 0.5)) for band, (_, ndm, _) in zip(BANDS, SIZES)]
    batch = host.batch(plans, "u8", [ns for _, _, ns in SIZES])
    host.reset()
    for _ in range(2):
        assert host.batch_execute(batch) == 0
    assert [r.beams for r in host.records(hostrt.GROUPED)] == [4, 4]
    assert host.records(hostrt.DIRECT)[-1].beams == 1


@pytest.mark.gpu
def test_threads_share_a_plan_whose_table_is_under_way(built_lib):
    """Four threads, each with a stream and an output of its own, from the first
    execution on: some take the direct kernel, later ones the group kernel."""
    import threading

    import torch
    nchan, top, width, ndm, lo, step, ns, G = CASES[3]
    plan = built_lib.Plan(nchan, top, width, TSAMP, _dms(ndm, lo, step))
    nin = ns + plan.maxshift
    gen = torch.Generator(device="cuda").manual_seed(2)
    x = torch.randint(0, 256, (nchan, (nin + 15) // 16 * 16), dtype=torch.uint8, device="cuda",
                      generator=gen)
    outs = [torch.zeros((8, ndm, (ns + 3) // 4 * 4), device="cuda") for _ in range(4)]
    streams = [torch.cuda.Stream() for _ in outs]
    torch.cuda.synchronize()

    def work(out, stream):
        for k in range(len(out)):
            plan.execute(x, out[k], nsamp_in=nin, nsamp_out=ns, stream=stream)

    threads = [threading.Thread(target=work, args=a) for a in zip(outs, streams)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    plan.sync(torch.cuda.current_stream())
    assert plan.groups(ns) == G
    for out in outs:
        assert bool((out[:, :, :ns] == outs[0][0, :, :ns]).all())
