"""FP16 and FP32 sums have the same bits in every shape that the library
chooses or tunes among: whatever an execution's length, in a batch, in blocks
of a host buffer and after another shape has been set."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

DTYPE = {"f16": torch.float16, "f32": torch.float32}
LENGTHS = (100, 1000, 4096, 9000, 16384, 30000, 44444)
STAGES = (4, 8, 12, 16, 24)


def _beam(dd, kind, ndm, nchan=300):
    gen = torch.Generator(device="cuda").manual_seed(ndm)
    plan = dd.Plan(nchan, 1500.0, -300.0 / nchan, 64e-6, np.arange(ndm, dtype=np.float32))
    nin = 50000 + plan.maxshift
    x = torch.rand((nchan, (nin + 15) // 16 * 16), device="cuda", generator=gen).to(DTYPE[kind])
    out = torch.zeros((ndm, 50000), device="cuda")
    plan.execute(x, out, nsamp_in=nin)
    return plan, x, nin, out


@pytest.mark.parametrize("kind", ["f16", "f32"])
@pytest.mark.parametrize("ndm", [1, 20, 100, 200])
def test_bits_do_not_depend_on_length_or_route(built_lib, kind, ndm):
    plan, x, nin, want = _beam(built_lib, kind, ndm)
    for ns in LENGTHS:
        out = torch.zeros((ndm, (ns + 3) // 4 * 4), device="cuda")
        plan.execute(x, out, nsamp_in=nin, nsamp_out=ns)
        assert torch.equal(out[:, :ns], want[:, :ns]), ns
    batch = built_lib.Batch([plan], kind)
    out = torch.zeros_like(want)
    batch.set_io(0, x, out, nsamp_in=nin)
    batch.execute()
    batch.sync(torch.cuda.current_stream())
    assert torch.equal(out, want)
    host = np.zeros((ndm, 50000), dtype=np.float32)
    plan.execute_host(x.cpu().numpy(), host, nsamp_in=nin)
    assert np.array_equal(host, want.cpu().numpy())


@pytest.mark.parametrize("kind", ["f16", "f32"])
def test_bits_do_not_depend_on_the_tuned_shape(built_lib, kind):
    plan, x, nin, want = _beam(built_lib, kind, 20)
    for dm_per_thread, dm_warps, words in ((4, 8, 8), (1, 8, 4)):
        for stage in STAGES:
            try:
                plan.set_tiles(kind, dm_per_thread, dm_warps, 1, stage, words)
            except built_lib.DDError:  # its windows do not fit
                assert stage > 8
                continue
            out = torch.zeros_like(want)
            plan.execute(x, out, nsamp_in=nin)
            assert torch.equal(out, want), (dm_per_thread, stage)
