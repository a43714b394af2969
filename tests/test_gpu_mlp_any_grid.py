"""A training step of the prefilter gives the same bits on any number of SMs: gradients,
weights and loss of one step with the context told of fewer SMs than the device has, which
makes smaller grids, equal those of the full grid."""
import ctypes
import struct

import pytest
import torch

pytestmark = pytest.mark.gpu


def _sm_count(ctx):
    """The context's number of SMs (int32), found between the launch counter and the shared-memory
    limit, its neighbours in the context."""
    p = torch.cuda.get_device_properties(0)
    want = struct.pack("<qiiQ", ctx.launches, p.multi_processor_count, 0, p.shared_memory_per_block_optin)
    raw = ctypes.string_at(ctx.h.value, 4096)
    assert raw.count(want) == 1
    return ctypes.c_int32.from_address(ctx.h.value + raw.index(want) + 8)


@pytest.mark.parametrize("n", [100, 64 * 100, 20000, 64 * 304 + 1])
def test_step_does_not_depend_on_the_number_of_sms(n):
    import paper_2009_14467_gb300 as P
    from paper_2009_14467_gb300 import prefilter as F
    ctx = P.Context(0)
    g = torch.Generator().manual_seed(n)
    x = torch.randn((n, 16), generator=g).bfloat16().cuda()
    y = (torch.rand(n, generator=g) < 0.3).float().cuda()
    field = _sm_count(ctx)
    full, want = field.value, None
    for sms in (full, 148, 37, 1):
        net, loss = F.MLP(seed=5), torch.zeros(1, device="cuda")
        field.value = sms
        F.train_step(ctx, net, x, y, 0.01, 3.0, loss)
        field.value = full
        got = [t.clone() for t in list(net.grads()) + [net.w1, net.b1, net.w2, net.b2, net.w3, net.b3, loss]]
        want = want or got
        for a, b in zip(got, want):
            assert torch.equal(a, b), sms
    ctx.close()
