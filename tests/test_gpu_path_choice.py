"""A gradient alone on a problem whose descriptor runs by transforms but whose gradient is faster on
the direct kernels, and the pyramid of a large field."""
import dataclasses

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wide", [0, 1])
@pytest.mark.parametrize("shape,window,levels,phases", [((256, 256), (8, 8), 1, 4), ((64, 64), (16, 16), 1, 6)])
def test_gradient_alone_of_many_phases(cuda_lib, shape, window, levels, phases, wide):
    """256^2, +-8, four phases: 142 us on the direct kernels, 205 by transforms."""
    dm = cuda_lib
    p = dm.Params(shape=shape, window=window, levels=levels, phases=phases)
    q = dataclasses.replace(p, path=dm.DMCR_PATH_DIRECT)
    assert dm.dmcr_workspace_size(p) != dm.dmcr_workspace_size(q)          # the descriptor: transforms
    g = torch.Generator("cuda").manual_seed(2)
    f = torch.rand((phases,) + shape, device="cuda", generator=g)
    if wide:
        f.view(-1)[4] = 3.0
    up = torch.randn(dm.dmcr_descriptor_length(p), device="cuda", generator=g)
    want = dm.descriptor_vjp(f, up, q)
    assert torch.equal(dm.descriptor_vjp(f, up, p), want)
    small = dm.Params(shape=(48, 40), window=(5, 6), levels=2)
    fs, us = [f, torch.rand(small.shape, device="cuda", generator=g)], [up, torch.randn(dm.dmcr_descriptor_length(small), device="cuda", generator=g)]
    out = [torch.empty_like(x) for x in fs]
    dm.dmcr_descriptor_vjp_batched([p, small], fs, us, out)
    assert torch.equal(out[0], want) and torch.equal(out[1], dm.descriptor_vjp(fs[1], us[1], small))
    # the loss' gradient, by transforms, is the same to rounding
    target = torch.full((dm.dmcr_descriptor_length(p),), 0.2, device="cuda")
    a, b = dm.loss_grad(f, target, p)[1], dm.loss_grad(f, target, q)[1]
    assert float(torch.linalg.norm(a - b)) <= 1e-5 * float(torch.linalg.norm(b))


def test_pyramid_of_a_large_field(cuda_lib):
    """One read of the field and a third of it written: within three times a copy of the field (one
    pass of 256 blocks for any size: 4.3 times)."""
    dm = cuda_lib
    p = dm.Params(shape=(8192, 8192), window=(1, 1), levels=3)
    f = torch.rand(p.shape, device="cuda")
    up = torch.randn(dm.dmcr_descriptor_length(p), device="cuda")
    out, ws = torch.empty_like(f), dm.workspace(p)

    def copy():
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        out.copy_(f)
        b.record()
        torch.cuda.synchronize()
        return a.elapsed_time(b)
    copies = np.median([copy() for _ in range(7)][2:])
    dm.dmcr_descriptor_vjp(p, f, up, out, ws)
    torch.cuda.synchronize()
    dm.dmcr_profile_enable(True)
    try:
        for _ in range(5):
            dm.dmcr_descriptor_vjp(p, f, up, out, ws)
        torch.cuda.synchronize()
        total = sum(ms for name, (ms, _) in dm.dmcr_profile_read().items() if name in ("pyramid", "restrict"))
    finally:
        dm.dmcr_profile_enable(False)
        dm.dmcr_profile_reset()
    assert total / 5 < 3 * copies, (total / 5, copies)
