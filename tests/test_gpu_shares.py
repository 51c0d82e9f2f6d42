"""Blocks that share the feature pairs of the separable path's column kernels (few columns, one
or several shares, shares without a pair), and table uploads of every size."""
import dataclasses

import pytest
import torch

pytestmark = pytest.mark.gpu

# both paths sum the same terms in FP32, each a few 1e-7 of the largest entry (of the norm) from FP64
TOL = 2e-6


@pytest.mark.parametrize("lo,hi", [(0.0, 1.0), (-0.2, 1.2)])
@pytest.mark.parametrize("shape,window,levels", [((512, 512), (64, 64), 3), ((512, 512), (100, 80), 1),
                                                 ((256, 256), (64, 64), 1), ((300, 250), (90, 80), 1)])
def test_shared_pairs_equal_direct(cuda_lib, shape, window, levels, lo, hi):
    dm = cuda_lib
    gen = torch.Generator("cuda").manual_seed(3)
    f = torch.rand(shape, device="cuda", generator=gen) * (hi - lo) + lo
    p = dm.Params(shape=shape, window=window, levels=levels)
    q = dataclasses.replace(p, path=dm.DMCR_PATH_DIRECT)
    a, b = dm.descriptor(f, p), dm.descriptor(f, q)
    assert float((a - b).abs().max()) <= TOL * float(b.abs().max())
    up = torch.randn(dm.dmcr_descriptor_length(p), device="cuda", generator=gen)
    ga, gb = dm.descriptor_vjp(f, up, p), dm.descriptor_vjp(f, up, q)
    assert float(torch.linalg.norm(ga - gb)) <= TOL * float(torch.linalg.norm(gb))
    target = (0.8 * b).contiguous()
    (la, ha), (lb, hb) = dm.loss_grad(f, target, p), dm.loss_grad(f, target, q)
    assert float(((la - lb).abs() / lb.abs().clamp_min(1e-30)).max()) <= 1e-5
    assert float(torch.linalg.norm(ha - hb)) <= 1e-5 * float(torch.linalg.norm(hb))


@pytest.mark.parametrize("count", [1, 2, 3, 5, 9, 20, 60])
def test_uploads_of_every_size(cuda_lib, count):
    dm = cuda_lib
    ps = [dm.Params(shape=(16 + 8 * (i % 3), 24), window=(4, 5), levels=1 + i % 2) for i in range(count)]
    gen = torch.Generator("cuda").manual_seed(4)
    fs = [torch.rand(p.shape, device="cuda", generator=gen) for p in ps]
    ds = [torch.empty(dm.dmcr_descriptor_length(p), device="cuda") for p in ps]
    dm.dmcr_descriptor_batched(ps, fs, ds)
    for p, f, d in zip(ps, fs, ds):
        assert torch.equal(d, dm.descriptor(f, p))
