"""The separable path (feature transforms) against the direct kernels.

PATH_AUTO takes the transforms where they are faster; PATH_DIRECT never does.  Both evaluate
the same sums in FP32: every difference is rounding.  Descriptor entries lie in [0, w] with
means of order 0.1 .. 1, each side is within a few 1e-7 of the FP64 value of its entry's level
scale, so entries agree to 2e-6 of the largest of their level; gradients agree to 2e-6 normwise
(two FP32 sums of the same terms, each a few 1e-7 from FP64).
"""
import dataclasses

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

TOL = 2e-6

# shape, window, levels, phases; windows large enough that AUTO takes the transforms
SHAPES = [
    ((128, 128), (64, 64), 1, 1),          # window = n / 2: both ends of the window alias
    ((16, 2048), (8, 300), 1, 1),          # shortest and longest register transforms
    ((1024, 32), (200, 16), 1, 1),
    ((256, 512), (32, 33), 3, 1),
    ((512, 256), (48, 48), 2, 2),          # two phases: cross blocks
    ((64, 128), (20, 40), 1, 3),
    ((64, 64, 64), (8, 7, 9), 2, 1),
    ((32, 16, 128), (16, 8, 20), 1, 1),
    ((32, 32, 32), (10, 10, 10), 1, 2),
    ((300, 250), (90, 80), 1, 1),          # mixed radices 2, 3, 5
    ((126, 245), (60, 90), 1, 1),          # 7
    ((264, 169), (100, 80), 1, 1),         # 11, 13: direct prime stages
    ((48, 40, 56), (12, 10, 14), 1, 1),
    ((2048, 96), (40, 48), 1, 1),
]


def _case(dm, shape, window, levels, phases, seed, lo=0.0, hi=1.0):
    rng = np.random.default_rng(seed)
    full = ((phases,) if phases > 1 else ()) + shape
    f = torch.tensor(rng.uniform(lo, hi, full).astype(np.float32), device="cuda")
    p = dm.Params(shape=shape, window=window, levels=levels, phases=phases)
    return f, p, dataclasses.replace(p, path=dm.DMCR_PATH_DIRECT)


def _levels(dm, p, D):
    k = dm.dmcr_descriptor_length(dataclasses.replace(p, levels=1))
    return D.reshape(p.levels, k)


def _separable(dm, p):
    """Whether AUTO runs the transforms for p: their kernels then appear in the profile."""
    f = torch.rand(((p.phases,) if p.phases > 1 else ()) + tuple(p.shape), device="cuda")
    dm.dmcr_profile_enable(True)
    try:
        dm.descriptor(f, p)
        torch.cuda.synchronize()
        names = dm.dmcr_profile_read()
    finally:
        dm.dmcr_profile_enable(False)
        dm.dmcr_profile_reset()
    return any(n.startswith("sep_") for n in names)


def _agree(dm, p, q, f, up):
    a, b = dm.descriptor(f, p), dm.descriptor(f, q)
    for x, y in zip(_levels(dm, p, a), _levels(dm, p, b)):
        assert float((x - y).abs().max()) <= TOL * float(y.abs().max())
    ga, gb = dm.descriptor_vjp(f, up, p), dm.descriptor_vjp(f, up, q)
    assert float(torch.linalg.norm(ga - gb)) <= TOL * float(torch.linalg.norm(gb))
    target = (0.8 * b).contiguous()
    for mode in (0, 1):
        la, ha = dm.loss_grad(f, target, p, dm.LossOpts(mode=mode))
        lb, hb = dm.loss_grad(f, target, q, dm.LossOpts(mode=mode))
        np.testing.assert_allclose(la.cpu().numpy(), lb.cpu().numpy(), rtol=1e-5)
        assert float(torch.linalg.norm(ha - hb)) <= 1e-5 * float(torch.linalg.norm(hb))


@pytest.mark.parametrize("shape,window,levels,phases", SHAPES)
def test_separable_equals_direct(cuda_lib, shape, window, levels, phases):
    dm = cuda_lib
    f, p, q = _case(dm, shape, window, levels, phases, 5)
    assert _separable(dm, p) and not _separable(dm, q)
    up = torch.randn(dm.dmcr_descriptor_length(p), generator=torch.Generator("cuda").manual_seed(1), device="cuda")
    _agree(dm, p, q, f, up)


@pytest.mark.parametrize("lo,hi", [(0.0, 0.0), (0.0, 1.0), (-0.06, 1.06), (-0.3, 1.3), (-0.55, 1.55), (-1.0, 1.6),
                                   (-1.5, 2.0), (-2.3, 2.5), (-3.0, 3.0), (-20.0, 20.0)])
def test_every_value_range(cuda_lib, lo, hi):
    """Each range of the bases, and fields beyond the widest: the gated direct kernels."""
    dm = cuda_lib
    f, p, q = _case(dm, (256, 256), (64, 64), 2, 1, 6, lo, hi)
    f.view(-1)[:2] = torch.tensor([lo, hi], device="cuda")
    up = torch.randn(dm.dmcr_descriptor_length(p), generator=torch.Generator("cuda").manual_seed(2), device="cuda")
    if lo == hi:
        assert float(dm.descriptor(f, p).abs().max()) < 1e-9
        return
    _agree(dm, p, q, f, up)


def test_non_finite_values_take_the_direct_kernels(cuda_lib):
    dm = cuda_lib
    f, p, q = _case(dm, (256, 256), (64, 64), 1, 1, 7)
    up = torch.randn(dm.dmcr_descriptor_length(p), generator=torch.Generator("cuda").manual_seed(3), device="cuda")
    for bad in (float("nan"), float("inf"), -float("inf")):
        h = f.clone()
        h[3, 5] = bad
        for a, b in ((dm.descriptor(h, p), dm.descriptor(h, q)), (dm.descriptor_vjp(h, up, p), dm.descriptor_vjp(h, up, q))):
            assert torch.equal(torch.isnan(a), torch.isnan(b)) and torch.equal(torch.nan_to_num(a), torch.nan_to_num(b))


@pytest.mark.parametrize("alpha", [2.0, 6.0, 20.0, 60.0])
def test_other_slopes(cuda_lib, alpha):
    """A basis of its own per slope; none for the steepest: direct kernels."""
    dm = cuda_lib
    f, p, q = _case(dm, (128, 256), (50, 60), 1, 1, 8)
    p, q = dataclasses.replace(p, alpha=alpha), dataclasses.replace(q, alpha=alpha)
    up = torch.randn(dm.dmcr_descriptor_length(p), generator=torch.Generator("cuda").manual_seed(4), device="cuda")
    _agree(dm, p, q, f, up)
