"""The gradient assembly of large fields, where a thread takes several positions in turn: every position
of the field, at sizes around the lines of the rule and with a ragged last block, against FP64
autograd of the definition, and the Adam update that the same kernel writes."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

# 2^21 = 2097152 and 2^23 = 8388608 positions a phase are where four and eight positions begin
CASES = [((1440, 1456), 1, 2), ((1456, 1448), 1, 1), ((1024, 2048), 2, 2), ((1448, 1456), 1, 2), ((2904, 2888), 1, 1), ((2904, 2896), 1, 2)]


def _reference(f, up, p):
    """Gradient of up . descriptor, the identity threshold, in FP64."""
    x = f.double().requires_grad_()
    d, M, k = [], x.reshape((p.phases,) + p.shape), 0
    for l in range(p.levels):
        if l:
            M = torch.nn.functional.avg_pool2d(M, 2)
        w, H = 2.0 ** l, oracle.half_window(2, p.window)
        for a in range(p.phases):
            for b in range(p.phases):
                for r in H:
                    s = torch.roll(M[b], (-int(r[0]), -int(r[1])), (0, 1))
                    d.append(w * (0.25 * (M[a] + s) ** 2).mean())
    total = (torch.stack(d) * up.double()).sum()
    return torch.autograd.grad(total, x)[0]


@pytest.mark.parametrize("shape,phases,levels", CASES)
def test_every_position(cuda_lib, shape, phases, levels):
    dm = cuda_lib
    p = dm.Params(shape=shape, window=(1, 1), levels=levels, phases=phases, threshold=dm.DMCR_IDENTITY, path=dm.DMCR_PATH_DIRECT)
    g = torch.Generator("cuda").manual_seed(3)
    f = torch.rand(((phases,) if phases > 1 else ()) + shape, device="cuda", generator=g)
    up = torch.randn(dm.dmcr_descriptor_length(p), device="cuda", generator=g)
    out = torch.full_like(f, float("nan"))
    dm.dmcr_descriptor_vjp(p, f, up, out)
    want = _reference(f, up, p).reshape(out.shape)
    # a sum of 9 shifts a level and phase, each of a few roundings; a position left out is NaN
    assert float((out.double() - want).abs().max()) <= 1e-5 * float(want.abs().max())


@pytest.mark.parametrize("shape", [(1448, 1456), (2904, 2904)])
def test_adam_update_of_every_position(cuda_lib, shape):
    dm = cuda_lib
    p = dm.Params(shape=shape, window=(1, 1), levels=1, threshold=dm.DMCR_IDENTITY, path=dm.DMCR_PATH_DIRECT)
    f = torch.rand(shape, device="cuda", generator=torch.Generator("cuda").manual_seed(4)) * 1.2 - 0.1
    target = torch.full((dm.dmcr_descriptor_length(p),), 0.1, device="cuda")
    o = dm.ReconOpts(lr=1e-2, eps=1e-12)
    _, grad = dm.loss_grad(f, target, p)
    M, m, v, loss = f.clone(), torch.zeros_like(f), torch.zeros_like(f), torch.empty(6, device="cuda")
    dm.dmcr_adam_step(p, o, target, M, m, v, 0, loss, dm.workspace(p))
    b1, b2 = np.float32(o.beta1), np.float32(o.beta2)
    g = grad.double()
    wm, wv = float(np.float32(1) - b1) * g, float(np.float32(1) - b2) * g * g
    # one to three roundings of a product; M: its own rounding, 1.2 * 2^-24, and
    # a few of a step of lr
    assert float((m.double() - wm).abs().max()) <= 3e-7 * float(wm.abs().max())
    assert float((v.double() - wv).abs().max()) <= 3e-7 * float(wv.abs().max())
    lr_t = o.lr * (1 - float(b2)) ** 0.5 / (1 - float(b1))
    step = lr_t * wm / (wv.sqrt() + o.eps)
    assert float((M.double() - (f.double() - step)).abs().max()) <= 2e-4 * o.lr
