"""Fields outside every range of the separable path: the direct kernels of the same call, their
blocks taken one by one from a counter.  The same results as DMCR_PATH_DIRECT, alone, among other
instances and over several steps, in the same time."""
import dataclasses

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _field(shape, seed, wide, phases=1):
    rng = np.random.default_rng(seed)
    f = rng.uniform(0, 1, ((phases,) if phases > 1 else ()) + shape)
    if wide:
        f.reshape(-1)[7] = 3.0
    return torch.tensor(f, dtype=torch.float32, device="cuda")


@pytest.mark.parametrize("wide", [(1, 0, 1), (0, 1, 0), (1, 1, 1)])
def test_batch_of_open_and_closed_gates(cuda_lib, wide):
    """Two phases, three levels and a single small level side by side, beside an instance that
    AUTO plans direct: each as it is alone, and the open ones as PATH_DIRECT."""
    dm = cuda_lib
    ps = [dm.Params(shape=(256, 256), window=(32, 32), levels=3), dm.Params(shape=(128, 256), window=(48, 40), phases=2),
          dm.Params(shape=(64, 64, 64), window=(8, 8, 8), levels=2), dm.Params(shape=(40, 48), window=(5, 6))]
    fs = [_field(p.shape, 3 + i, i < 3 and wide[i], p.phases) for i, p in enumerate(ps)]
    ts = [torch.full((dm.dmcr_descriptor_length(p),), 0.2, device="cuda") for p in ps]
    loss = torch.empty(6 * len(ps), device="cuda")
    grads = [torch.empty_like(f) for f in fs]
    for _ in range(2):                               # the counters start again in every call
        dm.dmcr_loss_grad_batched(ps, dm.LossOpts(), fs, ts, loss, grads)
    for i, p in enumerate(ps):
        l, g = dm.loss_grad(fs[i], ts[i], p)
        assert torch.equal(loss[6 * i:6 * i + 6], l) and torch.equal(grads[i], g)
        if i < 3 and wide[i]:
            q = dataclasses.replace(p, path=dm.DMCR_PATH_DIRECT)
            assert torch.equal(dm.loss_grad(fs[i], ts[i], q)[1], g)


def test_steps_outside_the_ranges(cuda_lib):
    dm = cuda_lib
    p = dm.Params(shape=(256, 256), window=(32, 32), levels=2)
    q = dataclasses.replace(p, path=dm.DMCR_PATH_DIRECT)
    target = torch.full((dm.dmcr_descriptor_length(p),), 0.3, device="cuda")
    out = []
    for x in (p, q):
        f = _field(p.shape, 5, True)
        m, v, loss, ws = torch.zeros_like(f), torch.zeros_like(f), torch.empty(6, device="cuda"), dm.workspace(x)
        step = 0
        for _ in range(5):
            step = dm.dmcr_adam_step(x, dm.ReconOpts(lr=1e-3), target, f, m, v, step, loss, ws)
        out.append((f, m, v))
    for a, b in zip(*out):
        assert torch.equal(a, b)


def test_time_outside_the_ranges(cuda_lib):
    """As PATH_DIRECT, to the start-up of the kernels that find nothing to do (a fixed share of the
    blocks each instead: 11 % longer)."""
    dm = cuda_lib
    p = dm.Params(shape=(96, 96, 96), window=(20, 20, 20), levels=2)
    f = _field(p.shape, 6, True)
    ms = []
    for path in (dm.DMCR_PATH_AUTO, dm.DMCR_PATH_DIRECT):
        x = dataclasses.replace(p, path=path)
        target = torch.full((dm.dmcr_descriptor_length(x),), 0.2, device="cuda")
        loss, grad, ws = torch.empty(6, device="cuda"), torch.empty_like(f), dm.workspace(x)
        times = []
        for i in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            dm.dmcr_loss_grad(x, dm.LossOpts(), f, target, loss, grad, None, ws)
            b.record()
            torch.cuda.synchronize()
            if i >= 3:
                times.append(a.elapsed_time(b))
        ms.append(float(np.median(times)))
    assert ms[0] < 1.05 * ms[1], ms
