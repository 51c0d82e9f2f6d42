"""The half-spectrum FP64 transforms at the sizes where packing row pairs, cropping to the window
and the columns of a block have edges: odd row counts and lengths, every radix, the aliased
shifts at half the length, one line per block and partly filled blocks."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

CASES = [((15, 9), (7, 4)), ((16, 16), (8, 8)), ((4, 4096), (2, 31)), ((4096, 4), (31, 2)), ((75, 50), (11, 25)),
         ((3, 4, 5), (1, 2, 2)), ((27, 20, 18), (5, 10, 9)), ((2, 135, 40), (1, 6, 7)), ((40, 8, 9), (20, 4, 4))]


@pytest.mark.parametrize("shape,window", CASES)
def test_half_spectrum_edges(cuda_lib, shape, window):
    dm = cuda_lib
    rng = np.random.default_rng(11)
    M = rng.uniform(0, 1, shape).astype(np.float32)
    p = dm.Params(shape=shape, window=window, threshold=dm.DMCR_IDENTITY, path=dm.DMCR_PATH_FFT)
    op = oracle.Params(ndim=len(shape), window=window, threshold="identity")
    H = oracle.half_window(len(shape), window)
    idx = np.unique(np.concatenate([[0, 1, len(H) - 1], rng.choice(len(H), min(40, len(H)), replace=False)]))
    got = dm.descriptor(torch.tensor(M, device="cuda"), p).cpu().numpy().astype(np.float64)[idx]
    # FP64 throughout: the float result is rounded once, its weight (1) is exact
    np.testing.assert_allclose(got, oracle.descriptor_shifts(M.astype(np.float64), op, 0, H[idx]), rtol=2e-7, atol=0)
    G = rng.standard_normal(dm.dmcr_descriptor_length(p)).astype(np.float32)
    g = dm.descriptor_vjp(torch.tensor(M, device="cuda"), torch.tensor(G, device="cuda"), p).cpu().numpy().ravel()
    pos = rng.choice(M.size, min(64, M.size), replace=False)
    want = oracle.level_vjp(M.astype(np.float64), op, G.astype(np.float64), pos)
    # the coefficients and the result are floats: each 6e-8, summed over random signs
    assert np.linalg.norm(g[pos] - want) / np.linalg.norm(want) < 1e-6


@pytest.mark.parametrize("shape,window,levels", [((96, 96, 96), (6, 6, 6), 1), ((64, 48, 80), (9, 12, 7), 2),
                                                 ((1024, 1024), (40, 40), 1), ((128, 128, 128), (4, 4, 5), 1)])
def test_auto_equals_direct_near_the_line(cuda_lib, shape, window, levels):
    """Problems on both sides of the line at which the identity threshold goes to the transforms:
    the chosen path against the direct kernels."""
    dm = cuda_lib
    M = torch.rand(shape, device="cuda", generator=torch.Generator("cuda").manual_seed(5)) * 1.4 - 0.2
    out = []
    for path in (dm.DMCR_PATH_AUTO, dm.DMCR_PATH_DIRECT):
        p = dm.Params(shape=shape, window=window, levels=levels, threshold=dm.DMCR_IDENTITY, path=path)
        target = torch.full((dm.dmcr_descriptor_length(p),), 0.3, device="cuda")
        out.append((dm.descriptor(M, p), *dm.loss_grad(M, target, p)))
    (d1, l1, g1), (d2, l2, g2) = out
    np.testing.assert_allclose(d1.cpu().numpy(), d2.cpu().numpy(), rtol=1e-5, atol=1e-9)
    np.testing.assert_allclose(l1.cpu().numpy(), l2.cpu().numpy(), rtol=1e-5)
    assert float(torch.linalg.norm(g1 - g2) / torch.linalg.norm(g2)) < 1e-5
