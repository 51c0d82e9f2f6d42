"""Three-point descriptor and its adjoint where the ensemble's blocks (128 positions x 64 shifts,
eight consecutive shifts and four consecutive positions a thread), the gather's shift chunks and
the paired tiles of G have edges: odd rows, shifts that change row inside a run, padded positions
and shifts, several tiles of G, both thresholds and an upstream gradient that is not symmetric."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

CASES = [((15, 9), (7, 4)), ((7, 6, 5), (2, 3, 2)), ((13, 37), (6, 18)), ((3, 2, 11), (1, 1, 5)), ((16, 24), (8, 12))]


@pytest.mark.parametrize("ident", [0, 1])
@pytest.mark.parametrize("shape,window", CASES)
def test_s3_block_edges(cuda_lib, shape, window, ident):
    dm = cuda_lib
    rng = np.random.default_rng(31)
    M = rng.uniform(-0.3, 1.3, shape).astype(np.float32)
    p = dm.Params(shape=shape, window=window, descriptor=dm.DMCR_DESC_S3,
                  threshold=dm.DMCR_IDENTITY if ident else dm.DMCR_SOFT)
    op = oracle.Params(ndim=len(shape), window=window, threshold="identity" if ident else "soft")
    dev = torch.tensor(M, device="cuda")
    got = dm.descriptor(dev, p).cpu().numpy().astype(np.float64)
    want = oracle.s3_descriptor(M.astype(np.float64), op)
    # operands to 22 bits, FP32 sums rounded every 256-512 terms: a few 1e-7 of the largest entry
    np.testing.assert_allclose(got, want, rtol=1e-5, atol=1e-6 * np.max(np.abs(want)))
    K = oracle.half_window(len(shape), window).shape[0]
    G = rng.standard_normal((K, K)).astype(np.float32)
    g = dm.descriptor_vjp(dev, torch.tensor(G.ravel(), device="cuda"), p).cpu().numpy().astype(np.float64)
    g_ref = oracle.s3_level_vjp(M.astype(np.float64), op, G.astype(np.float64))
    assert np.linalg.norm(g.ravel() - np.ravel(g_ref)) / np.linalg.norm(g_ref) < 1e-5
