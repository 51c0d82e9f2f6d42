"""Accuracy of the separable path entry by entry, against the FP64 oracle and the direct kernels:
dilute media, whose entries are small against the values of a bright pixel, in every range of
values; grey backgrounds; dark fields; the corrected descriptor; several phases.

Bounds: descriptor entries within 1e-5 relative plus 1e-9 absolute of FP64, gradients within 1e-5
normwise, as in test_gpu_parity.py.  Against the direct kernels, whose own error is below 1e-6
relative, 1.1e-5.
"""
import ctypes
import dataclasses

import numpy as np
import pytest
import torch

import oracle
import synthetic

pytestmark = pytest.mark.gpu

RTOL, ATOL, GTOL = 1e-5, 1e-9, 1e-5
SHAPE, WINDOW, LEVELS = (256, 256), (32, 32), 3


def _dev(a):
    return torch.tensor(np.asarray(a, dtype=np.float32), device="cuda")


def _f64(a):
    return np.asarray(a, dtype=np.float32).astype(np.float64)


def _separable(dm, p, f):
    """Whether AUTO plans the transforms for p: their kernels then appear in the profile."""
    dm.dmcr_profile_enable(True)
    try:
        dm.descriptor(f, p)
        torch.cuda.synchronize()
        names = dm.dmcr_profile_read()
    finally:
        dm.dmcr_profile_enable(False)
        dm.dmcr_profile_reset()
    return any(n.startswith("sep_") for n in names)


def _op(p):
    return oracle.Params(ndim=len(p.shape), window=tuple(p.window), levels=p.levels, alpha=p.alpha)


def _sampled_shifts(p, count, seed):
    H = oracle.half_window(len(p.shape), p.window)
    idx = np.random.default_rng(seed).choice(len(H), count, replace=False)
    return np.unique(np.concatenate([[0, 1, len(H) - 1], idx])), H


def _check_descriptor(dm, p, M, got, direct):
    np.testing.assert_allclose(got, direct, rtol=1.1 * RTOL, atol=ATOL)
    idx, H = _sampled_shifts(p, 24, 1)
    for l in range(p.levels):
        want = oracle.descriptor_shifts(_f64(M), _op(p), l, H[idx])
        np.testing.assert_allclose(got[l * len(H) + idx], want, rtol=RTOL, atol=ATOL, err_msg="level %d" % l)


def _check(dm, p, M):
    q = dataclasses.replace(p, path=dm.DMCR_PATH_DIRECT)
    f = _dev(M)
    assert _separable(dm, p, f) and not _separable(dm, q, f)
    got, direct = (dm.descriptor(f, x).cpu().numpy().astype(np.float64) for x in (p, q))
    _check_descriptor(dm, p, M, got, direct)
    rng = np.random.default_rng(2)
    G = rng.standard_normal(got.size).astype(np.float32)
    g, gd = (dm.descriptor_vjp(f, _dev(G), x).cpu().numpy().astype(np.float64).ravel() for x in (p, q))
    assert np.linalg.norm(g - gd) <= 1.1 * GTOL * np.linalg.norm(gd)
    # positions of the medium and of the background alike
    bright = np.flatnonzero(np.asarray(M).ravel() > 0.5)
    pos = np.unique(np.concatenate([rng.choice(bright, min(24, bright.size), replace=False), rng.choice(g.size, 40)]))
    want = oracle.vjp_at(_f64(M), _op(p), _f64(G), pos)
    assert np.linalg.norm(g[pos] - want) <= GTOL * np.linalg.norm(want)
    target = _dev(0.8 * direct)
    for mode in (0, 1):
        (la, ha), (lb, hb) = (dm.loss_grad(f, target, x, dm.LossOpts(mode=mode)) for x in (p, q))
        np.testing.assert_allclose(la.cpu().numpy(), lb.cpu().numpy(), rtol=1.1 * RTOL)
        assert float(torch.linalg.norm(ha - hb)) <= 1.1 * GTOL * float(torch.linalg.norm(hb))


@pytest.mark.parametrize("pixel", [1.0, 1.2, 1.5, 1.65, 2.0, 2.4])
@pytest.mark.parametrize("vf", [0.01, 0.02, 0.05, 0.35])
def test_dilute_media_in_every_range(cuda_lib, vf, pixel):
    """A medium with one overshooting pixel, which takes the field to a wider range."""
    dm = cuda_lib
    M = synthetic.target_2d_grf(SHAPE[0], 6.0, vf, seed=int(1000 * vf))
    M[5, 7] = pixel
    _check(dm, dm.Params(shape=SHAPE, window=WINDOW, levels=LEVELS), M)


@pytest.mark.parametrize("pixel", [1.0, 1.5, 2.4])
@pytest.mark.parametrize("low,high", [(-0.05, 0.05), (0.1, 0.1), (0.3, 0.3), (0.0, 0.3), (0.5, 0.5)])
def test_grey_backgrounds(cuda_lib, low, high, pixel):
    dm = cuda_lib
    rng = np.random.default_rng(4)
    M = rng.uniform(low, high, SHAPE)
    M[rng.random(SHAPE) < 0.002] = 1.0
    M[9, 3] = pixel
    _check(dm, dm.Params(shape=SHAPE, window=WINDOW, levels=LEVELS), M)


@pytest.mark.parametrize("phases", [1, 2])
@pytest.mark.parametrize("low,high", [(0.0, 0.02), (0.0, 0.1), (0.0, 0.49), (0.3, 0.3), (-0.05, 0.0), (-2.0, -0.1)])
def test_dark_fields_take_the_direct_kernels(cuda_lib, low, high, phases):
    """Without a value of 1/2 (in one phase of several) the pairs are small against the rounding
    of the features: the direct kernels of the same call, bit for bit."""
    dm = cuda_lib
    rng = np.random.default_rng(8)
    M = rng.uniform(low, high, ((phases,) if phases > 1 else ()) + SHAPE)
    if phases > 1:
        M[0] = rng.uniform(0.0, 1.0, SHAPE)
    p = dm.Params(shape=SHAPE, window=WINDOW, levels=2, phases=phases)
    q = dataclasses.replace(p, path=dm.DMCR_PATH_DIRECT)
    f = _dev(M)
    assert _separable(dm, p, f)
    up = _dev(rng.standard_normal(dm.dmcr_descriptor_length(p)))
    assert torch.equal(dm.descriptor(f, p), dm.descriptor(f, q))
    assert torch.equal(dm.descriptor_vjp(f, up, p), dm.descriptor_vjp(f, up, q))


@pytest.mark.parametrize("shape,window,levels", [((256, 256), (32, 32), 3), ((96, 96, 96), (8, 8, 8), 1),
                                                 ((64, 64, 64), (8, 8, 8), 2)])
@pytest.mark.parametrize("vf,pixel", [(0.02, 1.0), (0.02, 2.0), (0.35, 1.5)])
def test_corrected_descriptor(cuda_lib, shape, window, levels, vf, pixel):
    """S_tilde on the separable path: (S_bar(r) - q S_bar(0)) / (1 - q) beyond r = 0, and its VJP and
    loss against the direct kernels'."""
    dm = cuda_lib
    rng = np.random.default_rng(6)
    M = (rng.random(shape) < vf).astype(np.float64)
    M.reshape(-1)[11] = pixel
    p = dm.Params(shape=shape, window=window, levels=levels, descriptor=dm.DMCR_DESC_S2_TILDE)
    q = dataclasses.replace(p, path=dm.DMCR_PATH_DIRECT)
    f = _dev(M)
    assert _separable(dm, p, f) and not _separable(dm, q, f)
    got, direct = (dm.descriptor(f, x).cpu().numpy().astype(np.float64) for x in (p, q))
    idx, H = _sampled_shifts(p, 12, 3)
    c1, _, c3 = oracle.soft_constants(10.0)
    qt = 2.0 * (c1 / (1.0 + np.exp(2.5)) + c3) ** 2
    K = len(H)
    atol = 1e-6 * np.max(np.abs(direct))          # the bound of the corrected descriptor in test_gpu_tilde.py
    for l in range(levels):
        S = oracle.descriptor_shifts(_f64(M), _op(p), l, H[idx])
        want = np.where(idx == 0, S, (S - qt * S[0]) / (1.0 - qt))
        np.testing.assert_allclose(got[l * K + idx], want, rtol=RTOL, atol=atol, err_msg="level %d" % l)
    np.testing.assert_allclose(got, direct, rtol=1.1 * RTOL, atol=1.1 * atol)
    up = _dev(rng.standard_normal(got.size))
    g, gd = dm.descriptor_vjp(f, up, p), dm.descriptor_vjp(f, up, q)
    assert float(torch.linalg.norm(g - gd)) <= 1.1 * GTOL * float(torch.linalg.norm(gd))
    target = _dev(0.8 * direct)
    (la, ha), (lb, hb) = dm.loss_grad(f, target, p), dm.loss_grad(f, target, q)
    np.testing.assert_allclose(la.cpu().numpy(), lb.cpu().numpy(), rtol=1.1 * RTOL)
    assert float(torch.linalg.norm(ha - hb)) <= 1.1 * GTOL * float(torch.linalg.norm(hb))


@pytest.mark.parametrize("shape,window,levels", [((256, 256), (32, 32), 2), ((32, 32, 32), (10, 10, 10), 1),
                                                 ((300, 250), (90, 80), 1)])
@pytest.mark.parametrize("pixel", [1.0, 1.5, 2.4])
def test_dilute_phases(cuda_lib, shape, window, levels, pixel):
    """Two phases of 2 % and 20 %: their cross blocks carry the means of both."""
    dm = cuda_lib
    rng = np.random.default_rng(9)
    u = rng.random(shape)
    M = np.stack([(u < 0.02), (u > 0.8)]).astype(np.float64)
    M[0].reshape(-1)[5] = pixel
    p = dm.Params(shape=shape, window=window, levels=levels, phases=2)
    q = dataclasses.replace(p, path=dm.DMCR_PATH_DIRECT)
    f = _dev(M)
    assert _separable(dm, p, f) and not _separable(dm, q, f)
    a, b = (dm.descriptor(f, x).cpu().numpy().astype(np.float64) for x in (p, q))
    np.testing.assert_allclose(a, b, rtol=1.1 * RTOL, atol=ATOL)
    up = _dev(rng.standard_normal(a.size))
    g, gd = dm.descriptor_vjp(f, up, p), dm.descriptor_vjp(f, up, q)
    assert float(torch.linalg.norm(g - gd)) <= 1.1 * GTOL * float(torch.linalg.norm(gd))


@pytest.mark.parametrize("shape,window", [((2048, 96), (40, 48)), ((96, 2048), (48, 40)), ((264, 169), (100, 80)),
                                          ((32, 16, 128), (16, 8, 20)), ((48, 40, 56), (12, 10, 14))])
@pytest.mark.parametrize("pixel", [1.0, 2.0])
def test_dilute_media_of_every_row_kernel(cuda_lib, shape, window, pixel):
    """Rows of one line a block, lengths that are no power of two, 3-D."""
    dm = cuda_lib
    rng = np.random.default_rng(10)
    M = (rng.random(shape) < 0.02).astype(np.float64)
    M.reshape(-1)[7] = pixel
    _check(dm, dm.Params(shape=shape, window=window), M)


@pytest.mark.parametrize("alpha,separable", [(2.0, True), (6.0, True), (12.0, True), (20.0, True), (60.0, False)])
def test_the_path_of_other_slopes(cuda_lib, alpha, separable):
    dm = cuda_lib
    p = dm.Params(shape=(128, 256), window=(50, 60), alpha=alpha)
    rng = np.random.default_rng(12)
    M = (rng.random(p.shape) < 0.05).astype(np.float64)
    f = _dev(M)
    assert _separable(dm, p, f) == separable
    a = dm.descriptor(f, p).cpu().numpy().astype(np.float64)
    b = dm.descriptor(f, dataclasses.replace(p, path=dm.DMCR_PATH_DIRECT)).cpu().numpy().astype(np.float64)
    _check_descriptor(dm, p, M, a, b)


@pytest.mark.parametrize("vf,pixel", [(0.01, 2.0), (0.35, 1.0)])
def test_noalloc_is_the_direct_evaluation(cuda_lib, vf, pixel):
    """dmcr_descriptor_noalloc on a problem that dmcr_descriptor runs by transforms."""
    dm = cuda_lib
    from paper_2103_09686_gb300 import _lib
    M = synthetic.target_2d_grf(SHAPE[0], 6.0, vf, seed=3)
    M[5, 7] = pixel
    p, f = dm.Params(shape=SHAPE, window=WINDOW, levels=LEVELS), _dev(M)
    assert _separable(dm, p, f)
    got = torch.empty(dm.dmcr_descriptor_length(p), device="cuda")
    lib = _lib.load()
    st = lib.dmcr_descriptor_noalloc(ctypes.byref(p.c()), f.data_ptr(), got.data_ptr(),
                                     torch.cuda.current_stream().cuda_stream)
    assert st == 0, lib.dmcr_last_error().decode()
    assert torch.equal(got, dm.descriptor(f, dataclasses.replace(p, path=dm.DMCR_PATH_DIRECT)))
    np.testing.assert_allclose(got.cpu().numpy(), dm.descriptor(f, p).cpu().numpy(), rtol=1.1 * RTOL, atol=ATOL)
