"""Precise mode at dim voxels beside bright ones, where only the low parts of the double-float
lines keep the blur: a background of 1 with beads of 1e5, every line form, against the FP64 oracle.

An FP32 transform leaves an absolute error of about 2^-24 of the beads' level, 1e-3 and more of
the background. Double-float leaves 1e-10 of it; what remains is FP32 rounding of values near
their own size: the estimate, b, the view ratio, r - 1 through an x transform, c and the product
(6 a view update, the transform's spread over log2(X) <= 7 stages), for 4 updates of at most
2^-24 each: (5 + 7) 4 2^-24 = 2.9e-6. The bar is 1e-5, and the FP32 mode must miss it.
"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

BAR = 1e-5


@pytest.fixture(scope="module")
def mvd():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    from paper_1308_0730_gb300 import mvd as m

    m.load()
    return m


@pytest.mark.parametrize("dims", [(54, 25, 18), (75, 81, 6), (45, 12, 100), (20, 90, 27), (10, 9, 8), (128, 32, 64),
                                  (256, 15, 128)])
def test_dim_voxels_beside_beads(mvd, dims):
    X, Y, Z = dims
    box = tuple(5 if n >= 5 else 3 for n in dims)
    psfs = synth.small_case(70, dims=dims, n_views=2, boxes=[box, box], asymmetric=True).psfs
    rng = np.random.default_rng(X)
    truth = np.ones((Z, Y, X))
    n = max(2, X * Y * Z // 4000)
    truth[rng.integers(0, Z, n), rng.integers(0, Y, n), rng.integers(0, X, n)] = 1e5
    views = [oracle.conv(truth, p).astype(np.float32) for p in psfs]
    x = np.arange(X) / X
    start = (truth * (1 + 0.2 * np.sin(2 * np.pi * x))[None, None, :]).astype(np.float32)
    want, _ = oracle.deconvolve(views, psfs, 2, psi_init=start)
    err = {}
    for precision in ("precise", "fast"):
        with mvd.Deconvolver(views, psfs, path="fft", precision=precision) as d:
            d.set_estimate(start)
            d.iterate(2)
            err[precision] = float(np.max(np.abs(d.result() - want) / want))
    assert err["precise"] < BAR, err
    assert err["fast"] > BAR, err
