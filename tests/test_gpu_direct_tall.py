"""The direct engine's 16-row tiles, every kernel of them, and the compound kernels of boxes staged in
rows, against the FP64 oracle."""
import numpy as np
import pytest

import oracle
import synth
from tests._direct_shapes import TALL_TILES
from tests._util import PARITY_TOL, err_report, rel_err

pytestmark = pytest.mark.gpu


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


@pytest.mark.parametrize("dims, box", TALL_TILES)
def test_update(mvd, dims, box):
    rng = np.random.default_rng(sum(dims))
    psf = rng.uniform(0.1, 1.0, box[::-1]).astype(np.float32)  # no symmetry: the taps' order shows
    view = rng.uniform(1.0, 20.0, dims[::-1]).astype(np.float32)
    want, _ = oracle.deconvolve([view], [psf], 1, "plain")
    with mvd.Deconvolver([view], [psf], "plain", path="direct") as d:
        d.iterate(1)
        got = d.result()
    assert rel_err(got, want) < PARITY_TOL, err_report(got, want)


# as in test_gpu_box_conv.py, but a box that the tiling refuses fails
@pytest.mark.parametrize("boxes, variant", [
    ([(257, 129, 1), (129, 65, 3)], "efficient"),
    ([(257, 129, 1), (3, 5, 7)], "opt1"),
    ([(33, 17, 9), (9, 33, 17), (1, 1, 1), (3, 5, 7)], "efficient"),
])
def test_compound_kernels(mvd, boxes, variant):
    dims = tuple(synth.workloads.smooth235(max(8, int(1.15 * max(b[a] for b in boxes)) + 2)) for a in range(3))
    rng = np.random.default_rng(len(boxes))
    psfs = [rng.uniform(0.5, 1.5, size=b[::-1]).astype(np.float32) for b in boxes]
    views = [rng.uniform(1.0, 2.0, size=dims[::-1]).astype(np.float32) for _ in boxes]
    p64 = [p.astype(np.float64) / p.astype(np.float64).sum() for p in psfs]
    c = mvd.mvd_create(views, psfs, path="fft")
    try:
        mvd.mvd_precompute_kernels(c, variant)
        for v, p in enumerate(psfs):
            want = oracle.compound(p64, v, variant)
            got = mvd.mvd_get_compound_kernel(c, v, p.shape)
            # positive terms: at most kx + ky + 4 roundings of 2^-24 in each of the two nested
            # convolutions of each factor, and the products and norms
            k = max(b[0] + b[1] for b in boxes) + 4
            assert np.max(np.abs(got - want) / want) < (2 * (len(boxes) - 1) * k + 8) * 2.0 ** -24
    finally:
        mvd.mvd_destroy(c)
