"""The mixed-radix line transforms at the edges of their tiles: axes of one point and of one
stage, every radix first and last, lines longer than a block's butterflies, tiles with rows past
the end; both precisions, against the FP64 oracle."""
import numpy as np
import pytest

import oracle
import synth
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


@pytest.mark.parametrize("precision", ["precise", "fast"])
@pytest.mark.parametrize("dims", [(1, 9, 10), (10, 1, 6), (6, 5, 1), (2, 3, 4), (54, 25, 18), (75, 81, 6), (45, 12, 100),
                                  (2400, 3, 2), (3, 2400, 2), (2, 3, 2400), (20, 90, 27)])
def test_mixed_radix_axes(mvd, dims, precision):
    box = tuple(3 if n >= 3 else 1 for n in dims)
    w = synth.small_case(60 + dims[0] % 17, dims=dims, n_views=2, boxes=[box, box], n_iter=2, asymmetric=True)
    # a constant background keeps b away from the floor, where FP32 transforms lose the bar
    views = [v + np.float32(20) for v in w.views]
    want, _ = oracle.deconvolve(views, w.psfs, 2, "efficient")
    with mvd.Deconvolver(views, w.psfs, "efficient", path="fft", precision=precision) as d:
        d.iterate(2)
        got = d.result()
    assert rel_err(got, want) < PARITY_TOL, err_report(got, want)
