"""Boxes so wide that not one row of taps fits in shared memory beside a tile's inputs (rows are staged
in pieces): the direct update and the compound kernels against the FP64 oracle."""
import numpy as np
import pytest

import oracle
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


def _psfs(box, n, seed):
    """A peak on a long tail, off centre."""
    rng = np.random.default_rng(seed)
    x = np.arange(box[0]) - box[0] // 2
    return [(np.exp(-0.5 * ((x - 7 * v) / 40.0) ** 2) + 1e-3 * rng.uniform(0.5, 1.5, box[0]))
            .astype(np.float32)[None, None, :].repeat(box[2], 0).repeat(box[1], 1) for v in range(n)]


# one and three taps more than whole groups of four in the last piece; partial tiles
@pytest.mark.parametrize("dims, box", [((6600, 1, 1), (6397, 1, 1)), ((8200, 3, 2), (8003, 1, 1)),
                                       ((10200, 1, 1), (10001, 1, 1))])
def test_direct_update(mvd, dims, box):
    psfs = _psfs(box, 2, 1)
    rng = np.random.default_rng(2)
    views = [rng.uniform(1, 5, dims[::-1]).astype(np.float32) for _ in psfs]
    want, _ = oracle.deconvolve(views, psfs, 2, "efficient")
    with mvd.Deconvolver(views, psfs, "efficient", path="direct") as d:
        d.iterate(2)
        got = d.result()
    assert rel_err(got, want) < PARITY_TOL, err_report(got, want)


@pytest.mark.parametrize("variant", ["efficient", "opt1"])
def test_compound_kernels(mvd, variant):
    box, dims = (6501, 1, 1), (6561, 1, 2)
    psfs = _psfs(box, 2, 3)
    views = [np.random.default_rng(4).uniform(1, 2, dims[::-1]).astype(np.float32) for _ in psfs]
    p64 = [p.astype(np.float64) / p.astype(np.float64).sum() for p in psfs]
    c = mvd.mvd_create(views, psfs, path="fft")
    try:
        mvd.mvd_precompute_kernels(c, variant)
        for v, p in enumerate(psfs):
            want = oracle.compound(p64, v, variant)
            got = mvd.mvd_get_compound_kernel(c, v, p.shape)
            # positive terms in chains of at most 512 (a piece), the pieces added with compensation:
            # 516 roundings of 2^-24 in each of the two nested convolutions, and the products and norms
            assert np.max(np.abs(got - want) / want) < (2 * 516 + 8) * 2.0 ** -24
    finally:
        mvd.mvd_destroy(c)
