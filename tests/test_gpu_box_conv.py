"""The tiled convolution sums: the direct engine's view update and the compound kernels at the
edges of tiles, splits and staging, against the FP64 oracle."""
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


# tile edges (32 x 16 / 8 / 4 rows, 8 planes), volumes thinner than a tile, boxes of one
# tap, of three (no full group of four), as large as the axis, and of many planes
@pytest.mark.parametrize("dims, box", [
    ((32, 16, 8), (5, 5, 5)), ((33, 17, 9), (7, 3, 9)), ((31, 15, 7), (3, 15, 7)), ((1, 9, 70), (1, 3, 61)),
    ((97, 41, 19), (9, 9, 15)), ((130, 66, 35), (3, 1, 1)), ((64, 4, 3), (63, 3, 3)), ((5, 130, 12), (5, 41, 3)),
    ((40, 36, 44), (13, 11, 41)),
])
def test_direct_update_at_tile_edges(mvd, dims, box):
    w = synth.small_case(40 + dims[0], dims=dims, n_views=2, boxes=[box, box], n_iter=2, asymmetric=True)
    want, _ = oracle.deconvolve(w.views, w.psfs, 2, "efficient")
    with mvd.Deconvolver(w.views, w.psfs, "efficient", path="direct") as d:
        d.iterate(2)
        got = d.result()
    assert rel_err(got, want) < PARITY_TOL, err_report(got, want)


# boxes of which a whole tap plane does not fit in shared memory (staged in rows), uneven
# boxes in one batch, more pairs than one launch takes
@pytest.mark.parametrize("boxes, variant", [
    ([(257, 129, 1), (129, 65, 3)], "efficient"),
    ([(33, 17, 9), (9, 33, 17), (1, 1, 1), (3, 5, 7)], "efficient"),
    ([(7, 9, 5), (9, 7, 5), (5, 7, 9), (7, 5, 9), (9, 5, 7), (5, 9, 7)], "opt1"),
])
def test_compound_kernels_at_box_edges(mvd, boxes, variant):
    dims = tuple(synth.workloads.smooth235(max(8, int(1.15 * max(b[a] for b in boxes)) + 2)) for a in range(3))
    rng = np.random.default_rng(len(boxes))
    psfs = [rng.uniform(0.5, 1.5, size=b[::-1]).astype(np.float32) for b in boxes]
    views = [rng.uniform(1.0, 2.0, size=dims[::-1]).astype(np.float32) for _ in boxes]
    p64 = [p.astype(np.float64) / p.astype(np.float64).sum() for p in psfs]
    c = mvd.mvd_create(views, psfs)
    try:
        try:
            mvd.mvd_precompute_kernels(c, variant)
        except mvd.MvdError as e:  # the kernels are built before an engine is chosen for the grid
            assert e.status == mvd.MVD_ERR_UNSUPPORTED
            pytest.skip("no engine for this grid")
        for v, p in enumerate(psfs):
            want = oracle.compound(p64, v, variant)
            got = mvd.mvd_get_compound_kernel(c, v, p.shape)
            # positive terms: a row's chain of kx and the kx + ky rows' and planes' additions round by at most
            # (kx + ky + 4) 2^-24 of the sum, in each of the two nested convolutions of each factor
            k = max(max(b[0] + b[1] for b in boxes) + 4, 8)
            tol = 2.0 * (len(boxes) - 1) * k * 2.0 ** -24 + 8 * 2.0 ** -24
            assert np.max(np.abs(got - want) / want) < tol
    finally:
        mvd.mvd_destroy(c)
