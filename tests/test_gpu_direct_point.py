"""The direct engine on boxes of one tap, which take no tiles: every form of the update, against the
FP64 oracle; volumes of less than a block, of several and of more than the grid."""
import numpy as np
import pytest

import oracle
from tests._util import PARITY_TOL, err_report, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(4, 4, 4), (33, 17, 9), (160, 80, 60)])
def test_one_tap(dims):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    from paper_1308_0730_gb300 import mvd

    rng = np.random.default_rng(dims[0])
    psfs = [np.full((1, 1, 1), 0.7, np.float32)] * 2
    views = [rng.uniform(1, 20, dims[::-1]).astype(np.float32) for _ in psfs]
    weights = [rng.uniform(0.2, 0.8, dims[::-1]).astype(np.float32) for _ in psfs]

    def check(got, want):
        assert rel_err(got, want) < PARITY_TOL, err_report(got, want)

    with mvd.Deconvolver(views, psfs, path="direct") as d:
        d.iterate(3)
        check(d.result(), oracle.deconvolve(views, psfs, 3)[0])
        d.set_estimate(None)
        d.iterate_combined(3)
        check(d.result(), oracle.deconvolve_combined(views, psfs, 3)[0])
        d.set_weights(weights)
        d.set_regularization(0.01)
        d.set_estimate(None)
        d.iterate(3)
        check(d.result(), oracle.deconvolve_weighted(views, psfs, 3, oracle.normalize_weights(weights)[0], lam=0.01)[0])
