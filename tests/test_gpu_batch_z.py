"""The persistent batch kernel on volumes whose axes take its register-resident double-float tiles (64,
128 and 256 points), mixed with others in one launch, against per-volume runs and the FP64 oracle."""
import pytest

import oracle
import synth
from tests._util import PARITY_TOL, err_report, rel_err

pytestmark = pytest.mark.gpu


# columns that do not fill a z tile (Y = 15, 33), several tiles, every length on every axis
@pytest.mark.parametrize("specs", [
    [(12, 15, 128), (10, 33, 256), (9, 20, 64)],
    [(64, 12, 128), (128, 10, 9), (256, 9, 8), (10, 256, 6)],
    [(128, 64, 256), (24, 20, 45)],
])
def test_register_resident_axes(specs):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    from paper_1308_0730_gb300 import mvd

    smooth = [tuple(synth.workloads.smooth235(n) for n in dims) for dims in specs]
    ws = [synth.small_case(900 + i, dims=d, n_views=2, n_iter=2, asymmetric=True) for i, d in enumerate(smooth)]
    s = torch.cuda.Stream()
    plain = []
    for w in ws:
        with mvd.Deconvolver(w.views, w.psfs, "efficient", path="fft", stream=s) as d:
            d.iterate(2)
            plain.append(d.result())
    ds = [mvd.Deconvolver(w.views, w.psfs, "efficient", path="fft", stream=s) for w in ws]
    try:
        b = mvd.mvd_batch_create(ds, 2, "persistent")
        try:
            mvd.mvd_batch_run(b)
            mvd.mvd_batch_wait(b)
            got = [d.result() for d in ds]
        finally:
            mvd.mvd_batch_destroy(b)
    finally:
        for d in ds:
            d.close()
    for w, g, p in zip(ws, got, plain):
        assert rel_err(g, p) < PARITY_TOL, f"{w.name}: {err_report(g, p)}"
        if g.size < 200000:
            want, _ = oracle.deconvolve(w.views, w.psfs, 2, "efficient")
            assert rel_err(g, want) < PARITY_TOL, f"{w.name}: {err_report(g, want)}"


@pytest.mark.parametrize("dims", [(64, 12, 9), (128, 10, 9), (256, 9, 8), (128, 64, 64), (64, 33, 10)])
def test_fp32_x_tiles(dims):
    """FP32 persistent runs on register-resident x lengths: full tiles and tiles with rows past the end."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import numpy as np

    import __graft_entry__

    __graft_entry__.build()
    from paper_1308_0730_gb300 import mvd

    dims = tuple(synth.workloads.smooth235(n) for n in dims)
    w = synth.small_case(950, dims=dims, n_views=2, n_iter=2, asymmetric=True)
    # a constant background keeps b away from the floor, where FP32 transforms lose the bar
    views = [v + np.float32(20) for v in w.views]
    want, _ = oracle.deconvolve(views, w.psfs, 2, "efficient")
    with mvd.Deconvolver(views, w.psfs, "efficient", path="fft", precision="fast", stream=torch.cuda.Stream()) as d:
        b = mvd.mvd_batch_create([d], 2, "persistent")
        try:
            mvd.mvd_batch_run(b)
            mvd.mvd_batch_wait(b)
            got = d.result()
        finally:
            mvd.mvd_batch_destroy(b)
    assert rel_err(got, want) < PARITY_TOL, err_report(got, want)
