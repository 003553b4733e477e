"""The factors of the compound kernels are scratch of the precompute: a context does not keep them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_factors_are_given_back():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    from paper_1308_0730_gb300 import mvd

    # four views: opt1 builds 12 factors of 61^3 values (10.4 MiB), plain none
    psfs = [np.random.default_rng(v).uniform(0.5, 1.5, (61, 61, 61)).astype(np.float32) for v in range(4)]
    views = [np.ones((64, 64, 64), np.float32) for _ in psfs]
    held = {}
    for variant in ("opt1", "plain", "opt1"):  # the first run loads the kernels
        with mvd.Deconvolver(views, psfs, variant, path="fft", precision="fast") as d:
            d.synchronize()
            held[variant] = torch.cuda.mem_get_info()[0]
    assert abs(held["plain"] - held["opt1"]) < 6 << 20, held
