"""The reverse pass after a precompute that failed: its kernels, spectra and autocorrelations are
gone, so it reports MVD_ERR_STATE, as the forward run does, and works again after a precompute."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("path", ["direct", "fft"])
def test_backward_after_a_failed_precompute(path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    from paper_1308_0730_gb300 import mvd

    # single taps at different offsets: P_0^* and P_0^* * P_1 do not overlap, so opt1's kernel sums to zero
    psfs = [np.zeros((5, 5, 5), np.float32) for _ in range(2)]
    psfs[0][2, 2, 4] = psfs[1][2, 2, 3] = 1
    views = [np.random.default_rng(v).uniform(1, 2, (12, 16, 16)).astype(np.float32) for v in range(2)]
    with mvd.Deconvolver(views, psfs, "plain", path=path) as d:
        g = torch.ones((12, 16, 16), device="cuda")
        gv = [torch.empty_like(g) for _ in range(2)]
        mvd.mvd_unrolled_forward(d.ctx, 2)
        want = mvd.mvd_unrolled_backward(d.ctx, g, gv, [p.shape for p in psfs])
        with pytest.raises(mvd.MvdError) as e:
            mvd.mvd_precompute_kernels(d.ctx, "opt1")
        assert e.value.status == mvd.MVD_ERR_ARG
        with pytest.raises(mvd.MvdError) as e:
            mvd.mvd_unrolled_backward(d.ctx, g, gv, [p.shape for p in psfs])
        assert e.value.status == mvd.MVD_ERR_STATE
        mvd.mvd_precompute_kernels(d.ctx, "plain")
        got = mvd.mvd_unrolled_backward(d.ctx, g, gv, [p.shape for p in psfs])
        # the flat start's share is summed by atomics: equal to rounding
        assert all(np.allclose(a, b, rtol=1e-4, atol=1e-6) for a, b in zip(got, want))
