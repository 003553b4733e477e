"""Kernel gradients of the FFT engine, summed over the iterations as spectra:
each kind of axis length that the passes and the z mirror of the cropped
correlation meet, against the FP64 oracle's reverse-mode gradient."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

# relative to the largest component, as in the other gradient tests: FP32
# transforms of a few thousand voxels leave 1e-6 of the volume's norm, and the
# chain through the compound kernels and the view ratio magnifies it up to 1e2
GRAD_TOL = 1e-3


def _rel(got, want):
    got, want = np.asarray(got, np.float64), np.asarray(want, np.float64)
    return float(np.abs(got - want).max() / max(np.abs(want).max(), 1e-300))


@pytest.mark.parametrize("dims,boxes,n_iter", [
    ((32, 16, 16), None, 3),                                     # powers of two: double-float adjoint terms
    ((32, 18, 15), [(5, 3, 15), (3, 5, 1)], 2),                  # mixed y and z, box as long as z and of one plane
    ((15, 9, 25), None, 2),                                      # odd x: FP32 adjoint terms through conjugate spectra
    ((24, 20, 1), [(5, 3, 1), (3, 7, 1), (3, 3, 1)], 4),         # a single plane
    ((16, 16, 32), [(7, 5, 9)], 1),                              # one view, one iteration
])
def test_kernel_gradients(dims, boxes, n_iter):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    from paper_1308_0730_gb300 import autograd as ag

    n = len(boxes) if boxes else 3
    w = synth.small_case(37, dims=dims, n_views=n, boxes=boxes, asymmetric=True, n_iter=n_iter)
    views = torch.from_numpy(np.stack([np.asarray(v, np.float32) for v in w.views])).cuda().requires_grad_(True)
    ps = [torch.from_numpy(np.asarray(p, np.float32)).requires_grad_(True) for p in w.psfs]
    psi = ag.unrolled_deconvolve(views, ps, n_iter, "efficient", "fft")
    truth = torch.from_numpy(np.asarray(w.truth, np.float32)).cuda()
    torch.mean((psi.double() - truth.double()) ** 2).backward()
    _, ogv, ogp, _ = oracle.unrolled_grad(w.views, w.psfs, n_iter, w.truth, "efficient")
    assert _rel(views.grad.cpu().numpy(), np.stack(ogv)) < GRAD_TOL
    for v in range(n):
        assert _rel(ps[v].grad.numpy(), ogp[v]) < GRAD_TOL, f"PSF {v}"
