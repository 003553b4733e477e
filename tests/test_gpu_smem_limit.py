"""The dynamic shared-memory limit belongs to a kernel function, not to a launch: objects of other
sizes, made later or by other threads, must not lower it under one that needs more."""
import threading

import numpy as np
import pytest

import synth

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


def _batch(mvd, dims, seed):
    w = synth.small_case(seed, dims=dims, n_views=2, n_iter=1)
    d = mvd.Deconvolver(w.views, w.psfs, path="fft", precision="precise")
    return d, mvd.mvd_batch_create([d], 1, "persistent")


def test_a_smaller_batch_made_later(mvd):
    """On the default stream, where a run launches the kernel anew."""
    big, bb = _batch(mvd, (90, 54, 45), 3)
    small, bs = _batch(mvd, (16, 8, 8), 4)
    try:
        for b in (bb, bs, bb):
            mvd.mvd_batch_run(b)
            mvd.mvd_batch_wait(b)
        plain = mvd.Deconvolver(*(lambda w: (w.views, w.psfs))(synth.small_case(3, dims=(90, 54, 45), n_views=2)),
                                path="fft", precision="precise")
        plain.iterate(2)
        assert np.allclose(big.result(), plain.result(), rtol=1e-4, atol=1e-4)
        plain.close()
    finally:
        for b, d in ((bb, big), (bs, small)):
            mvd.mvd_batch_destroy(b)
            d.close()


def test_threads_with_boxes_of_other_sizes(mvd):
    """Compound kernels and direct updates of small and large boxes, each in a thread of its own."""
    import torch

    cases = [((40, 40, 36), (21, 21, 21)), ((24, 20, 16), (3, 3, 5)), ((40, 40, 36), (15, 27, 13))]
    errors, results = [], [[] for _ in cases]
    start = threading.Barrier(len(cases))

    def run(i):
        try:
            dims, box = cases[i]
            rng = np.random.default_rng(i)
            psfs = [rng.uniform(0.5, 1.5, box[::-1]).astype(np.float32) for _ in range(2)]
            views = [rng.uniform(1, 2, dims[::-1]).astype(np.float32) for _ in range(2)]
            with mvd.Deconvolver(views, psfs, "opt1", path="direct", stream=torch.cuda.Stream()) as d:
                start.wait(60)
                for _ in range(40):
                    mvd.mvd_precompute_kernels(d.ctx, "opt1")
                    d.set_estimate(None)
                    d.iterate(1)
                    results[i].append(d.result().copy())
        except BaseException as e:  # reported by the test's own thread
            errors.append(e)
            start.abort()

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(cases))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for r in results:
        assert all(np.array_equal(a, r[0]) for a in r[1:])
