"""The direct engine's two tile choices give the same bits where their tiles do differ (16 and 8 rows),
and for boxes whose tap planes are staged in rows."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims, box", [((80, 136, 128), (5, 5, 17)), ((43, 186, 40), (3, 17, 15)), ((200, 80, 40), (101, 41, 3)),
                                       ((20, 194, 78), (11, 95, 1)), ((64, 229, 97), (9, 113, 1))])
def test_tile_heights_give_the_same_bits(tmp_path, dims, box):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    from paper_1308_0730_gb300 import mvd

    rng = np.random.default_rng(dims[0])
    psfs = [rng.uniform(0.5, 1.5, box[::-1]).astype(np.float32) for _ in range(2)]
    views = [rng.uniform(1, 50, dims[::-1]).astype(np.float32) for _ in range(2)]
    outs = []
    cache = tmp_path / "t.txt"
    with mvd.Deconvolver(views, psfs, "plain", path="direct") as d:
        d.autotune(str(cache))
    key = open(cache).read().split("|")[0]
    for ty in (8, 4):
        cache.write_text(f"{key}| 1 {ty} 1 1.0\n")
        with mvd.Deconvolver(views, psfs, "plain", path="direct") as d:
            r = d.autotune(str(cache))
            assert r["from_cache"] and r["direct_tile_y"] == ty
            d.iterate(2)
            outs.append(d.result())
    assert np.array_equal(*outs)
