"""The metrics' tiles (512 x 32 pixels, bit words of 32) at their edges against the metric oracle: exact.
Radii that end inside a word, at its end and at the largest; sparse boundaries, so that the spread of the
superpixel bits decides the result; a batch of uneven images; labels out of range."""
import numpy as np
import pytest

from oracle import metrics as om

pytestmark = pytest.mark.gpu


def blocky(rng, H, W, n, step):
    """A map of n values in blocks of about `step` pixels with a little noise: long runs and few boundaries."""
    m = rng.integers(0, n, (H // step + 1, W // step + 1)).repeat(step, 0).repeat(step, 1)[:H, :W].copy()
    for _ in range(max(1, H * W // 2000)):
        m[rng.integers(H), rng.integers(W)] = rng.integers(n)
    return m.astype(np.int32)


def check(gm, maps, radius, eps=0.05):
    import torch
    dev = [(torch.from_numpy(l).cuda(), torch.from_numpy(g).cuda()) for l, g, _, _ in maps]
    res = gm.gmmsp_segmentation_metrics_many([d[0] for d in dev], [d[1] for d in dev], [m[2] for m in maps],
                                             [m[3] for m in maps], radius, eps)
    for (l, g, _, _), r in zip(maps, res):
        assert r == om.all_metrics(l, g, radius, eps)


@pytest.mark.parametrize("H,W,radius", [(1, 1, 2), (33, 31, 1), (32, 32, 0), (31, 33, 31), (65, 511, 32), (32, 512, 2),
                                        (33, 513, 33), (64, 545, 63), (40, 1057, 64), (97, 130, 2)])
def test_tile_edges_exact(H, W, radius):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1612_08792_gb300 as gm
    rng = np.random.default_rng(H * 7 + W + radius)
    check(gm, [(blocky(rng, H, W, 40, 23), blocky(rng, H, W, 7, 41), 40, 7)], radius)


def test_uneven_batch_scratch_and_bad_ids():
    import torch
    import paper_1612_08792_gb300 as gm
    rng = np.random.default_rng(5)
    maps = [(blocky(rng, H, W, K, 9), blocky(rng, H, W, G, 17), K, G)
            for H, W, K, G in ((48, 70, 300, 33), (5, 700, 1, 1), (130, 64, 31, 400), (32, 513, 64, 32))]
    check(gm, maps, 2)
    gm.gmmsp_release_scratch()
    check(gm, maps, 3, 0.0)
    l, g, K, G = maps[0]
    bad = l.copy()
    bad[20, 33] = K
    with pytest.raises(gm.GmmspError):
        gm.gmmsp_segmentation_metrics(torch.from_numpy(bad).cuda(), torch.from_numpy(g).cuda(), K, G)
