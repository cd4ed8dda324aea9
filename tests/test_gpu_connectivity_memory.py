"""Device scratch of the connectivity post-processing: 112 bytes per pixel of the call (a call that fits the device
today must fit tomorrow), and the same labels from the rings of group members whatever order they are joined in."""
import numpy as np
import pytest

from oracle import connectivity as oconn

pytestmark = pytest.mark.gpu


def test_scratch_bytes_per_pixel():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_1612_08792_gb300 as gm
    n, H, W = 48, 1024, 1024
    x = torch.full((n, H, W, 3), 90, dtype=torch.uint8, device="cuda")
    bt = gm.SuperpixelsBatch([(H, W)] * n, spacing=32)
    bt.segment_stacked(x, 0)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    bt.connectivity()
    used = before - torch.cuda.mem_get_info()[0]
    assert used <= 112 * n * H * W + (8 << 20), used / (n * H * W)
    bt.close()


@pytest.mark.parametrize("W,H,v,levels,seed", [(97, 61, 12, 3, 0), (160, 120, 20, 2, 1), (64, 200, 30, 5, 2),
                                               (230, 31, 15, 2, 3)])
def test_long_merge_chains(W, H, v, levels, seed):
    """Labels of a few levels drawn per pixel: clusters of many small components, whose groups merge into groups."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_1612_08792_gb300 as gm
    rng = np.random.default_rng(seed)
    K = (W // v) * (H // v)
    labels = rng.integers(0, levels, (H, W)).astype(np.int32)
    labels[: H // 3] = np.where(rng.random((H // 3, W)) < 0.9, 0, labels[: H // 3])
    lab = (rng.normal(0, 20, (3, H, W)) + np.array([50, 0, 0])[:, None, None]).astype(np.float32)
    got = torch.from_numpy(labels).cuda()
    stats = gm.gmmsp_enforce_connectivity(got, torch.from_numpy(lab).cuda(), W, H, K)
    want, wstats = oconn.enforce_connectivity(labels, lab.transpose(1, 2, 0), K)
    np.testing.assert_array_equal(got.cpu().numpy(), want)
    assert stats == wstats
