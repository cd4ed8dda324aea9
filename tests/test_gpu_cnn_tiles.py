"""The 3 x 3 layers' tiles (k_conv3, k_wgrad3) and the fused pixel-level backward pass at the edges of
their tiling: one cell, one column or row, a full tile, strips of 126 columns and their remainders, wide
grids of several strips, cells of 1 and of 121 patches.  Reference: the BF16-emulating FP64 network
oracle; tolerances as for the other network tests (BF16 rounding flips between accumulation orders)."""
import numpy as np
import pytest

from oracle import cnn as ocnn

pytestmark = pytest.mark.gpu


def rel_l2(a, b):
    return float(np.linalg.norm(np.ravel(a) - np.ravel(b)) / max(np.linalg.norm(np.ravel(b)), 1e-30))


# (n_x, n_y, v, images): v = 3 has one patch per cell (128 cells per row block), v = 33 121 of 128 rows
CASES = [(1, 1, 3, 1), (1, 7, 9, 3), (5, 1, 33, 2), (126, 2, 3, 2), (127, 3, 3, 1), (253, 2, 3, 1), (43, 3, 6, 2),
         (6, 16, 15, 1), (130, 1, 12, 1)]


@pytest.mark.parametrize("nx,ny,v,B", CASES)
def test_forward_and_gradient_at_tile_edges(nx, ny, v, B):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_1612_08792_gb300.learned_init import InitNet, init_weights
    W, H = nx * v + v // 2, ny * v + 1            # remainder strips that the network does not read
    rng = np.random.default_rng(nx * 1000 + ny * 10 + v)
    lab = (rng.normal(0, 25, (B, 3, H, W)) + np.array([50, 0, 0])[None, :, None, None]).astype(np.float32)
    tgt = rng.normal(0, 1, (B, nx * ny, 10)).astype(np.float32)
    net = InitNet(v, weights=init_weights(5))
    dev = torch.from_numpy(lab).cuda()
    out = net.forward(dev, B, W, H).cpu().numpy()
    loss, g = net.grad(dev, B, W, H, torch.from_numpy(tgt).cuda())
    net.check()
    ref, cache = ocnn.forward(net.get_weights(), lab, v, emulate_bf16=True)
    assert rel_l2(out, ref) < 2e-3
    ref_loss, g_out = ocnn.loss(ref, tgt)
    gref = ocnn.backward(cache, g_out)
    assert loss == pytest.approx(ref_loss, rel=1e-5)
    o = 0
    for layer, (taps, cout) in enumerate(ocnn.LAYERS):
        for size in (cout * taps * 32, cout):
            assert rel_l2(g[o:o + size], gref[o:o + size]) < 5e-3, (layer, size)
            o += size
    net.close()
