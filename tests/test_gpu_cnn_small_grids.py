"""Many images of small cell grids, whose 3 x 3 layers stack images in their tiles: one cell per image in two
stacks, grids of a few cells whose tiles hold several images and cut others, several strips of columns, a stack
whose last images are fewer.  Reference and tolerances: the BF16-emulating FP64 network oracle, as in the other
network tests; and every image's output must have the bits of that image alone."""
import numpy as np
import pytest

from oracle import cnn as ocnn

pytestmark = pytest.mark.gpu


def rel_l2(a, b):
    return float(np.linalg.norm(np.ravel(a) - np.ravel(b)) / max(np.linalg.norm(np.ravel(b)), 1e-30))


# (n_x, n_y, v, images); a stack holds 2^17 positions of (n_y + 1) (n_x + 2) per image
CASES = [(1, 1, 3, 30001), (2, 2, 6, 77), (6, 4, 15, 21), (2, 7, 9, 33), (5, 1, 33, 12), (130, 1, 3, 40),
         (126, 2, 3, 9), (3, 3, 3, 9001)]


@pytest.mark.parametrize("nx,ny,v,B", CASES)
def test_stacked_images(nx, ny, v, B):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_1612_08792_gb300.learned_init import InitNet, init_weights
    W, H = nx * v + v // 2, ny * v + 1
    rng = np.random.default_rng(nx * 1000 + ny * 10 + v)
    lab = (rng.normal(0, 25, (B, 3, H, W)) + np.array([50, 0, 0])[None, :, None, None]).astype(np.float32)
    tgt = rng.normal(0, 1, (B, nx * ny, 10)).astype(np.float32)
    net = InitNet(v, weights=init_weights(5))
    dev = torch.from_numpy(lab).cuda()
    out = net.forward(dev, B, W, H).clone()
    loss, g = net.grad(dev, B, W, H, torch.from_numpy(tgt).cuda())
    net.check()
    for i in (0, 1, B // 2, B - 1):
        alone = net.forward(dev[i:i + 1].contiguous(), 1, W, H)
        assert torch.equal(out.view(B, ny * nx, -1)[i], alone.view(ny * nx, -1)), i
    ref, cache = ocnn.forward(net.get_weights(), lab, v, emulate_bf16=True)
    assert rel_l2(out.cpu().numpy(), ref) < 2e-3
    ref_loss, g_out = ocnn.loss(ref, tgt)
    gref = ocnn.backward(cache, g_out)
    assert loss == pytest.approx(ref_loss, rel=1e-5)
    o = 0
    for layer, (taps, cout) in enumerate(ocnn.LAYERS):
        for size in (cout * taps * 32, cout):
            assert rel_l2(g[o:o + size], gref[o:o + size]) < 5e-3, (layer, size)
            o += size
    net.close()
