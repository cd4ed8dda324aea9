"""The network's kernels where a block takes several tiles: more tiles than k_conv3 has resident blocks, more
than two per block of k_wgrad3 and more than two row blocks per block of k_pix_bwd, each with a remainder, so
that some blocks take one more than others (accumulators kept in tensor memory over the tiles, barrier phases
after the first, shared memory refilled, the next tile's loads held in registers).  Reference and tolerances:
the BF16-emulating FP64 network oracle, as in the other network tests."""
import numpy as np
import pytest

from oracle import cnn as ocnn

pytestmark = pytest.mark.gpu


def rel_l2(a, b):
    return float(np.linalg.norm(np.ravel(a) - np.ravel(b)) / max(np.linalg.norm(np.ravel(b)), 1e-30))


def cases(sms):
    """(n_x, n_y, v, images, what must exceed its grid): a long grid of 100 columns (102 with the border) at one
    patch per cell, with at least 6 sms + 10 tiles (at most 5 blocks of its 41 KB fit on an SM); one cell of 121
    patches per row block."""
    rows = -(-(6 * sms + 10) * 128 // 102)
    yield (100, rows, 3, 1, "tiles")
    yield (6, 5, 33, -(-(8 * sms + 40) // 30), "row blocks")


@pytest.mark.parametrize("which", [0, 1])
def test_forward_and_gradient_over_many_tiles(which):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_1612_08792_gb300.learned_init import InitNet, init_weights
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nx, ny, v, B, what = list(cases(sms))[which]
    tiles = B * -(-ny * (nx + 2) // 128)
    row_blocks = -(-B * nx * ny // (128 // (v // 3) ** 2))
    if what == "tiles":
        assert tiles > 5 * sms and tiles % (sms // 4) != 0 and tiles > 2 * (sms // 4)
    else:
        assert row_blocks > 2 * 4 * sms and row_blocks % (4 * sms) != 0
    W, H = nx * v, ny * v
    rng = np.random.default_rng(11 + which)
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
