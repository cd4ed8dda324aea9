"""The register-bound variants of the single-image E+M and label kernels, which the number of blocks chooses: on
either side of every line (3 blocks of one cell, 5, 6, 7 and 8 blocks of four cells per SM) one warp per cell gives the bits of a batch
of that one image (whose kernels do not vary), for every colour model; four warps per cell agree with that to
their summation order; and the allocation-free call gives the labels of a context."""
import numpy as np
import pytest

from synth import voronoi_image

pytestmark = pytest.mark.gpu

V = 4
# cell grids: blocks of one cell (four warps per cell) up to 3 on each of 152 SMs, 3 to 5; blocks of four cells up to 5
# on each, 5 to 6, 6 to 7, 7 to 8, more
GRIDS = [(19, 20), (19, 40), (58, 52), (60, 55), (65, 62), (70, 66), (80, 70)]


def setup(nx, ny):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_1612_08792_gb300 as gm
    W, H = nx * V, ny * V
    img = torch.from_numpy(voronoi_image(W, H, 60, 8.0, nx)).cuda()
    return torch, gm, W, H, img


@pytest.mark.parametrize("colour", ["full", "split", "gray"])
@pytest.mark.parametrize("nx,ny", GRIDS)
def test_variants_agree(nx, ny, colour):
    torch, gm, W, H, img = setup(nx, ny)
    gray = colour == "gray"
    if gray:
        img = img[..., 1].contiguous()
    bt = gm.SuperpixelsBatch([(H, W)], spacing=V, colour=colour, gray_input=gray)
    # a single context finalizes up to 4096 superpixels of the full model with 16 lanes each
    gm.gmmsp_batch_set_tuning(bt.b, 6, colour == "full" and nx * ny <= 4096)
    want, ll = bt.segment([img], 3, want_loglik=True)
    params = bt.get_params(0, nx * ny)
    for wpc in (1, 2, 4):
        sp = gm.Superpixels(img, spacing=V, colour=colour)
        sp.set_launch(wpc)
        labels, trace = sp.segment(img, 3, want_loglik=True)
        plain = sp.segment(img, 3)  # labels without log-likelihood
        assert torch.equal(labels, plain)
        if wpc == 1:
            assert torch.equal(labels, want[0])
            for a, b in zip(sp.get_params(), params):
                np.testing.assert_array_equal(a, b)
        else:
            assert float((labels == want[0]).float().mean()) > 0.999
            for a, b in zip(sp.get_params(), params):
                np.testing.assert_allclose(a, b, rtol=2e-3, atol=2e-3)
        assert trace[-1] == pytest.approx(ll[0], rel=1e-6)
        sp.close()
    bt.close()


@pytest.mark.parametrize("nx,ny", [g for g in GRIDS if g[0] * g[1] <= 4096])
def test_caller_rows(nx, ny):
    torch, gm, W, H, img = setup(nx, ny)
    lab = torch.rand((H, W, 3), device="cuda") * 40 + img.float() / 8
    p = gm.gmmsp_default_params()
    p.spacing, p.input_format = V, gm.GMMSP_LAB32
    out = torch.full((H, W), -1, dtype=torch.int32, device="cuda")
    gm.gmmsp_segment_lab_noalloc(lab, W, H, W * 12, p, 3, out)
    sp = gm.Superpixels(lab, spacing=V)
    sp.em_iters(3)
    assert torch.equal(out, sp.labels())
    sp.close()
