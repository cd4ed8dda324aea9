"""A single context's first E+M pass after a start runs without the zero off-diagonal terms: the same bits as the
general pass on the same theta (given back through set_params), at every launch shape, after every kind of start,
and only then."""
import numpy as np
import pytest

from synth import voronoi_image

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,v", [(97, 61, 8), (128, 96, 15), (70, 52, 6)])
@pytest.mark.parametrize("wpc", [1, 2, 4])
def test_first_pass_bits(W, H, v, wpc):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_1612_08792_gb300 as gm
    img = torch.from_numpy(voronoi_image(W, H, 12, 8.0, 5)).cuda()
    a, b = gm.Superpixels(img, spacing=v), gm.Superpixels(img, spacing=v)
    K = a.grid.K
    rng = np.random.default_rng(1)
    dmu, le = (torch.from_numpy(rng.normal(0, s, (K, 5)).astype(np.float32)).cuda() for s in (0.2, 0.5))

    def compare(iters):
        b.set_params(*a.get_params())              # the general pass from here
        ll = [s.em_iters(iters, want_loglik=True) for s in (a, b)]
        np.testing.assert_array_equal(*ll)
        for x, y in zip(a.get_params(), b.get_params()):
            np.testing.assert_array_equal(x, y)
    for s in (a, b):
        s.set_launch(wpc)
    compare(1)                                     # the start's theta
    compare(2)                                     # fitted theta: no longer diagonal
    a.reinit(img)
    compare(2)
    a.set_init(dmu, le)
    compare(2)
    lab = [s.segment(img, 3).cpu().numpy() for s in (a, b)]
    np.testing.assert_array_equal(*lab)
    compare(1)                                     # after a segment (and its replay) theta is fitted
    a.segment(img, 0)
    compare(1)
    a.close()
    b.close()
