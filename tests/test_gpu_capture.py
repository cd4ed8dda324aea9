"""Steps of a context that the caller captures into a CUDA graph of its own and replays: theta after any mix of
replays and plain calls is that of the same steps called plainly (the first E+M pass after a start has a kernel
of its own, which must not stay in a graph that is replayed on a later theta)."""
import numpy as np
import pytest

from synth import voronoi_image

pytestmark = pytest.mark.gpu

W, H, V = 161, 122, 13


@pytest.fixture()
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_1612_08792_gb300 as gm
    img = torch.from_numpy(voronoi_image(W, H, 20, 8.0, 3)).cuda()
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()

    def capture(fn):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            fn()
        return g

    def replay(g):
        with torch.cuda.stream(stream):
            g.replay()

    with torch.cuda.stream(stream):
        sp = gm.Superpixels(img, spacing=V, stream=stream)
    yield gm, img, stream, sp, capture, replay
    stream.synchronize()
    sp.close()


def plain(gm, img, stream, iters):
    import torch
    with torch.cuda.stream(stream):
        sp = gm.Superpixels(img, spacing=V, stream=stream)
        sp.em_iters(iters)
        p = sp.get_params()
        sp.close()
    return p


def same(got, want):
    for a, b in zip(got, want):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("per_graph", [1, 2])
def test_replayed_iterations(env, per_graph):
    gm, img, stream, sp, capture, replay = env
    g = capture(lambda: sp.em_iters(per_graph))
    for _ in range(3):
        replay(g)
    same(sp.get_params(), plain(gm, img, stream, 3 * per_graph))


def test_replay_between_calls(env):
    gm, img, stream, sp, capture, replay = env
    g = capture(lambda: sp.em_iters(1))
    sp.reinit(img)          # a start
    replay(g)               # theta is general from here on
    sp.em_iters(2)
    same(sp.get_params(), plain(gm, img, stream, 3))
    sp.segment(img, 0)      # the start again
    replay(g)
    sp.em_iters(2)
    same(sp.get_params(), plain(gm, img, stream, 3))


def test_captured_start_has_not_run(env):
    gm, img, stream, sp, capture, replay = env
    sp.em_iters(2)
    g = capture(lambda: sp.reinit(img))
    sp.em_iters(1)
    same(sp.get_params(), plain(gm, img, stream, 3))
    replay(g)
    sp.em_iters(2)
    same(sp.get_params(), plain(gm, img, stream, 2))
