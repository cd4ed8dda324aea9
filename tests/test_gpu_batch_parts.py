"""A batch of 16 cells per SM or more runs as two parts on two streams: labels, log-likelihoods and parameters are
those of each image alone (always one part), below and above the line, wherever the cells' middle falls, on the
default stream and on one of the caller's, from several threads at once."""
import threading

import numpy as np
import pytest

from synth import voronoi_image

pytestmark = pytest.mark.gpu

# sizes (W, H), spacing: one part (too few cells); two equal images; a first and a last image with most of the cells;
# many small ones and a remainder of a few cells
SIZES = {
    "below": ([(160, 120)] * 2, 8),
    "two": ([(403, 401)] * 2, 8),
    "first": ([(513, 390), (64, 48), (33, 70)], 8),
    "last": ([(64, 48), (17, 9), (513, 390)], 8),
    "many": ([(90 + 3 * i, 70 + 5 * i) for i in range(20)], 7),
}


def run(gm, torch, sizes, v, stream, colour="full", iters=3, bps=None):
    imgs = [torch.from_numpy(voronoi_image(w, h, 12, 8.0, 3 + i)).cuda() for i, (w, h) in enumerate(sizes)]
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        bt = gm.SuperpixelsBatch([(h, w) for w, h in sizes], spacing=v, colour=colour)
        if bps is not None:
            bt.set_launch(bps, bps)
        out = []
        for _ in range(2):
            labels, ll = bt.segment(imgs, iters, want_loglik=True)
            stream.synchronize()
            out.append(([x.cpu().numpy().copy() for x in labels], np.array(ll),
                        [bt.get_params(i, (w // v) * (h // v)) for i, (w, h) in enumerate(sizes)]))
        for x, y in zip(out[0][0] + [out[0][1]], out[1][0] + [out[1][1]]):  # again through the kept graph
            np.testing.assert_array_equal(x, y)
        bt.close()
    return out[0]


@pytest.mark.parametrize("own_stream", [False, True])
@pytest.mark.parametrize("colour", ["full", "split"])
@pytest.mark.parametrize("name", list(SIZES))
def test_parts_equal_single_images(name, colour, own_stream):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_1612_08792_gb300 as gm
    sizes, v = SIZES[name]
    cells = sum(-(-w // v) * -(-h // v) for w, h in sizes)
    assert (cells >= 16 * torch.cuda.get_device_properties(0).multi_processor_count) == (name != "below")
    stream = torch.cuda.Stream() if own_stream else torch.cuda.default_stream()
    imgs = [torch.from_numpy(voronoi_image(w, h, 12, 8.0, 3 + i)).cuda() for i, (w, h) in enumerate(sizes)]
    labels, ll, params = run(gm, torch, sizes, v, stream, colour)
    for i, (w, h) in enumerate(sizes):
        one = gm.SuperpixelsBatch([(h, w)], spacing=v, colour=colour)
        l1, ll1 = one.segment([imgs[i]], 3, want_loglik=True)
        np.testing.assert_array_equal(labels[i], l1[0].cpu().numpy())
        assert ll[i] == ll1[0]
        for x, y in zip(params[i], one.get_params(0, (w // v) * (h // v))):
            np.testing.assert_array_equal(x, y)
        one.close()


def test_parts_from_threads():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_1612_08792_gb300 as gm
    sizes, v = SIZES["many"]
    want = run(gm, torch, sizes, v, torch.cuda.Stream())
    got = [None] * 4

    def work(i):
        got[i] = run(gm, torch, sizes, v, torch.cuda.Stream(), bps=7 if i & 1 else None)
    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    [t.start() for t in threads]
    [t.join() for t in threads]
    for g in got:
        for x, y in zip(want[0] + [want[1]], g[0] + [g[1]]):
            np.testing.assert_array_equal(x, y)
