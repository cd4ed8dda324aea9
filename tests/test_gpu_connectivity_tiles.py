"""Connectivity post-processing at the edges of its tiles (32 x 32 labelling tiles, chunks of 128 pixels by 16 and 8 rows)
against the oracle: exact.  Components that wind through many tiles, widths and heights around the tile sizes,
one-pixel checkerboards (every pixel a component, full adjacency lists), a call large enough for the
multi-block scans, and one of so many pixel rows that tiles and chunks take their full heights."""
import numpy as np
import pytest

from oracle import connectivity as oc

pytestmark = pytest.mark.gpu


def winding(H, W, rng, noise):
    """Comb and ring shaped components that cross tile borders back and forth, with speckles."""
    y, x = np.mgrid[0:H, 0:W]
    L = np.where((y // 3) % 2 == 0, 0, 1)
    L[:, :2] = 0                                     # joins the even stripes
    L[:, -2:] = np.where(y[:, -2:] > 1, 1, 0)        # joins the odd ones
    r = np.maximum(abs(y - H // 2), abs(x - W // 2))
    L = np.where(r % 11 < 4, 2 + r // 11 % 3, L)
    m = rng.random((H, W)) < noise
    L[m] = rng.integers(0, 9, m.sum())
    return L.astype(np.int32)


def run(gm, maps):
    import torch
    for L, lab, K in maps:
        ref, rst = oc.enforce_connectivity(L, lab, K)
        dev = torch.from_numpy(L.copy()).cuda()
        st = gm.gmmsp_enforce_connectivity(dev, torch.from_numpy(np.ascontiguousarray(lab.transpose(2, 0, 1))).cuda(),
                                           L.shape[1], L.shape[0], K)
        assert st == rst
        np.testing.assert_array_equal(dev.cpu().numpy(), ref)


@pytest.mark.parametrize("H,W,K,noise", [(1, 1, 1, 0), (1, 300, 9, 0.2), (260, 1, 9, 0.2), (32, 32, 4, 0.1),
                                         (33, 31, 6, 0.05), (31, 129, 12, 0.1), (65, 128, 20, 0.02), (96, 131, 30, 0.3)])
def test_tile_edges(H, W, K, noise):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1612_08792_gb300 as gm
    rng = np.random.default_rng(H * 1000 + W)
    lab = rng.normal(40, 20, (H, W, 3)).astype(np.float32)
    lab[rng.random((H, W)) < 0.3] = 40.0             # colour ties
    run(gm, [(winding(H, W, rng, noise), lab, K)])


def test_checkerboards():
    import paper_1612_08792_gb300 as gm
    rng = np.random.default_rng(3)
    y, x = np.mgrid[0:40, 0:70]
    lab = rng.normal(0, 30, (40, 70, 3)).astype(np.float32)
    run(gm, [(((x + y) % 2).astype(np.int32), lab, 5), ((x % 3 + 3 * (y % 3)).astype(np.int32), lab, 400)])


def test_large_call_uses_the_multi_block_scans():
    import torch
    import paper_1612_08792_gb300 as gm
    rng = np.random.default_rng(4)
    H, W, K = 520, 530, 4                            # above 2^18 pixels
    L = np.zeros((H, W), dtype=np.int32)
    L[:, W // 2:] = 1
    pts = rng.integers(0, [H, W], (9000, 2))
    L[pts[:, 0], pts[:, 1]] = rng.integers(2, 9, len(pts))
    lab = rng.normal(40, 20, (H, W, 3)).astype(np.float32)
    run(gm, [(L, lab, K)])


@pytest.mark.parametrize("spread", [0.0, 1e-4, 1e-2, 1.0])
def test_near_ties_are_decided_in_fp64(spread):
    """Islands of 1 to 40 members whose neighbours' colours differ by nothing, by less than FP32 can tell, or by
    little: the nearest group and the tie rule are the oracle's."""
    import paper_1612_08792_gb300 as gm
    rng = np.random.default_rng(int(spread * 1e6) + 1)
    H, W, K = 60, 90, 12
    L = (np.arange(W)[None, :] // 15 + 6 * (np.arange(H)[:, None] // 20)).astype(np.int32)
    m = rng.random((H, W)) < 0.25
    L[m] = rng.integers(20, 24, m.sum())
    lab = (np.array([60.0, -35.0, 80.0]) + spread * rng.normal(0, 1, (H, W, 3))).astype(np.float32)
    run(gm, [(L, lab, K)])


def test_full_tile_rows_over_many_images():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_1612_08792_gb300 as gm
    rng = np.random.default_rng(11)
    v, n = 15, 1620
    sizes = [(97, 33), (98, 31), (99, 64), (100, 65), (128, 32), (96, 130), (101, 40), (33, 97)]
    sizes = [sizes[i % 8] for i in range(n)]
    chunk_rows = sum(-(-w // 128) * h for h, w in sizes)
    assert chunk_rows >= 32 * 152 * 32               # the full 32 rows
    maps, ref = [], []
    for i, (h, w) in enumerate(sizes[:8]):
        lab = rng.normal(40, 20, (h, w, 3)).astype(np.float32)
        lab[rng.random((h, w)) < 0.3] = 40.0
        L, K = winding(h, w, rng, 0.02 * (i + 1)), (w // v) * (h // v)
        maps.append((torch.from_numpy(L).cuda(), torch.from_numpy(lab).cuda()))
        ref.append(oc.enforce_connectivity(L, lab, K))
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        bt = gm.SuperpixelsBatch(sizes, spacing=v, lab_input=True)
        bt.segment([maps[i % 8][1] for i in range(n)], 0)      # the CIELAB planes
        for i, x in enumerate(bt.labels):
            x.copy_(maps[i % 8][0])
        st = bt.connectivity()
        got = [x.cpu().numpy() for x in bt.labels]
    for i in range(n):
        np.testing.assert_array_equal(got[i], ref[i % 8][0])
    for key in st:
        assert st[key] == sum(ref[i % 8][1][key] for i in range(n))
    bt.close()
