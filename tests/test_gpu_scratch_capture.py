"""Calls without a context (metrics, connectivity) on a stream that is being captured: refused as before they took
their scratch from a pool, without ending the caller's capture and without a trace in the next call."""
import pytest

pytestmark = pytest.mark.gpu


def test_refused_while_capturing_then_fine():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_1612_08792_gb300 as gm
    labels = torch.arange(48 * 64, device="cuda", dtype=torch.int32).view(48, 64) // 512
    lab = torch.rand((3, 48, 64), device="cuda") * 50
    x = torch.zeros(16, device="cuda")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        want = gm.gmmsp_segmentation_metrics(labels, labels, 6, 6)
        conn = gm.gmmsp_enforce_connectivity(labels.clone(), lab, 64, 48, 6)
    calls = [lambda: gm.gmmsp_segmentation_metrics(labels, labels, 6, 6),
             lambda: gm.gmmsp_segmentation_metrics_many([labels], [labels], 6, 6),
             lambda: gm.gmmsp_enforce_connectivity(labels, lab, 64, 48, 6)]
    for call in calls:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            x += 1
            with pytest.raises(gm.GmmspError):
                call()
        x.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert float(x.sum()) == 16
        with torch.cuda.stream(stream):
            assert gm.gmmsp_segmentation_metrics(labels, labels, 6, 6) == want
            assert gm.gmmsp_enforce_connectivity(labels.clone(), lab, 64, 48, 6) == conn
