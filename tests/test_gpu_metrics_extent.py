"""The metrics of a map with a side of 2^31 - 1 pixels (any side and radius that fits an int is accepted): the
kernel's columns and rows beside the image are not representable there and must not be formed.  One pixel at
the end is another segment; labels and ground truth are the same map, so every count is known."""
import pytest

pytestmark = [pytest.mark.gpu, pytest.mark.slow]


@pytest.mark.parametrize("tall", [False, True])
@pytest.mark.parametrize("radius", [0, 3])
def test_longest_side(tall, radius):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_1612_08792_gb300 as gm
    n = 2 ** 31 - 1
    if torch.cuda.mem_get_info()[0] < 12 << 30:
        pytest.skip("needs 12 GB of device memory")
    m = torch.zeros((n, 1) if tall else (1, n), dtype=torch.int32, device="cuda")
    m.view(-1)[-1] = 1
    r = gm.gmmsp_segmentation_metrics(m, m, 2, 2, radius)
    assert (r["br_total"], r["br_recovered"]) == (2, 2)
    assert (r["asa_sum"], r["ue_sum"]) == (n, n)
