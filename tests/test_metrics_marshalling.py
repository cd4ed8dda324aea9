"""gmmsp_segmentation_metrics_many reads a map's first two extents, whatever follows them ((H, W, 1) maps are
accepted, equal sizes or not), and keeps refusing maps that differ or are not contiguous.  The stand-ins have a
null address, so the library refuses the call itself before it touches a device."""
import pytest


class Map:
    is_cuda = True

    def __init__(self, *shape, contiguous=True):
        self.shape, self._c = tuple(shape), contiguous

    def is_contiguous(self):
        return self._c

    def data_ptr(self):
        return 0


@pytest.fixture(scope="module")
def gm():
    from paper_1612_08792_gb300 import build
    build.build()
    import paper_1612_08792_gb300 as gm
    return gm


@pytest.mark.parametrize("shapes", [[(5, 7)] * 3, [(5, 7), (4, 7)], [(5, 7, 1)] * 2, [(5, 7, 1), (6, 7, 1)],
                                    [(5, 7, 1)]])
def test_accepted_shapes_reach_the_library(gm, shapes):
    maps = [Map(*s) for s in shapes]
    with pytest.raises(gm.GmmspError):  # the null addresses
        gm.gmmsp_segmentation_metrics_many(maps, maps, 2, 2, stream=0)


@pytest.mark.parametrize("labels,gts", [([Map(5, 7)], [Map(7, 5)]), ([Map(5, 7, contiguous=False)], [Map(5, 7)]),
                                        ([Map(5, 7)], [Map(5, 7, contiguous=False)]), ([Map(5, 7)], [])])
def test_refused(gm, labels, gts):
    with pytest.raises(ValueError):
        gm.gmmsp_segmentation_metrics_many(labels, gts, 2, 2, stream=0)
