"""C entry points must not throw: the ones below keep their host buffers in the context or allocate them without
exceptions, instead of building a container between the caller's arguments and the return (a failed allocation
there would end the process)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1612_08792_gb300", "csrc")


@pytest.mark.parametrize("path,name", [("gmmsp_batch.cu", "gmmsp_batch_segment"),
                                       ("gmmsp_batch.cu", "gmmsp_batch_first_pass_partials"),
                                       ("gmmsp_cnn.cu", "grad_to_host"),
                                       ("gmmsp_conn.cu", "enforce_connectivity_many")])
def test_no_container_is_built(path, name):
    text = open(os.path.join(CSRC, path)).read()
    body = re.search(r"\n(?:static )?gmmsp_status " + name + r"\([^;{]*\{(.*?)\n\}", text, re.S).group(1)
    assert not re.search(r"std::vector<[^&]*>\s+\w|\.resize\(|new (?!\(std::nothrow\))", body)
