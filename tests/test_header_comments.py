"""The public header's bounds-check block: every GMMSP_BND_* site carries its own comment on its line, and the
function that the block describes follows the sites; gmmsp_release_scratch stands outside, behind its comment."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_bounds_sites_and_scratch_release():
    text = open(os.path.join(ROOT, "include", "gmmsp.h")).read()
    start = text.index("#define GMMSP_BND_GP")
    block = text[start:text.index("gmmsp_status gmmsp_bounds_status(")].splitlines()
    assert len(block) == 11
    for i, line in enumerate(block):
        m = re.fullmatch(r"#define GMMSP_BND_[A-Z_]+ (\d+)\s+/\*\s(.*)\*/", line)
        assert m and int(m.group(1)) == i + 1 and "scratch" not in m.group(2), line
    assert "a batch item" in block[-1]
    comment = re.search(r"/\*((?:(?!\*/).)*)\*/\s*gmmsp_status gmmsp_release_scratch\(void\);", text, re.S)
    assert comment and "scratch" in comment.group(1)
