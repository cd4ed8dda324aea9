"""Warp-wide tensor-core instructions (.sync.aligned) are undefined unless all lanes of the warp execute them
together; whether lanes have come together again after a branch does not show in a run.  So their helpers must
bring the lanes together themselves, and nothing else may issue them."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1612_08792_gb300", "csrc")


def test_aligned_instructions_follow_a_syncwarp():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = open(path).read()
        bodies = re.findall(r"__device__ __forceinline__ [^{;]*\{(.*?)\n\}", text, re.S)
        aligned = re.compile(r'asm volatile\(\s*"[^"]*\.sync\.aligned')
        covered = sum(len(aligned.findall(b)) for b in bodies)
        assert covered == len(aligned.findall(text)), path
        for b in bodies:
            m = aligned.search(b)
            assert m is None or "__syncwarp();" in b[:m.start()], (path, b)
