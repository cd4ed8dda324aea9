"""The batch context's launch rules that are plain integer arithmetic (gmmsp_batch_rules.h), checked on the host:
a batch's finalizes go one level before the caller's stream, never to the device's most urgent level at once; a
batch that leaves an SM part empty does not start with the tightest register bound."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_rules(tmp_path):
    exe = str(tmp_path / "batch_rules_check")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_1612_08792_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "batch_rules_check.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0 and out.stdout.startswith("ok"), out.stdout + out.stderr


def test_the_context_uses_them():
    text = open(os.path.join(ROOT, "paper_1612_08792_gb300", "csrc", "gmmsp_batch.cu")).read()
    assert "default_blocks(n, cells, b->sm_count" in text
    assert "finalize_priority(prio, most)" in text and "two_parts(" in text and "high_priority" not in text
