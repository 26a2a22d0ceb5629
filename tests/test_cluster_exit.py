"""How a block leaves its cluster in the on-chip solvers: a block whose wait ran out goes straight to the one cluster
barrier that all blocks meet last, so that none leaves while another may still store into its shared memory."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2503_16028_gb300", "csrc")


@pytest.mark.parametrize("source,kernel", [("onchip.cu", "k_onchip("), ("onchip64.cu", "k_onchip64(")])
def test_no_cluster_barrier_between_the_first_and_the_last(source, kernel):
    """Cluster barriers have no bound: one inside the loops is met by the others while a block whose wait ran out
    waits at the last one, which pairs the two and lets that block leave early."""
    text = open(os.path.join(CSRC, source)).read()
    body = text[text.index(kernel):]
    body = body[:body.index("\n}\n")]
    loops = body.index("A.max_outer; ++o")
    assert len(re.findall(r"oc_sync<", body[:loops])) == 1
    assert "oc_sync<" not in body[loops:]
    assert body.rstrip().endswith("oc_leave(t, A.err);")


@pytest.mark.gpu
def test_a_lost_message_ends_in_the_error_flag(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "cluster_exit")
    build = subprocess.run([nvcc, "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a", "-o", exe,
                            os.path.join(HERE, "cluster_exit.cu")], capture_output=True, text=True)
    assert build.returncode == 0, build.stderr[-3000:]
    run = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert run.returncode == 0 and "cluster exit ok" in run.stdout, run.stdout + run.stderr
