"""The copy's two producer warps leave their loop at the same round whichever
of their waits give up (a producer alone at their barrier would never leave):
the kernel's own round keeping, run on the host over every interleaving."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2609_18703_gb300", "csrc")


def _run(tmp_path, *flags):
    exe = str(tmp_path / "model")
    subprocess.run([shutil.which("g++"), "-std=c++17", "-O1", "-I", CSRC, *flags,
                    os.path.join(HERE, "copy_rounds_model.cpp"), "-o", exe], check=True)
    return subprocess.run([exe], capture_output=True, text=True)


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_producers_leave_together(tmp_path):
    r = _run(tmp_path)
    assert r.returncode == 0, r.stdout


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_the_model_finds_a_producer_left_alone(tmp_path):
    r = _run(tmp_path, "-DPRIVATE_BASE")
    assert r.returncode == 1 and "waits at the barrier" in r.stdout, r.stdout


def _copy_kernel():
    with open(os.path.join(CSRC, "k_assemble.cu")) as f:
        src = f.read()
    return src[src.index("asm_copy_kernel(const __grid_constant__"):src.index("void launch_assemble_plan")]


def test_the_exit_ticket_is_drawn_behind_a_barrier():
    """The last CTA out of a copy advances the cursor, which every warp reads at
    its start: on every path a CTA barrier lies between its warps' reads and its
    ticket."""
    body = _copy_kernel()
    read = max(body.index("= *a.plan.hdr;"), body.index("= a.cursor ? *a.cursor"))
    assert "\n  __syncthreads();" in body[read:body.index("ticket(&ds->exit_ctr[TS_ASM_COPY])")]   # (two spaces in: for all paths)


def test_a_late_cta_of_a_copy_changes_nothing():
    """A CTA that starts after the copy's last participant is out may read the
    advanced cursor: CTA 0 alone reports a refusal, and nothing else that decides
    who takes part (the plan's header) is written by the copy."""
    body = _copy_kernel()
    head = body[:body.index("if (blockIdx.x >= n_part) return;")]
    marks = [line for line in head.splitlines() if "atomicOr(&ds->err" in line]
    assert len(marks) == 2 and all(line.strip().startswith("if (blockIdx.x + threadIdx.x == 0)") for line in marks)
    assert "plan.hdr->" not in body
