"""The waits of the one-launch factorisation of the innovation covariance (eqn 8), on the CPU.

The kernel's source is compiled for the host (tests/host_cuda.h: every CUDA thread a coroutine, barriers and flags as
the kernel uses them) and run under random schedules that hold warps back at any synchronisation.  Work space starts
as NaN, so a read that no wait orders after its write shows; a barrier that some threads never reach is a deadlock.
"""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SOURCE = os.path.join(os.path.dirname(HERE), "paper_1107_4192_gb300", "csrc", "innov_factor.cu")


def host_source(text):
    """The device code and its sizes, with shared memory handed out by the host scheduler."""
    def swap(old, new):
        nonlocal text
        assert text.count(old) == 1, old
        text = text.replace(old, new)

    swap("extern __shared__ __align__(16) unsigned char smem_raw[];", "unsigned char* smem_raw = emu::shared_memory();")
    swap("__shared__ int ticket_s;", "int& ticket_s = emu::shared_int(0);")
    lines = [ln for ln in text.splitlines() if not ln.startswith("#include")]
    text = "\n".join(lines)
    cut = text.index("kf_status innovation_factor(")
    return text[:cut] + "}  // namespace kfm\n"


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("schedule")
    src = d / "innov_factor_host.inc"
    src.write_text(host_source(open(SOURCE).read()))
    exe = d / "schedule"
    r = subprocess.run([gxx, "-O1", "-std=c++17", "-w", "-ffp-contract=off", "-I", HERE, f'-DSOURCE="{src}"', "-o",
                        str(exe), os.path.join(HERE, "innovation_schedule.cpp")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return str(exe)


def run(program, m, seeds, resident=400, bad=-1, release=0.0, barrier=0.0):
    r = subprocess.run([program, *map(str, (m, seeds, resident, bad, release, barrier))], capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("m", [33, 70])
def test_every_read_is_ordered_after_its_write(program, m):
    """Warps held back where they have released a flag: what they store after it must have a wait of its own (the
    inverse of a diagonal tile by rows, which the rows of L^{-1} read)."""
    run(program, m, 12, release=0.2)


@pytest.mark.parametrize("bad", [0, 40])
def test_a_failure_ends_every_wait(program, bad):
    """A bad pivot while warps are held back after a barrier: every CTA ends and the first pivot is reported."""
    run(program, 70, 16, bad=bad, barrier=0.01)


@pytest.mark.parametrize("resident", [1, 3])
def test_progress_with_few_resident_ctas(program, resident):
    """A task waits only for tasks handed out before it: one resident CTA at a time is enough."""
    run(program, 70, 2, resident=resident)
