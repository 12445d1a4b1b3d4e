"""qs_explicit_step when a launch fails part way: the state holds the steps that
were completed, in all three arrays and in t and step.  The failing call is a
fake; no GPU is used."""
import os
import subprocess

import pytest

from paper_1904_03808_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    build.build()
    exe = str(tmp_path_factory.mktemp("fault") / "explicit_step_fault")
    cuda = os.path.dirname(os.path.dirname(build._nvcc()))
    subprocess.check_call(
        ["g++", "-std=c++17", "-I", os.path.join(cuda, "include"), "-o", exe,
         os.path.join(HERE, "explicit_step_fault.cpp"), os.path.join(build.OUT_DIR, "qsmg_host.o"),
         "-Wl,--unresolved-symbols=ignore-all"])  # the kernels of the other calls
    return exe


def run(harness, *args):
    out = subprocess.check_output([harness] + [str(a) for a in args], text=True).split()
    return [float(x) for x in out]


@pytest.mark.parametrize("nsteps", [1, 2, 5])
def test_all_steps(harness, nsteps):
    assert run(harness, nsteps) == [0, nsteps, nsteps] + [nsteps] * 6


@pytest.mark.parametrize("done", range(5))
@pytest.mark.parametrize("kernel", range(4))  # stress, chi, velocity, walls
def test_failure_leaves_the_completed_steps(harness, done, kernel):
    st, *rest = run(harness, 5, 4 * done + kernel)
    assert st != 0
    assert rest == [done] * 8
