"""Host code of the plans (plan.cpp, plan_sums.cpp) without a GPU: built here
with the undefined-behaviour sanitizer and a CUDA runtime made of host memory
(plan_host.cpp)."""
import os
import subprocess

import pytest

from paper_2606_27262_gb300 import build as spbuild

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("plan_host") / "plan_host")
    src = [os.path.join(HERE, "plan_host.cpp")] + [os.path.join(spbuild.CSRC, f) for f in ("plan.cpp", "plan_sums.cpp")]
    inc = ["-I", os.path.join(spbuild.cuda_home(), "include"), "-I", os.path.join(spbuild.ROOT, "include")]
    subprocess.run(["g++", "-std=c++17", "-O1", "-g", "-ffp-contract=off", "-fsanitize=undefined",
                    "-fno-sanitize-recover=all", *inc, *src, "-o", exe, "-pthread"], check=True)

    def call(*args):
        r = subprocess.run([exe, *map(str, args)], capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stdout + r.stderr
        return r.stdout

    return call


def test_trial_blocks_end_at_the_last_trial(run):
    """Threads take blocks from a counter that passes the end: near 2^31 trials
    it may not wrap."""
    run("blocks")


def test_no_room_for_the_shared_sum_tables(run):
    """A plan whose direct tables fit is not refused for the larger tables."""
    run("no_room")


@pytest.mark.parametrize("apart", [[], ["apart"]])
def test_delays_that_differ_by_hundreds_of_millions_of_samples(run, apart):
    """Windows and rows too long for any slot: their sizes are not summed in 32
    bits, and no paths are laid out for them (a plan of 64 trials took seconds)."""
    run("late_band", *apart)


# Measured on a GB300, us with the direct kernel and with shared sums.
@pytest.mark.parametrize("nchan,first,step,ndm,n_out,us", [
    (1024, 0, 0.1, 512, 2048, (293, 172)), (4096, 0, 0.1, 64, 1, (1142, 346)), (4096, 300, 0.3, 512, 40000, (4296, 1790)),
    (4096, 900, 1.0, 129, 700, (843, 917)), (4096, 900, 1.0, 129, 16384, (1101, 924)),
    (4096, 900, 1.0, 256, 8192, (825, 919)), (1024, 900, 1.0, 256, 2048, (211, 334)),
    (1024, 900, 1.0, 256, 20000, (495, 335)), (2049, 900, 1.0, 70, 2047, (416, 543)),
    (64, 0, 0.1, 512, 2048, (26, 41)), (64, 0, 0.1, 512, 40000, (81, 108)), (256, 0, 0.1, 512, 12288, (113, 75)),
])
def test_launches_go_to_the_faster_kernel(run, nchan, first, step, ndm, n_out, us):
    direct, sums = us
    assert int(run("clocks", nchan, first, step, ndm, n_out).split()[2]) == (sums < direct)
