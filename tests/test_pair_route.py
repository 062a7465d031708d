"""The double-float step at the limits of what it accepts (csrc/pair.cuh): on the host the
kernels' own step, on the GPU the routes that lead to it."""
import json
import os
import subprocess

import pytest

from paper_2310_15183_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("pair") / "pair_route")
    cuda_inc = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I" + cuda_inc,
                    os.path.join(HERE, "pair_route.cpp"), "-o", exe], check=True)

    def run(*args):
        return json.loads(subprocess.run([exe, *map(str, args)], check=True, capture_output=True,
                                         text=True).stdout)
    return run


def test_a_step_whose_new_state_is_not_finite_is_refused(host):
    """NONFINITE keeps the last finite state: the step leaves the ray as it was and hands it to
    the FP64 step, also where every rate was finite and only the increments overflow."""
    r = host("new_state")
    assert r["n"] == 64 and r["refused"] == r["untouched"] == r["taken"] == r["n"], r
