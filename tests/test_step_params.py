"""The host side of a step's parameters, compiled and run without a GPU."""
import os
import re
import subprocess

import pytest

from paper_1411_6121_gb300 import _build

PROGRAM = r"""
#include <string.h>
#include <stdio.h>
#include "dugks_device.cuh"
// The bits of omega that a kernel is given, and whether the host takes it for an oscillation (the
// test by which the table of time factors is made).
int main() {
    const double omegas[] = {0.0, -0.0, 0.25, -0.25, 4.9e-324};
    for (double w : omegas) {
        dugks::StepParams p;
        memset(&p, 0, sizeof p);
        p.rho0 = p.inv_c = 1.0;
        p.omega = w;
        dugks::finish_step_params(p);
        unsigned long long b;
        memcpy(&b, &p.omega, sizeof b);
        printf("%d %d\n", b != 0, w != 0.0);
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    d = tmp_path_factory.mktemp("params")
    src, exe = str(d / "params.cu"), str(d / "params")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.run([_build.nvcc()] + _build.ARCH + ["-O3", "-std=c++17", "--expt-relaxed-constexpr", "-I" + _build.INCLUDE,
                    "-I" + _build.CSRC, src, "-o", exe], check=True, capture_output=True)
    assert os.path.exists(exe)
    return subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split("\n")[:5]


def test_kernels_and_host_agree_on_a_zero_omega(lines):
    """A kernel tells a steady force by the bits of omega, the host by its value: -0.0 must not reach the
    kernel, which would read a table that the host did not make."""
    assert lines == ["0 0", "0 0", "1 1", "1 1", "1 1"]


def test_chained_kernels_read_states_by_coherent_loads():
    """A kernel launched as a programmatic dependent is resident while the step before it still writes
    the state: none may read the state, or the table of time factors, by the non-coherent path, which
    wants memory that is read-only for the life of the grid."""
    def code(name):
        with open(os.path.join(_build.CSRC, name)) as f:
            return re.sub(r"//[^\n]*", "", f.read())

    chained = [n for n in sorted(os.listdir(_build.CSRC)) if n.endswith(".cuh") and "chain_wait();" in code(n)]
    assert chained
    for name in chained:
        text = code(name)
        assert "Store<S>::ld(" not in text, name
        for line in text.split("\n"):
            for arg in re.findall(r"__ldg\(([^;]*)", line):  # what no step writes
                assert re.match(r"(p\.field|p\.metric|fr \+|items)", arg), (name, line)
    table = code("dugks_device.cuh")
    table = table[table.index("void time_factors("):table.index("struct FromTable")]
    assert "__ldg" not in table
