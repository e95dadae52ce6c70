"""The integer arithmetic of the FP64 heat update (csrc/exact64.cuh) on the CPU:
the same functions as in the kernels, compiled for the host, against the FP64
operations, bit for bit, over every diffusion number they take."""
import os
import subprocess

import pytest

from paper_1602_07558_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
RS = [0.2499999999, 0.2, 0.1875, 0.125, 0.1, 0.0625, 0.05, 0.01, 2.0 ** -11 * 1.3, 2.0 ** -11]


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("fixed") / "fixed_heat")
    subprocess.run([build._nvcc()] + build.ARCH + ["-O2", "-std=c++17", "-Xcompiler",
                   "-ffp-contract=off", f"-I{build.CSRC}", os.path.join(HERE, "fixed_heat.cu"),
                   "-o", exe], check=True, capture_output=True)

    def run(r, kind, blocks):
        out = subprocess.run([exe, repr(r), kind, str(blocks), "7"], check=True,
                             capture_output=True, text=True).stdout
        return [int(v) for v in out.split()]
    return run


@pytest.mark.parametrize("kind", ["one_binade", "negative", "two_binades", "binades", "smooth", "ties",
                                  "few_bits", "powers", "smallest", "huge"])
@pytest.mark.parametrize("r", RS)
def test_integer_update_has_the_bits_of_the_fp64_one(program, r, kind):
    taken, _, differ = program(r, kind, 400)
    assert taken == 400 and differ == 0


@pytest.mark.parametrize("kind", ["one_binade", "negative", "smooth", "ties", "few_bits"])
def test_a_block_of_one_binade_never_fails(program, kind):
    """Neighbours in one binade differ by less than its lowest value, however rough
    the field: no block has to be repeated by the FP64 operations."""
    assert program(0.2, kind, 2000)[1] == 0


@pytest.mark.parametrize("r", [0.25, 0.2500001, 2.0 ** -11 * 0.9999999, 0.0, -0.1, float("inf"),
                               float("nan")])
def test_other_diffusion_numbers_are_left_to_the_fp64_operations(program, r):
    assert program(r, "smooth", 5)[0] == 0
