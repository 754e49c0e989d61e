"""The bounded waits of the tensor-pipe kernels, by themselves: a barrier that nobody completes ends a wait with an error."""
import ctypes
import os
import subprocess

import pytest

from paper_2201_12667_b200 import build

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    lib = str(tmp_path_factory.mktemp("waits") / "wait_probe.so")
    subprocess.run([build._nvcc(), "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-Xcompiler", "-fPIC", "-shared",
                    "-I", build.CSRC, os.path.join(HERE, "wait_probe.cu"), "-o", lib], check=True)
    return ctypes.CDLL(lib)


def test_a_wait_that_nothing_ends(probe):
    """It gives up within its limit (a second's cycles, and one try of the hardware's own length beyond), later waits at once."""
    out, cycles = (ctypes.c_int * 4)(), (ctypes.c_longlong * 2)()
    assert probe.run_waits(0, out, cycles) == 0
    assert list(out) == [0, 0, 1, 1]
    assert 2.0e9 < cycles[0] < 2.5e9, cycles[0]
    assert cycles[1] < 0.5e9, cycles[1]


def test_a_pair_gives_up_together(probe):
    """The block whose wait has run out tells the other block of the pair, whose waits then return at once; what is in flight
    is waited for by the clock too."""
    out, cycles = (ctypes.c_int * 4)(), (ctypes.c_longlong * 2)()
    assert probe.run_waits(1, out, cycles) == 0
    assert list(out) == [0, 1, 1, 0]
    assert cycles[0] < 0.5e9 and 2.0e7 <= cycles[1] < 5.0e8, list(cycles)


def test_a_warp_gets_one_answer(probe):
    """Lanes whose own waits would end differently once the block has given up: none goes on while others leave."""
    out, cycles = (ctypes.c_int * 4)(), (ctypes.c_longlong * 2)()
    assert probe.run_waits(2, out, cycles) == 0
    assert list(out) == [0, 1, 32, 1]
    assert cycles[1] < 0.5e9, list(cycles)


def test_a_warp_gives_up_together(probe):
    """Half of the lanes' waits run out, the others' do not: all lanes are told so, after the limit of one wait."""
    out, cycles = (ctypes.c_int * 4)(), (ctypes.c_longlong * 2)()
    assert probe.run_waits(3, out, cycles) == 0
    assert list(out)[:2] == [0, 32]
    assert 2.0e9 < cycles[0] < 2.5e9, list(cycles)
