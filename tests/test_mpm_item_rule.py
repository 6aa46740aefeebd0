"""The rule that sizes the full-order kernel's work items and CTAs (csrc/mpm_items.cuh, plain C++, compiled here):
what may not depend on the two or three sizes it was measured at."""
import ctypes as C
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2109_12390_gb300", "csrc")


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("items")
    (d / "r.cc").write_text('#include "mpm_items.cuh"\nextern "C" int rule(int dim, long long P, int n_sm) {\n'
                            "  const mpmrom::ItemRule r = mpmrom::item_rule(dim, P, n_sm);\n"
                            "  return r.narrow ? -r.cap : r.cap;\n}\n")
    so = d / "r.so"
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "r.cc"), "-o", str(so)], check=True)
    lib = C.CDLL(str(so))
    lib.rule.argtypes = [C.c_int, C.c_longlong, C.c_int]
    return lambda dim, P, n_sm: (abs(lib.rule(dim, P, n_sm)), lib.rule(dim, P, n_sm) < 0)


def _sizes():
    P = 1
    while P < 1 << 30:
        yield P
        P += max(1, P // 37)


@pytest.mark.parametrize("n_sm", [132, 148, 152])
def test_bounds(rule, n_sm):
    for dim in (2, 3):
        for P in _sizes():
            cap, narrow = rule(dim, P, n_sm)
            assert 128 <= cap <= 512 and cap % 32 == 0
            assert dim == 2 or not narrow


@pytest.mark.parametrize("n_sm", [132, 148, 152])
def test_narrow_ctas_only_past_one_wave_of_wide_ones(rule, n_sm):
    # 256-thread CTAs hold 768 particles per SM at once: below that, narrow ones only halve an SM's threads
    for P in _sizes():
        assert not rule(2, P, n_sm)[1] or P > 768 * n_sm
    assert rule(2, 2000 * n_sm, n_sm)[1]


@pytest.mark.parametrize("n_sm", [132, 148, 152])
def test_blocks_are_split_only_while_the_items_are_resident(rule, n_sm):
    # 3 items per SM: bodies of full blocks (256 particles in 2D, 512 in 3D) and nothing else
    for dim, full in ((2, 256), (3, 512)):
        for P in _sizes():
            cap, narrow = rule(dim, P, n_sm)
            items = -(-P // full) * -(-full // cap)
            assert cap == 512 or items <= 3 * n_sm
