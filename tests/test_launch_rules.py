"""The rules that choose launch shapes and forms from sizes (csrc/launch_rules.h),
compiled for the host and gone through without a GPU."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1307_6720_gb300", "csrc")

SOURCE = """
#include "launch_rules.h"
extern "C" {
int plane_results(int ko, int planes, int least, int grouped) { return mhs::plane_results(ko, planes, least, grouped != 0); }
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    src, lib = d / "rules.cpp", d / "rules.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)],
                   check=True)
    return ctypes.CDLL(str(lib))


@pytest.mark.parametrize("least", [1, 4])
@pytest.mark.parametrize("grouped", [0, 1])
def test_plane_blocks_have_no_room_for_twice_their_results(rules, least, grouped):
    """No block of the plane transforms is shaped for twice the results that a
    line has (it would form them all), and a level that could give every SM a
    block does."""
    for ko in range(1, 65):
        for planes in (1, 2, 3, 7, 15, 31, 63, 76, 127, 152, 153, 255, 511, 1023, 2047):
            sp = rules.plane_results(ko, planes, least, grouped)
            assert least <= sp <= 16 and sp & (sp - 1) == 0
            assert sp == least or sp < 2 * ko, (ko, planes)
            if not grouped and sp > least:
                assert -(-ko // sp) * planes >= 152 or sp // 2 < least, (ko, planes)
