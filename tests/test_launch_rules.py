"""The host-side rules that choose a launch's form (csrc/rc_rules.h), compiled
by themselves and called on the CPU."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1211_5595_gb300", "csrc")
SHIM = r"""
#include "rc_rules.h"
extern "C" {
int persistent_ctas(int chunks, int sms) { return rc::persistent_ctas(chunks, sms); }
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("rules")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC,
                    "-o", str(d / "shim.so"), str(d / "shim.cpp")], check=True)
    return C.CDLL(str(d / "shim.so"))


# a chunk gets an SM of its own before two share one
@pytest.mark.parametrize("chunks,ctas", [(1, 1), (3, 3), (64, 64), (151, 151), (152, 152), (153, 152), (456, 152),
                                         (1 << 27, 152)])
def test_a_small_image_spreads_over_the_sms(rules, chunks, ctas):
    assert rules.persistent_ctas(chunks, 152) == ctas
