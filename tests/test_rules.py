"""Index and size rules of csrc/rules.h over ranges no device buffer of a test reaches, compiled
with the host compiler (no GPU)."""
import ctypes
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1709_05418_gb300", "csrc")
SHIM = r"""
#include "rules.h"
using namespace rpnn;
extern "C" {
int64_t t_query_at(int64_t i) { return query_at(i); }
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "rules.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-I" + CSRC,
                    str(d / "shim.cpp"), "-o", so], check=True)
    L = ctypes.CDLL(so)
    L.t_query_at.argtypes, L.t_query_at.restype = [ctypes.c_int64], ctypes.c_int64
    return L


def test_shading_point_offsets_need_64_bits(rules):
    """Up to 2^31 - 1 shading points: every offset is exact, and no kernel that reads the lists
    works one out by itself."""
    for i in (0, 1, 715827882, 715827883, 2 ** 31 - 2):
        assert rules.t_query_at(i) == 3 * i
    src = open(os.path.join(CSRC, "render.cu")).read()
    assert not re.findall(r"\bq[xd]\[3 \*", src)
    # a point's index runs to 2^31 - 1 and its grid stride beyond
    for kernel in ("k_nee_env", "k_scatter"):
        body = src[src.index(kernel + "("):]
        body = body[:body.index("\n}\n")]
        assert not re.search(r"\bint i = blockIdx", body), kernel
