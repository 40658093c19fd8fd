"""Grid sizes follow the device, not one chip: at most one CTA an SM in the
dendrogram's middle rounds, for SM counts below and above this one's."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2311_10337_gb300", "csrc")


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("grids")
    src, lib = str(d / "grids.cpp"), str(d / "grids.so")
    with open(src, "w") as f:
        f.write('#include "grids.h"\n'
                'extern "C" int mid_ctas(int64_t live, int sms, int room) { return dgec::mid_ctas(live, sms, room); }\n')
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", lib, src], check=True)
    L = ctypes.CDLL(lib)
    L.mid_ctas.argtypes = [ctypes.c_int64, ctypes.c_int, ctypes.c_int]
    return L


@pytest.mark.parametrize("sms", [1, 76, 100, 132, 152, 200, 1000])
def test_middle_rounds_take_at_most_one_cta_an_sm(rules, sms):
    for live in (1, 511, 512, 513, 4097, 512 * sms, 512 * sms + 1, 1 << 19, 1 << 30):
        g = rules.mid_ctas(live, sms, 1024)
        assert g == min(sms, (live + 511) // 512)
    assert rules.mid_ctas(1 << 30, 5000, 1024) == 1024
