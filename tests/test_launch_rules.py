"""Launch rules that are plain host code (csrc/hr_internal.h), compiled for the host."""
import ctypes
import os
import subprocess

import pytest

from paper_2412_03489_gb300 import build as hb


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    src, out = d / "rules.cpp", d / "rules.so"
    src.write_text('#include <cmath>\n#include "hr_internal.h"\n'
                   'extern "C" int resident(int v, int M, int sms) { return hr::ptbox_resident(v, M, sms); }\n')
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I" + cuda, "-I" + hb.CSRC, "-I" + hb.INCLUDE,
                    str(src), "-o", str(out)], check=True, capture_output=True, text=True)
    return ctypes.CDLL(str(out))


@pytest.mark.parametrize("sms", [1, 152])
def test_path_tracer_variants_only_cap_the_launch_size_rule(rules, sms):
    """A variant tuned on a full launch leaves launches below its cap as they are."""
    sizes = {2 * k * sms + e for k in range(1, 8) for e in (-2, 0, 2)} | {3 * sms + e for e in (-1, 0, 1)} | {2}
    for M in sorted(m for m in sizes if m > 0):
        free = rules.resident(0, M, sms)
        assert free == min(4, max(2, -(-M // sms)))
        for variant, cap in ((1, 3), (2, 2)):
            assert rules.resident(variant, M, sms) == min(free, cap)
