"""The rule by which register keeps or drops the status word of an evaluation that
it throws away (a first trial along a direction that does not descend): only a
non-finite value is dropped with its point.  The rule is a host function of the
library's internal header, compiled here by itself."""
import ctypes
import os
import shutil
import subprocess

import pytest

import paper_1907_04839_gb300 as gsh

CSRC = os.path.join(os.path.dirname(os.path.abspath(gsh.__file__)), "csrc")
TIMEOUT, NONFINITE, BAD_LAUNCH = 1, 2, 4


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("rule")
    (d / "rule.cpp").write_text('#include "gs_internal.h"\n'
                                'extern "C" int rule(unsigned s) { return gs::goes_with_its_point(s); }\n'
                                'extern "C" unsigned bits() { return gs::kErrTimeout | gs::kErrNonFinite << 4 | gs::kErrBadLaunch << 8; }\n')
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    so = str(d / "rule.so")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-I", cuda, str(d / "rule.cpp"), "-o", so],
                   check=True)
    lib = ctypes.CDLL(so)
    assert lib.bits() == TIMEOUT | NONFINITE << 4 | BAD_LAUNCH << 8
    return lib.rule


@pytest.mark.parametrize("status", range(8))
def test_only_a_nonfinite_value_is_dropped(rule, status):
    assert bool(rule(status)) == (status in (0, NONFINITE))
