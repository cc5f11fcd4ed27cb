"""The message of a CG wait that ran out names the wait (csrc/sso_internal.cuh),
and the kernels raise the flag of their own wait."""
import ctypes
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2407_20026_gb300", "csrc")
CUDA = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")


def test_messages_name_the_wait(tmp_path):
    src = tmp_path / "m.cpp"
    src.write_text('#include "sso_internal.cuh"\n'
                   'extern "C" const char* text(int f) { return sso::wait_failure(f); }\n'
                   'extern "C" int team() { return sso::WAIT_TEAM; }\n'
                   'extern "C" int copy() { return sso::WAIT_COPY; }\n')
    lib = tmp_path / "m.so"
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-I", CUDA, str(src),
                    "-o", str(lib)], check=True)
    L = ctypes.CDLL(str(lib))
    L.text.restype = ctypes.c_char_p
    assert b"team" in L.text(L.team()) and b"copy" not in L.text(L.team())
    assert b"bulk copy" in L.text(L.copy())


@pytest.mark.parametrize("source,flag", [("cluster.cu", "WAIT_TEAM"), ("pcg.cu", "WAIT_COPY")])
def test_kernels_raise_their_own_flag(source, flag):
    with open(os.path.join(CSRC, source)) as f:
        raised = re.findall(r"atomicExch\((?:sh\.)?flags \+ 1, (\w+)\)", f.read())
    assert raised and set(raised) == {flag}
