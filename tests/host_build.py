"""Host builds of the library's index arithmetic: a C++ file of tests/host/ compiled with g++
against the headers of csrc/ and loaded through ctypes, for tests without a GPU."""
import ctypes
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1301_4019_gb300", "csrc")


def load(name, out_dir):
    lib = os.path.join(str(out_dir), name + ".so")
    subprocess.run(["g++", "-std=c++20", "-O2", "-ffp-contract=off", "-fPIC", "-shared", "-pthread",
                    "-I", CSRC, "-I", os.path.join(HERE, "host"), "-o", lib,
                    os.path.join(HERE, "host", name + ".cpp")], check=True)
    return ctypes.CDLL(lib)
