"""Function attributes and occupancies are remembered per device: a kernel that
opted in to more shared memory on one device has to do so on the next."""
import ctypes
import os
import re
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2405_04237_gb300", "csrc")


def test_one_opt_in_for_each_device(tmp_path):
    so = str(tmp_path / "per_device.so")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I" + CSRC,
                           "-I" + cuda + "/include", os.path.join(HERE, "device_on_cpu", "per_device.cpp"), "-o", so])
    lib = ctypes.CDLL(so)
    order = (ctypes.c_int * 6)(0, 0, 1, 0, 1, 3)
    assert lib.opt_ins(order, 6) == 3


def test_no_opt_in_is_remembered_for_the_process():
    """Every attribute call is made on each launch or guarded by a PerDevice value."""
    for name in os.listdir(CSRC):
        text = open(os.path.join(CSRC, name)).read()
        assert not re.search(r"static bool \w+ = false", text), name
        if "cudaFuncSetAttribute" in text and name != "k_batched.cu":  # k_batched: on each launch
            assert "PerDevice<" in text, name
