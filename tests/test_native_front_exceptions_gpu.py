"""A C++ exception out of a library call (an allocation that fails, say) reaches
the caller of the native front as a Python exception, with the GIL held."""
import ctypes
import subprocess
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_cs_0603115_gb300 as ff
    from paper_cs_0603115_gb300 import _lib

SOURCE = """
#include <cstddef>
#include <stdexcept>
extern "C" int refuse(const void*, void*, size_t, void*) { throw std::runtime_error("no memory for the plan"); }
"""


def test_exception_of_a_call_is_raised(tmp_path):
    src, lib = tmp_path / "refuse.cpp", tmp_path / "refuse.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-shared", "-fPIC", "-o", str(lib), str(src)], check=True)
    address = ctypes.cast(ctypes.CDLL(str(lib)).refuse, ctypes.c_void_p).value
    ff.load()
    x = torch.tensor([[1.0, 0.0]] * 5, device="cuda")
    raised = []

    def calls():
        for _ in range(50):
            try:
                _lib.native.unary(address, x, None)
            except RuntimeError as e:
                raised.append(str(e))

    threads = [threading.Thread(target=calls) for _ in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert len(raised) == 200 and all("no memory for the plan" in m for m in raised)
    assert torch.equal(ff.add(x, x), x + x)
