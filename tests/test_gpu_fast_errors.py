"""A C++ exception that leaves a decode entry point arrives in Python as an exception, with the interpreter's lock held again."""
import ctypes
import subprocess
import threading

import pytest
import torch

from paper_2602_01744_b200 import api

pytestmark = pytest.mark.gpu

SRC = r"""
#include <stdexcept>
#include <stdint.h>
extern "C" int throws(void *, int32_t, const void *, const void *, const void *, const float *, const float *, const float *, const float *, float *, void *, void *) {
    throw std::runtime_error("no room for a record");
}
extern "C" int odd(void *, int32_t, const void *, const void *, const void *, const float *, const float *, const float *, const float *, float *, void *, void *) { throw 7; }
"""


@pytest.mark.parametrize("entry,text", [("throws", "no room for a record"), ("odd", "unknown C\\+\\+ exception")])
def test_an_exception_behind_the_boundary(tmp_path, entry, text):
    (tmp_path / "throws.cpp").write_text(SRC)
    subprocess.run(["g++", "-shared", "-fPIC", "-o", str(tmp_path / "throws.so"), str(tmp_path / "throws.cpp")], check=True)
    L = ctypes.CDLL(str(tmp_path / "throws.so"))
    api.lib()
    B, H, d = 2, 4, 32
    x = lambda *s: torch.zeros(*s, device="cuda")
    args = (x(B, H, d), x(B, H, d), x(B, H, d), x(H), x(B, H), x(B, H), x(B, H, d, d), None, None)
    address = ctypes.cast(getattr(L, entry), ctypes.c_void_p).value
    seen = []

    def call():
        for _ in range(50):
            with pytest.raises(RuntimeError, match=text):
                api._fast[0](address, 1, H, d, 0, 0, *args)
        seen.append(1)

    threads = [threading.Thread(target=call) for _ in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert len(seen) == 3
