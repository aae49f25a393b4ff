"""The native marshalling (csrc/call.cpp) gives up the interpreter lock around a call of the library.  A C++ exception
that leaves the call becomes a Python exception, raised with the lock held again."""
import subprocess
import sys

from paper_2601_12212_b200 import build

CHILD = """
import ctypes, sys, threading
import torch
from paper_2601_12212_b200 import binding
binding.load()
lib = ctypes.CDLL(sys.argv[1])
call = binding._call.bind("resps_tree_expand_begin", ctypes.cast(lib.begin, ctypes.c_void_p).value)
stop = False
def spin():
    while not stop:
        pass
other = threading.Thread(target=spin)  # takes the lock whenever it is given up
other.start()
for i in range(200):
    assert call(None, None, 7, 1) == 7
    try:
        call(None, None, -1, 1)
    except RuntimeError as e:
        assert str(e) == "out of something"
    else:
        raise SystemExit("no exception")
stop = True
other.join()
print("survived")
"""


def test_an_exception_comes_back_with_the_lock(tmp_path):
    build.build()
    src, lib = tmp_path / "thrower.cpp", tmp_path / "thrower.so"
    src.write_text('#include <stdexcept>\nextern "C" int begin(void*, const void*, int batch, int) {\n'
                   '    if (batch < 0) throw std::runtime_error("out of something");\n    return batch;\n}\n')
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", str(src), "-o", str(lib)], check=True)
    res = subprocess.run([sys.executable, "-c", CHILD, str(lib)], capture_output=True, text=True, timeout=300)
    assert res.returncode == 0 and "survived" in res.stdout, (res.returncode, res.stderr[-800:])
