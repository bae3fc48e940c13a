"""Dynamic shared memory beyond 48 KB (rbe_optin.h) is asked for by each context and kernel, contexts being on devices of
their own, and again after a failure; and no request of the library is made once for the process."""
import glob
import os
import re
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2110_14362_gb300", "csrc")


def test_each_context_asks(tmp_path):
    exe = str(tmp_path / "optin")
    subprocess.run(["g++", "-std=c++17", "-o", exe, os.path.join(HERE, "host", "optin_main.cpp")], check=True)
    launches = [(0, 0, 0), (0, 0, 0), (0, 14, 0), (1, 0, 0), (1, 0, 0), (2, 3, 700), (2, 3, 700), (2, 3, 0), (2, 3, 0), (3, 3, 0)]
    text = "\n".join(" ".join(map(str, x)) for x in launches)
    out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split("\n")[:-1]
    assert out == ["1 0", "0 0", "1 0", "1 0", "0 0", "1 700", "1 700", "1 0", "0 0", "1 0"]


def test_no_request_for_the_whole_process():
    """A static initialiser would ask on the first context's device only, and keep its failure."""
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        assert not re.search(r"static const cudaError_t", open(path).read()), path
