"""The bounded wait of the specialised warps' kernels: one that nothing ever
completes reports BM_ETIMEDOUT and makes the block's other waits give up too,
instead of each of them polling to its own limit; the device stays usable."""
import ctypes
import os
import re
import subprocess

import pytest

from paper_2310_12441_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.gpu
def test_a_wait_that_nothing_completes(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    so = str(tmp_path / "wait_limit.so")
    subprocess.run([B._nvcc(), *B.ARCH, *B.FLAGS, "-I", B.CSRC, "-shared", os.path.join(HERE, "native", "wait_limit.cu"),
                    "-o", so], check=True)
    got = (ctypes.c_int * 4)()
    assert ctypes.CDLL(so).wait_limit(got) == 0
    header = open(os.path.join(B.INCLUDE, "bootmmpm.h")).read()
    timed_out = int(re.search(r"BM_ETIMEDOUT\s*=?\s*\(?(-?\d+)", header).group(1))
    assert list(got) == [1, 0, 0, timed_out]
    assert int(torch.arange(5, device="cuda").sum()) == 10
