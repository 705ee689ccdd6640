"""The tensor-core GEMM after a device reset, which frees the pinned word and
the kernel attributes that earlier calls left: in a process of its own, from two
threads, with a product that fits the default shared memory and one that does
not."""
import glob
import os
import subprocess
import sys

import pytest

from paper_2408_00559_gb300 import build as BLD

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
RUN = """
import ctypes as C
import sys
import threading
import numpy as np
from paper_2408_00559_gb300 import _lib as B
rt = C.CDLL(sys.argv[1])
lib = B.lib()


def product(M, N, K):
    # A and B all ones (BF16 0x3f80): C is K everywhere
    ptr = []
    for n in (M * K * 2, N * K * 2, M * N * 4):
        p = C.c_void_p()
        assert rt.cudaMalloc(C.byref(p), C.c_size_t(n)) == 0
        ptr.append(p)
    for p, n in ((ptr[0], M * K), (ptr[1], N * K)):
        h = np.full(n, 0x3f80, dtype=np.uint16)
        assert rt.cudaMemcpy(p, h.ctypes.data_as(C.c_void_p), C.c_size_t(2 * n), C.c_int(1)) == 0
    assert lib.amfrw_tc_gemm_bf16(ptr[0], K, ptr[1], K, ptr[2], N, M, N, K, None) == 0
    c = np.zeros((M, N), dtype=np.float32)
    assert rt.cudaMemcpy(c.ctypes.data_as(C.c_void_p), ptr[2], C.c_size_t(4 * M * N), C.c_int(2)) == 0
    assert np.all(c == K), c
    for p in ptr:
        rt.cudaFree(p)


def both():
    product(130, 64, 64)
    product(300, 256, 512)


assert rt.cudaSetDevice(0) == 0
for _ in range(3):
    both()
    t = threading.Thread(target=both)
    t.start()
    t.join()
    assert rt.cudaDeviceReset() == 0
both()
print("ok")
"""


def test_products_after_a_device_reset():
    BLD.build()
    paths = glob.glob("/usr/local/cuda/lib64/libcudart.so") + glob.glob("/usr/local/cuda/targets/*/lib/libcudart.so")
    if not paths:
        pytest.skip("no shared CUDA runtime to reset the device with")
    r = subprocess.run([sys.executable, "-c", RUN, paths[0]], cwd=ROOT, capture_output=True, text=True, timeout=120,
                       env=dict(os.environ, PYTHONPATH=ROOT))
    assert r.returncode == 0 and "ok" in r.stdout, (r.returncode, r.stdout, r.stderr)
