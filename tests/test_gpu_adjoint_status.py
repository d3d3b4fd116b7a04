"""A status word set on the device while a gradient call runs (a bounded wait of a demag pass that runs out) fails the
call.  Nothing times out here: the word is written from the host, over and over on a stream of its own, while
nm_adjoint_continuous works.
"""
import ctypes
import subprocess
import threading

import numpy as np
import pytest

import nm_inputs as inp
from helpers import gpu_mesh

pytestmark = pytest.mark.gpu

SOURCE = """
#include "mesh.cuh"
extern "C" void *status_word(nm_mesh M) { return &M->ctl->status; }
"""


@pytest.fixture(scope="module")
def nmgb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2411_11725_gb300 as nmgb
    nmgb.load()
    return nmgb


@pytest.fixture(scope="module")
def status_word(nmgb, tmp_path_factory):
    from paper_2411_11725_gb300 import build
    d = tmp_path_factory.mktemp("status")
    src, lib = str(d / "status_word.cu"), str(d / "status_word.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([build.nvcc()] + build.ARCH + build.NVCC_FLAGS + ["-I" + build.CSRC, "-shared", "-o", lib, src],
                   check=True)
    fn = ctypes.CDLL(lib).status_word
    fn.restype, fn.argtypes = ctypes.c_void_p, [ctypes.c_void_p]
    return fn


def test_status_during_the_sweep(nmgb, status_word):
    import torch
    p = inp.random_problem(np.random.default_rng(7), (12, 10, 3), vacuum=False)
    me = gpu_mesh(nmgb, p, 1)
    W = np.ones(p.nodes + (3,))
    me.set_state(p.m0, 0.0, 1e-14)
    loss = me.adjoint_continuous(4e-13, 40, W)[0]
    try:  # the CUDA runtime that the library is linked against
        rt = ctypes.CDLL("libcudart.so.13")
    except OSError:
        rt = ctypes.CDLL("libcudart.so")
    rt.cudaMemcpyAsync.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int, ctypes.c_void_p]
    word, value, stop = status_word(me._h), ctypes.c_int(nmgb.ERR_TIMEOUT), threading.Event()
    stream = torch.cuda.Stream()

    def write():
        while not stop.is_set():
            assert rt.cudaMemcpyAsync(word, ctypes.addressof(value), 4, 1, stream.cuda_stream) == 0
            stream.synchronize()

    me.set_state(p.m0, 0.0, 1e-14)
    th = threading.Thread(target=write)
    th.start()
    try:
        with pytest.raises(nmgb.NMError) as e:
            me.adjoint_continuous(4e-13, 40, W)
    finally:
        stop.set()
        th.join()
    assert e.value.code == nmgb.ERR_TIMEOUT
    # the word of one call is not the next one's
    me.set_state(p.m0, 0.0, 1e-14)
    assert me.adjoint_continuous(4e-13, 40, W)[0] == loss
    me.close()
