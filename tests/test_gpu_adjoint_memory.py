"""Device memory of the gradient calls.  The fields that the reverse sweep keeps for its transpose products are
allocated for a sweep alone, the demag part only with the demag term, and a call that lacks the room for them forms the
fields again and returns the same gradients (as accurate as the two ways of forming one field agree: FP64 1e-12).
The high-water mark of the device's default memory pool, where the workspaces come from, shows what a call takes.
"""
import ctypes

import numpy as np
import pytest

import nm_inputs as inp
from helpers import rel_l2

pytestmark = pytest.mark.gpu

_RESERVED_MEM_HIGH, _USED_MEM_HIGH = 6, 8  # cudaMemPoolAttrReservedMemHigh, cudaMemPoolAttrUsedMemHigh


@pytest.fixture(scope="module")
def nmgb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2411_11725_gb300 as nmgb
    nmgb.load()
    return nmgb


class _Device:
    """the CUDA runtime that the library is linked against"""

    def __init__(self):
        import torch
        for name in ("libcudart.so.13", "libcudart.so"):
            try:
                self.rt = ctypes.CDLL(name)
                break
            except OSError:
                continue
        self.rt.cudaMalloc.argtypes = [ctypes.POINTER(ctypes.c_void_p), ctypes.c_size_t]
        self.rt.cudaFree.argtypes = [ctypes.c_void_p]
        self.rt.cudaMemPoolTrimTo.argtypes = [ctypes.c_void_p, ctypes.c_size_t]
        self.pool = ctypes.c_void_p()
        assert self.rt.cudaDeviceGetDefaultMemPool(ctypes.byref(self.pool), torch.cuda.current_device()) == 0

    def trim(self):
        assert self.rt.cudaDeviceSynchronize() == 0
        assert self.rt.cudaMemPoolTrimTo(self.pool, 0) == 0

    def peak(self, call, attribute=_USED_MEM_HIGH):
        """(result, bytes of the pool at its highest) of a call"""
        self.trim()
        zero, v = ctypes.c_uint64(0), ctypes.c_uint64()
        assert self.rt.cudaMemPoolSetAttribute(self.pool, attribute, ctypes.byref(zero)) == 0
        out = call()
        assert self.rt.cudaMemPoolGetAttribute(self.pool, attribute, ctypes.byref(v)) == 0
        return out, v.value

    def leave_free(self, nbytes):
        """allocate all but about nbytes of the device; returns the blocks to free"""
        self.trim()
        free, total = ctypes.c_size_t(), ctypes.c_size_t()
        blocks = []
        for _ in range(2):
            assert self.rt.cudaMemGetInfo(ctypes.byref(free), ctypes.byref(total)) == 0
            if free.value > nbytes:
                p = ctypes.c_void_p()
                assert self.rt.cudaMalloc(ctypes.byref(p), free.value - nbytes) == 0
                blocks.append(p)
        return blocks

    def free(self, blocks):
        for p in blocks:
            assert self.rt.cudaFree(p) == 0


N = (400, 300, 6)
NS, NC = int(np.prod([v + 1 for v in N])), int(np.prod(N))


def _call(nmgb, kind, terms, **kw):
    """(call, bytes of the kept fields) of a gradient over two steps"""
    stages = 7 if kind == "DP54" else 4
    rng = np.random.default_rng(6)
    nodes = tuple(v + 1 for v in N)
    m0, W, tgt = inp.unit_vectors(rng, nodes), rng.uniform(0.5, 1.5, nodes + (3,)), inp.unit_vectors(rng, nodes)
    me = nmgb.Mesh(N, (3e-9,) * 3, nmgb.F64)
    me.set_material(1e6, 1.5e-11, 5e5)
    me.set_terms(terms)

    def call():
        me.set_state(m0, 0.0, 1e-14)
        if kind == "continuous":
            return me.adjoint_continuous(2e-14, 2, W, tgt)
        return me.adjoint_run(2e-14, W, tgt, method=getattr(nmgb, kind), dt0=1e-14, rtol=1e3, atol=1e3,
                              checkpoint_every=1, **kw)

    return me, call, stages * 24 * NS, stages * 24 * NC


@pytest.mark.parametrize("kind", ["RK4", "DP54"])
def test_loss_alone_keeps_no_fields(nmgb, kind):
    """The loss alone needs the stage vectors of the gradient's call, less than the fields on top of them."""
    dev = _Device()
    me, call, nodal, cells = _call(nmgb, kind, 15, loss_only=True)
    call()
    _, loss_only = dev.peak(call)
    me.close()
    me, call, nodal, cells = _call(nmgb, kind, 15)
    call()
    _, gradient = dev.peak(call)
    me.close()
    assert loss_only <= gradient - nodal - cells


@pytest.mark.parametrize("kind", ["RK4", "continuous"])
def test_no_cell_fields_without_demag(nmgb, kind):
    dev, peak = _Device(), {}
    for terms in (15, 7):
        me, call, nodal, cells = _call(nmgb, kind, terms)
        call()
        _, peak[terms] = dev.peak(call)
        me.close()
    assert peak[7] <= peak[15] - cells


@pytest.mark.parametrize("kind", ["RK4", "DP54", "continuous"])
def test_without_room_for_the_fields(nmgb, kind):
    dev = _Device()
    me, call, nodal, cells = _call(nmgb, kind, 15)
    want = call()
    _, peak = dev.peak(call, _RESERVED_MEM_HIGH)
    blocks = dev.leave_free(peak - (nodal + cells) // 2)
    try:
        got = call()
    finally:
        dev.free(blocks)
    me.close()
    for a, b in zip(want, got):
        assert rel_l2(a, b) < 1e-12
