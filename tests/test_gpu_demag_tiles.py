"""Demag convolution at the edges of its z and y-z tiles, against the FP64 oracle: every z transform length with the
smallest and the largest number of layers it takes, one and several rows (octant rows without and with a mirror,
more rows than a block), one column to several blocks of columns, and single layers with every y length up to the
longest.  Bars as for every field test: FP64 1e-12, FP32 1e-5 relative L2 on the same rounded input.
"""
import numpy as np
import pytest

import nm_inputs as inp
from helpers import gpu_mesh, oracle_mesh, rel_l2, rounded

pytestmark = pytest.mark.gpu

TOL = {0: 1e-5, 1: 1e-12}
LAYERED = [(3, 5, 2), (1, 7, 2), (17, 2, 3), (9, 1, 4), (4, 33, 4), (2, 40, 3), (3, 9, 5), (2, 11, 8), (33, 2, 8), (3, 2, 9),
           (2, 6, 16), (2, 3, 17), (3, 3, 31), (2, 4, 32), (1, 1, 7)]
SINGLE = [(1, 1, 1), (40, 1, 1), (3, 2, 1), (5, 4, 1), (2, 8, 1), (130, 3, 1), (4, 16, 1), (3, 17, 1), (2, 60, 1), (2, 100, 1),
          (300, 2, 1), (2, 200, 1), (2, 400, 1), (1, 600, 1), (1, 1024, 1)]


@pytest.fixture(scope="module")
def nmgb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2411_11725_gb300 as nmgb
    nmgb.load()
    return nmgb


@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("shape", LAYERED + SINGLE)
def test_demag(oracle_mod, nmgb, precision, shape):
    import torch
    p = inp.random_problem(np.random.default_rng(sum(shape)), shape, vacuum=False)
    m = rounded(p.m0, precision)
    ref = oracle_mesh(oracle_mod, p).h_eff(m, oracle_mod.DEMAG, 0.0)
    me = gpu_mesh(nmgb, p, precision)
    h = me.h_eff(torch.tensor(m, dtype=me.dtype, device="cuda"), nmgb.DEMAG, 0.0).double().cpu().numpy()
    me.close()
    assert rel_l2(h, ref) < TOL[precision]
