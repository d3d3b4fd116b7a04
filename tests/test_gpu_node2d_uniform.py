"""2D-basis node kernel of a uniform material against the FP64 oracle at the edges of its 32 x 4 blocks, and its steps
(every number of earlier slopes a stage combines) against the general kernel, which a constant map of A selects.
Bars: fields FP64 1e-12, FP32 1e-5 relative L2 on the same rounded input; one step FP64 1e-12, FP32 1e-6 on unit
vectors (the field's bar times a displacement of a tenth).
"""
import numpy as np
import pytest

import nm_inputs as inp
from helpers import rel_l2, rounded
from test_gpu_basis2d import _gpu2, _h_gpu, _m2, _oracle2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nmgb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2411_11725_gb300 as nmgb
    nmgb.load()
    return nmgb


@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("shape", [(1, 1, 1), (30, 3, 1), (31, 4, 2), (32, 2, 3), (63, 7, 1), (64, 8, 1), (2, 33, 4)])
@pytest.mark.parametrize("cell_field", [False, True])
def test_field(oracle_mod, nmgb, precision, shape, cell_field):
    rng = np.random.default_rng(sum(shape))
    p = inp.random_problem(rng, shape, heterogeneous=False)
    if not cell_field:
        p.h_cell = None
    m = rounded(_m2(rng, p), precision)
    ref = _oracle2(oracle_mod, p).h_eff(m, oracle_mod.ALL, 2.3e-10)
    me = _gpu2(nmgb, p, precision)
    h = _h_gpu(nmgb, me, m, nmgb.ALL, 2.3e-10)
    me.close()
    assert rel_l2(h, ref) < {0: 1e-5, 1: 1e-12}[precision]


@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("method", ["rk4", "dp5"])
def test_step(nmgb, precision, method):
    rng = np.random.default_rng(11)
    p = inp.random_problem(rng, (37, 6, 2), heterogeneous=False)
    m0, out = _m2(rng, p), []
    for A in (p.A, np.full(p.n, p.A)):
        p.A = A
        me = _gpu2(nmgb, p, precision)
        me.set_state(m0, 0.0, 5e-14)
        me.llg_step(nmgb.DP54 if method == "dp5" else nmgb.RK4, 0.0, 5e-14)
        out.append(me.get_state()[0])
        me.close()
    assert rel_l2(out[0], out[1]) < {0: 1e-6, 1: 1e-12}[precision]
