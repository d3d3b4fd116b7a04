"""Uniform materials in the transpose product (3D and 2D basis) and DMI on a uniform material: the node kernels of
uniform materials against those of cell maps, which a constant map of A selects and the oracle covers.  Bars: FP64
1e-12, FP32 1e-5 relative L2 (the field's), the Ms gradient included.
"""
import numpy as np
import pytest

import nm_inputs as inp
from helpers import rel_l2

pytestmark = pytest.mark.gpu

TOL = {0: 1e-5, 1: 1e-12}


@pytest.fixture(scope="module")
def nmgb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2411_11725_gb300 as nmgb
    nmgb.load()
    return nmgb


def _pair(nmgb, shape, basis, precision, D=None):
    """(a uniform mesh, the same with a constant map of A)"""
    p = inp.random_problem(np.random.default_rng(sum(shape)), shape, heterogeneous=False)
    out = []
    for A in (p.A, np.full(shape, p.A)):
        me = nmgb.Mesh(shape, p.dx, precision, basis=basis)
        me.set_material(p.Ms, A, p.Ku, p.axis, p.alpha, p.gamma)
        me.set_zeeman(p.h_uniform, p.h_freq, p.h_phase, p.h_cell, p.cell_freq, p.cell_phase)
        if D is not None:
            me.set_dmi(D)
        out.append(me)
    return out


def _nodal(me, seed):
    import torch
    return torch.tensor(inp.unit_vectors(np.random.default_rng(seed), me.nodes), dtype=me.dtype, device="cuda")


@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("basis, shape, dmi", [(3, (1, 1, 1), False), (3, (33, 5, 4), False), (3, (3, 9, 40), False),
                                               (3, (1, 1, 1), True), (3, (33, 5, 4), True), (3, (3, 9, 40), True),
                                               (2, (1, 1, 1), False), (2, (33, 9, 3), False)])
def test_transpose_product(nmgb, precision, basis, shape, dmi):
    out = []
    for me in _pair(nmgb, shape, basis, precision, 2.5e-3 if dmi else None):
        gm, gMs = me.h_eff_vjp(_nodal(me, 1), _nodal(me, 2), nmgb.ALL | (nmgb.DMI if dmi else 0), 1e-10)
        out.append((gm.double().cpu().numpy(), gMs.double().cpu().numpy()))
        me.close()
    assert rel_l2(out[0][0], out[1][0]) < TOL[precision]
    assert rel_l2(out[0][1], out[1][1]) < TOL[precision]


@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("shape", [(1, 1, 1), (33, 5, 4), (5, 2, 33)])
@pytest.mark.parametrize("D_map", [False, True])
def test_dmi(nmgb, precision, shape, D_map):
    D = np.random.default_rng(3).uniform(-3e-3, 3e-3, shape) if D_map else 2.5e-3
    out = []
    for me in _pair(nmgb, shape, 3, precision, D):
        h = me.h_eff(_nodal(me, 1), nmgb.ALL | nmgb.DMI, 1e-10).double().cpu().numpy()
        me.set_terms(nmgb.ALL | nmgb.DMI)
        me.set_state(_nodal(me, 1).double(), 0.0, 5e-14)
        me.run_steps(1, nmgb.RK4)
        me.run_steps(1, nmgb.DP54)
        out.append((h, me.get_state()[0]))
        me.close()
    assert rel_l2(out[0][0], out[1][0]) < TOL[precision]
    # two steps on unit vectors: the field's bar times a displacement of a tenth
    assert rel_l2(out[0][1], out[1][1]) < {0: 1e-6, 1: 1e-12}[precision]
