"""Node kernel of a uniform material (separable stencil, tiles of 32 x 4 nodes walked along z) against the FP64
oracle, at the edges of its tiles and of its walk: one to three tiles along x, ragged rows, one cell layer, long
walks split into chunks.  Bars as for every field test: FP64 1e-12, FP32 1e-5 relative L2 on the same rounded
input; one step of each integrator (every number of earlier slopes a stage combines) FP64 1e-12, FP32 1e-6 on
unit vectors (the field's bar times a displacement of a tenth).
"""
import numpy as np
import pytest

import nm_inputs as inp
from helpers import gpu_mesh, oracle_mesh, rel_l2, rounded

pytestmark = pytest.mark.gpu

TOL = {0: 1e-5, 1: 1e-12}
SHAPES = [(1, 1, 1), (30, 3, 1), (31, 4, 2), (32, 2, 3), (63, 5, 1), (64, 3, 2), (3, 33, 4), (2, 3, 64), (1, 9, 31)]


@pytest.fixture(scope="module")
def nmgb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2411_11725_gb300 as nmgb
    nmgb.load()
    return nmgb


@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("cell_field", [False, True])
def test_field(oracle_mod, nmgb, precision, shape, cell_field):
    import torch
    p = inp.random_problem(np.random.default_rng(sum(shape)), shape, heterogeneous=False)
    if not cell_field:
        p.h_cell = None
    terms = oracle_mod.ALL if np.prod(shape) <= 400 else oracle_mod.ALL & ~oracle_mod.DEMAG
    m = rounded(p.m0, precision)
    ref = oracle_mesh(oracle_mod, p).h_eff(m, terms, 1e-10)
    me = gpu_mesh(nmgb, p, precision)
    h = me.h_eff(torch.tensor(m, dtype=me.dtype, device="cuda"), terms, 1e-10).double().cpu().numpy()
    me.close()
    assert rel_l2(h, ref) < TOL[precision]


@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("method", ["rk4", "dp5"])
def test_step(oracle_mod, nmgb, precision, method):
    p = inp.random_problem(np.random.default_rng(7), (33, 4, 2), heterogeneous=False)
    ref_mesh, me = oracle_mesh(oracle_mod, p), gpu_mesh(nmgb, p, precision)
    me.set_state(p.m0, 0.0, 5e-14)
    if method == "dp5":
        st = ref_mesh.dp5_stepper(p.m0, 0.0, 5e-14, oracle_mod.ALL)
        assert st.step()
        ref = st.m
        assert me.llg_step(nmgb.DP54, 0.0, 5e-14)[0]
    else:
        ref = ref_mesh.rk4_step(p.m0, 0.0, 5e-14, oracle_mod.ALL, True)
        me.llg_step(nmgb.RK4, 0.0, 5e-14)
    m = me.get_state()[0]
    me.close()
    assert rel_l2(m, ref) < {0: 1e-6, 1: 1e-12}[precision]
