"""Node kernel for cell maps (layer sums carried along z, tiles of 32 x 4 nodes) against the FP64 oracle at the edges of
its tiles and of its walk, with and without vacuum cells, and with one map beside uniform values.  Bars as for every
field test: FP64 1e-12, FP32 1e-5 relative L2 on the same rounded input; one step of each integrator FP64 1e-12, FP32
1e-6 on unit vectors (the field's bar times a displacement of a tenth).
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


def _field(oracle_mod, nmgb, p, precision, terms):
    import torch
    m = rounded(p.m0, precision)
    ref = oracle_mesh(oracle_mod, p).h_eff(m, terms, 1e-10)
    me = gpu_mesh(nmgb, p, precision)
    h = me.h_eff(torch.tensor(m, dtype=me.dtype, device="cuda"), terms, 1e-10).double().cpu().numpy()
    me.close()
    return rel_l2(h, ref)


@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("vacuum", [False, True])
def test_field(oracle_mod, nmgb, precision, shape, vacuum):
    p = inp.random_problem(np.random.default_rng(sum(shape)), shape, vacuum=vacuum)
    terms = oracle_mod.ALL if np.prod(shape) <= 400 else oracle_mod.ALL & ~oracle_mod.DEMAG
    assert _field(oracle_mod, nmgb, p, precision, terms) < TOL[precision]


@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("one_map", ["Ms", "A", "Ku"])
@pytest.mark.parametrize("term", ["EXCH", "ANIS"])
def test_one_map(oracle_mod, nmgb, precision, one_map, term):
    p = inp.random_problem(np.random.default_rng(3), (35, 6, 3), vacuum=False)
    for name in {"Ms", "A", "Ku"} - {one_map}:
        setattr(p, name, float(np.asarray(getattr(p, name)).flat[0]))
    assert _field(oracle_mod, nmgb, p, precision, getattr(oracle_mod, term)) < TOL[precision]


@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("method", ["rk4", "dp5"])
def test_step(oracle_mod, nmgb, precision, method):
    p = inp.random_problem(np.random.default_rng(8), (33, 4, 2), vacuum=True)
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
