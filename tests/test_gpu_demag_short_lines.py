"""Demag passes that the shapes of test_gpu_demag_tiles.py do not reach, against the FP64 oracle: thin meshes that are too
wide for the fused y-z pass (register z kernels of the shortest lines), z lines of 128 values, and x lines of 128 values
in radix-16 stages (from 3243 lines a component on), there against the oracle's sampled nodes of a sparse source.
Bars as for every field test: FP64 1e-12, FP32 1e-5 relative L2 on the same rounded input.
"""
import numpy as np
import pytest

import nm_inputs as inp
from helpers import gpu_mesh, oracle_mesh, rel_l2, rounded

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


@pytest.mark.parametrize("precision, shape", [(0, (3, 65, 2)), (0, (2, 33, 5)), (0, (2, 33, 7)), (0, (2, 33, 8)),
                                              (1, (2, 400, 2)), (1, (2, 260, 3)), (1, (2, 260, 4)),
                                              (0, (2, 3, 33)), (1, (2, 3, 33)), (0, (1, 2, 64)), (1, (1, 2, 64))])
def test_demag(oracle_mod, nmgb, precision, shape):
    import torch
    p = inp.random_problem(np.random.default_rng(sum(shape)), shape, vacuum=False)
    m = rounded(p.m0, precision)
    ref = oracle_mesh(oracle_mod, p).h_eff(m, oracle_mod.DEMAG, 0.0)
    me = gpu_mesh(nmgb, p, precision)
    h = me.h_eff(torch.tensor(m, dtype=me.dtype, device="cuda"), nmgb.DEMAG, 0.0).double().cpu().numpy()
    me.close()
    assert rel_l2(h, ref) < TOL[precision]


def test_wide_x_lines(nmgb):
    import torch
    from oracle import sampled
    n, dx = (70, 60, 55), (3e-9, 3e-9, 3e-9)
    nodes = tuple(v + 1 for v in n)
    rng = np.random.default_rng(9)
    m = np.zeros(nodes + (3,))
    for nd in [(1, 1, 1), (2, 1, 1), (1, 2, 1), (1, 1, 2), (69, 58, 30), (35, 30, 54)]:
        m[nd] = inp.unit_vector(rng)
    m = rounded(m, 0)
    at = [(0, 0, 0), (1, 2, 1), (3, 1, 2), (68, 58, 31), (70, 60, 29), (35, 31, 55), (40, 20, 10), (70, 60, 55), (0, 60, 55)]
    at += [tuple(int(rng.integers(0, v)) for v in nodes) for _ in range(12)]
    me = nmgb.Mesh(n, dx, nmgb.F32)
    me.set_material(1e6, 1.5e-11)
    h = me.h_eff(torch.tensor(m, dtype=me.dtype, device="cuda"), nmgb.DEMAG, 0.0).double().cpu().numpy()
    me.close()
    ref = sampled.demag_at_nodes(n, dx, 1e6, m, at)
    got = np.array([h[a] for a in at])
    assert rel_l2(got, ref) < TOL[0]
    assert np.abs(got - ref).max() <= TOL[0] * np.abs(ref).max()
