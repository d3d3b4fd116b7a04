"""FP32 exchange field of uniform materials on smooth states (a rotation of theta per cell), against the FP64 oracle on
the same rounded input.  The field is a sum of second differences, of the order theta^2, of values of order one.
Bar: a difference of two neighbours carries at most one rounding of 2^-24 theta; a second difference takes two of them
and a sum, and the weights of one plane can exceed the result's by the ratio r of the largest to the smallest of the
element constants along the axes: 4 r 2^-24 / theta relative to the result, taken inside the mesh (at the free faces
the field is of the order theta).  Sums of the values themselves leave 2^-24 / theta^2.
"""
import numpy as np
import pytest

import nm_inputs as inp
from helpers import gpu_mesh, oracle_mesh, rel_l2, rounded
from test_gpu_basis2d import _gpu2, _oracle2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nmgb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2411_11725_gb300 as nmgb
    nmgb.load()
    return nmgb


def _errors(nmgb, oracle_mod, p, nodes, theta, basis):
    import torch
    i = np.stack(np.meshgrid(*[np.arange(v) for v in nodes], indexing="ij"), -1)
    ph = theta * (i @ np.array([1.0, 0.7, 0.5])) + 0.3
    m = rounded(np.stack([0.8 * np.cos(ph), 0.8 * np.sin(ph), np.full(nodes, 0.6)], -1), 0)
    ref = (oracle_mesh if basis == 3 else _oracle2)(oracle_mod, p).h_eff(m, oracle_mod.EXCH, 0.0)
    me = (gpu_mesh if basis == 3 else _gpu2)(nmgb, p, 0)
    h = me.h_eff(torch.tensor(m, dtype=me.dtype, device="cuda"), nmgb.EXCH, 0.0).double().cpu().numpy()
    me.close()
    inside = tuple(slice(1, -1) if v > 2 else slice(None) for v in nodes)
    return rel_l2(h, ref), rel_l2(h[inside], ref[inside])


def _check(err, r, theta):
    assert err[0] < 1e-5  # the bar of every field test
    assert err[1] < 4 * r * 2.0 ** -24 / theta


@pytest.mark.parametrize("theta", [0.1, 0.01, 0.003])
@pytest.mark.parametrize("shape, dx", [((70, 33, 1), (3e-9, 3e-9, 3e-9)), ((40, 50, 3), (4e-9, 3e-9, 2e-9))])
def test_2d_basis(oracle_mod, nmgb, shape, dx, theta):
    p = inp.random_problem(np.random.default_rng(1), shape, dx=dx, heterogeneous=False)
    err = _errors(nmgb, oracle_mod, p, (shape[0] + 1, shape[1] + 1, 1), theta, 2)
    _check(err, max(dx[0] / dx[1], dx[1] / dx[0]) ** 2, theta)


@pytest.mark.parametrize("theta", [0.1, 0.01, 0.003])
@pytest.mark.parametrize("shape, dx", [((70, 9, 5), (3e-9, 3e-9, 3e-9)), ((40, 30, 2), (5e-9, 5e-9, 1e-9)),
                                       ((33, 20, 40), (2e-9, 2.5e-9, 3e-9)), ((60, 40, 1), (2.5e-9, 2.5e-9, 3e-9))])
def test_3d_basis(oracle_mod, nmgb, shape, dx, theta):
    p = inp.random_problem(np.random.default_rng(2), shape, dx=dx, heterogeneous=False)
    err = _errors(nmgb, oracle_mod, p, p.nodes, theta, 3)
    _check(err, (max(dx) / min(dx)) ** 2, theta)
