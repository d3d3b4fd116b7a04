"""FP32 Dormand-Prince steps on uniform materials form the error in the node kernels of stages 6 and 7, and the last block
of stage 7 takes the step decision.  One attempt from a random state at the edges of the node tiles, on one to many
blocks, accepted and rejected, against the separate error kernel with every term in FP64 (nm_set_error_norm), which sees
the same FP32 slopes.  The terms differ by the FP32 rounding of sum_j e_j (k_j - k_1): at most a dozen roundings of
values below 2 max|k| sum|e_j|, with |k| below twice gamma' (1 + alpha) max|H| over a step, weighted by dt / atol.  The
step that follows an accepted attempt takes the stored increment: the state against the same step with the other
kernel, which forms it from the slopes (bitwise the same sum).
"""
import numpy as np
import pytest

import nm_inputs as inp

pytestmark = pytest.mark.gpu

E = [71 / 57600, -71 / 16695, 71 / 1920, -17253 / 339200, 22 / 525, -1 / 40]


@pytest.fixture(scope="module")
def nmgb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2411_11725_gb300 as nmgb
    nmgb.load()
    return nmgb


@pytest.mark.parametrize("basis, shape", [(3, (1, 1, 1)), (3, (31, 4, 2)), (3, (32, 3, 1)), (3, (70, 9, 5)), (3, (3, 40, 33)),
                                          (2, (1, 1, 1)), (2, (31, 4, 1)), (2, (33, 9, 2)), (2, (260, 700, 1))])
@pytest.mark.parametrize("dt", [1e-13, 6e-13, 1.2e-12])
def test_attempt(nmgb, basis, shape, dt):
    import torch
    rng = np.random.default_rng(sum(shape))
    m0 = inp.unit_vectors(rng, (shape[0] + 1, shape[1] + 1, shape[2] + 1 if basis == 3 else 1))
    alpha, gamma, tol = 0.1, 2.2127614872e5, 1e-5
    out = []
    for f64_terms in (False, True):
        me = nmgb.Mesh(shape, (3e-9, 3e-9, 3e-9), nmgb.F32, basis=basis)
        me.set_material(1e6, 1.5e-11, 5e5, (0.0, 0.0, 1.0), alpha, gamma)
        me.set_terms(nmgb.EXCH | nmgb.ANIS | nmgb.DEMAG)
        me.set_error_norm(f64_terms)
        hmax = float(me.h_eff(torch.tensor(m0, dtype=torch.float32, device="cuda"),
                              nmgb.EXCH | nmgb.ANIS | nmgb.DEMAG).norm(dim=-1).max())
        me.set_state(m0, 0.0, dt)
        acc, _, _ = me.llg_step(nmgb.DP54, 0.0, dt, tol, tol)
        out.append((acc, me.counters()[2], me.get_state()[0]))
        me.close()
    (a, e, m), (b, f, n) = out
    bound = 12 * 2.0 ** -24 * 2 * sum(abs(v) for v in E) * dt / tol * 2 * gamma / (1 + alpha ** 2) * (1 + alpha) * hmax
    assert a == b
    assert abs(e - f) <= bound, (e, f, bound)
    # (FP32 increments; a contraction of their last product differs by one rounding of at most dt |k|)
    assert np.abs(m - n).max() <= 2.0 ** -22
