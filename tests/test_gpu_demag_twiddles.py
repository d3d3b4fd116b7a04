"""FP32 transforms of 128 and 256 values in radix-16 stages are as accurate as longer or equal ones in radix-8 stages,
whose twiddles all come from the table.  Error of the demag field of a random state against the FP64 mesh.  A
transform's error grows with its number of stages, so the reference lengths are at least as long; the error is an
average over more than 10^4 roundings (a per cent of scatter), hence a factor of 1.1.
"""
import numpy as np
import pytest

import nm_inputs as inp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nmgb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2411_11725_gb300 as nmgb
    nmgb.load()
    return nmgb


def _error(nmgb, n):
    import torch
    m = inp.unit_vectors(np.random.default_rng(3), tuple(v + 1 for v in n))
    m = torch.tensor(m, dtype=torch.float32, device="cuda")
    h = []
    for precision, dtype in ((nmgb.F32, torch.float32), (nmgb.F64, torch.float64)):
        me = nmgb.Mesh(n, (3e-9,) * 3, precision)
        me.set_material(1e6, 1.5e-11)
        h.append(me.h_eff(m.to(dtype), nmgb.DEMAG).double())
        me.close()
    return float((h[0] - h[1]).norm() / h[1].norm())


# y lines of 256 values in the fused y-z pass and in the y passes against 512; x lines of 128 values (256 cells) in
# 16 and 8 values per thread (by the number of lines)
@pytest.mark.parametrize("n, ref", [((30, 100, 1), (30, 200, 1)), ((30, 100, 8), (30, 200, 8)),
                                    ((128, 200, 17), (128, 130, 20))])
def test_radix16_lines(nmgb, n, ref):
    assert _error(nmgb, n) < 1.1 * _error(nmgb, ref)
