"""The slope that a Dormand-Prince run keeps for its next step is formed anew whenever the state or the field behind it
has changed.  Each sequence against a fresh mesh that starts from the state in between; the same kernels on the same
values, so the states agree bit for bit.
"""
import numpy as np
import pytest

import nm_inputs as inp
from helpers import gpu_mesh

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nmgb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2411_11725_gb300 as nmgb
    nmgb.load()
    return nmgb


def _problem(heterogeneous):
    p = inp.random_problem(np.random.default_rng(4), (9, 6, 3), heterogeneous=heterogeneous)
    p.h_freq = 0.0
    p.h_cell = None
    return p


def _restart(nmgb, p, precision, me):
    """a new mesh at the resident state, time and step of me"""
    other = gpu_mesh(nmgb, p, precision)
    other.set_state(*me.get_state())
    return other


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("heterogeneous", [False, True])
def test_rk4_between_dp5_runs(nmgb, precision, heterogeneous):
    p = _problem(heterogeneous)
    me = gpu_mesh(nmgb, p, precision)
    me.set_state(p.m0, 0.0, 1e-13)
    me.run_steps(2, nmgb.DP54)
    me.run_steps(3, nmgb.RK4)
    ref = _restart(nmgb, p, precision, me)
    for mesh in (me, ref):
        mesh.run_steps(2, nmgb.DP54)
    assert np.array_equal(me.get_state()[0], ref.get_state()[0])
    me.close()
    ref.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("kind", ["uniform", "cell", "cell off"])
def test_field_changed_between_dp5_runs(nmgb, precision, kind):
    p = _problem(False)
    h_cell = np.random.default_rng(5).standard_normal(p.n + (3,)) * 1e5
    if kind == "cell off":
        p.h_cell = h_cell
    me = gpu_mesh(nmgb, p, precision)
    me.set_state(p.m0, 0.0, 1e-13)
    me.run_steps(2, nmgb.DP54)
    if kind == "uniform":
        p.h_uniform = (2e5, -1e5, 3e5)
        me.set_uniform_field(p.h_uniform)
    else:
        p.h_cell = h_cell if kind == "cell" else None
        me.set_zeeman(p.h_uniform, 0.0, p.h_phase, p.h_cell, p.cell_freq, p.cell_phase)
    ref = _restart(nmgb, p, precision, me)
    for mesh in (me, ref):
        mesh.run_steps(2, nmgb.DP54)
    assert np.array_equal(me.get_state()[0], ref.get_state()[0])
    me.close()
    ref.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_step_from_another_time(nmgb, precision):
    """With a field that oscillates, a step from a time other than the resident one has another first slope."""
    p = _problem(False)
    p.h_uniform, p.h_freq = (3e6, 0.0, 0.0), 1e12
    me = gpu_mesh(nmgb, p, precision)
    me.set_state(p.m0, 0.0, 1e-14)
    me.run_steps(1, nmgb.DP54)
    m, t, _ = me.get_state()
    ref = gpu_mesh(nmgb, p, precision)
    ref.set_state(m, t + 3e-13, 1e-14)
    for mesh in (me, ref):
        assert mesh.llg_step(nmgb.DP54, t + 3e-13, 1e-14)[0]
    assert np.array_equal(me.get_state()[0], ref.get_state()[0])
    me.close()
    ref.close()


@pytest.mark.parametrize("method", ["RK4", "DP54"])
@pytest.mark.parametrize("precision", [0, 1])
def test_profiled_step_first(nmgb, precision, method):
    """The first use of a state: the FP32 copy of the one before must not be used."""
    p = _problem(False)
    out = []
    for profiled in (True, False):
        me = gpu_mesh(nmgb, p, precision)
        me.set_state(np.roll(p.m0, 1, axis=0), 0.0, 1e-13)
        me.run_steps(1, getattr(nmgb, method))
        me.set_state(p.m0, 0.0, 1e-13)
        if profiled:
            me.profile_step(getattr(nmgb, method), reps=1)
        else:
            me.run_steps(1, getattr(nmgb, method))
        out.append(me.get_state()[0])
        me.close()
    assert np.array_equal(out[0], out[1])
