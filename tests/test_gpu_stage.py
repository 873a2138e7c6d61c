"""The one-launch stage of the FP32 Euler forms against the oracle: tiles that are
not full (cell counts that no tile divides), boundary points and mortars worked
by the first blocks of the launch, several zones, both integrators, every N.
And captured steps continued over other calls: the stage tables merged beside
the last step, and the trace buffer it wrote, serve the next call only while
time, step size and state are what they were.  Tolerances are those of the
FP32 forms (residual: the FP64 round-off amplification times the FP32 unit
round-off, 5e-5; state after steps 1e-5, relative L2)."""
import numpy as np
import pytest

from helpers import small_rotor, small_twin
from ssd_inputs import fields, meshes
from ssd_inputs.workloads import FlowParams

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ssd():
    import paper_1503_02198_gb300 as pkg
    pkg.build()
    return pkg


def _rel(a, b):
    return float(np.sqrt(((a - b) ** 2).sum() / (b ** 2).sum()))


def _mesh(kind):
    if kind == "channel":  # 35 straight cells with inlet, outlet and slip walls, no interface
        return meshes.channel_mesh(7, 5, 3.0, 2.0), FlowParams(u_inf=0.3)
    if kind == "channel_cubic":  # 12-node cells of a rotating zone: per-point face rows
        return meshes.channel_mesh(5, 3, 3.0, 2.0, cubic=True, zone=1), FlowParams(omega=0.4, u_inf=0.3)
    if kind == "twin":
        return small_twin(n_core2=5), FlowParams(omega=0.6)
    return small_rotor(shift_R=0.05), FlowParams(omega=0.8)


@pytest.mark.parametrize("N", [3, 4, 5, 6])
@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("kind", ["channel", "channel_cubic", "rotor", "twin"])
def test_residual_and_steps_match_the_oracle(ssd, oracle_mod, kind, precision, N):
    m, prm = _mesh(kind)
    o = oracle_mod.Oracle(m, N, prm)
    Q = o.state_from(lambda x, y: fields.random_smooth_state(x, y, seed=N, amp=0.05, scale=3.0))
    for rk in (3, 5):
        prm.rk_stages = rk
        s = ssd.Solver(m, N - 1, prm, precision=precision)
        s.sd_set_state(Q)
        s.sd_set_time(0.7)
        if rk == 3:
            assert _rel(s.sd_residual(), o.residual(Q, 0.7)) <= 5e-5
        s.sd_step(1e-3, 3)
        s.sd_sync()
        q, _ = o.step(Q, 0.7, 1e-3, 3, rk)
        assert _rel(s.sd_get_state(), q) <= 1e-5
        s.close()


@pytest.mark.parametrize("precision,viscous", [(0, 0), (1, 0), (2, 0), (1, 1)])
def test_steps_continue_over_other_calls(ssd, oracle_mod, precision, viscous):
    m = small_rotor(shift_L=0.02)
    prm = FlowParams(omega=0.8, viscous=viscous, mu=1e-3)
    a, b = (ssd.Solver(m, 3, prm, precision=precision) for _ in range(2))
    Q = a.state_from(lambda x, y: fields.isentropic_vortex(x, y, x0=2.5, y0=0.5))
    for s in (a, b):
        s.sd_set_state(Q)
        s.sd_set_time(0.3)
    # (a state out and in again is a FP64 sum split anew, so both handles do it)
    a.sd_step(1e-3, 5)
    a.sd_set_state(a.sd_get_state())
    a.sd_step(1e-3, 3)
    b.sd_step(1e-3, 3)  # odd: the second stage-table set and trace buffer come next
    b.sd_residual()
    b.sd_step(1e-3, 2)
    q = b.sd_get_state()
    b.sd_set_state(q)  # new traces into the current buffer
    b.sd_step(1e-3, 1)
    b.sd_profile_step(1e-3, 1)  # a step outside the captured ones: tables merged again after it
    b.sd_step(1e-3, 1)
    a.sd_sync()
    b.sd_sync()
    assert np.array_equal(a.sd_get_state(), b.sd_get_state())
    # a new time between calls of the same step size
    b.sd_set_time(1.1)
    q = b.sd_get_state()
    b.sd_step(1e-3, 1)
    b.sd_sync()
    ref, _ = oracle_mod.Oracle(m, 4, prm).step(q, 1.1, 1e-3, 1)
    assert _rel(b.sd_get_state(), ref) <= (1e-12 if precision == 0 else 1e-5)
    a.close()
    b.close()
