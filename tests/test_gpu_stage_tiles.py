"""The one-launch stage of the FP32 Euler forms with several tiles per block (the
refill of its buffers, the face records and traces that arrive one tile ahead,
tiles in both directions), and with more coupling blocks than blocks.  Other
tests' meshes give a block one tile at most, but for N = 6 with a double-float
state and three stages."""
import numpy as np
import pytest

from ssd_inputs import fields, meshes
from ssd_inputs.workloads import FlowParams, stable_dt

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ssd():
    import paper_1503_02198_gb300 as pkg
    pkg.build()
    return pkg


@pytest.fixture(scope="module")
def mesh():
    """28,185 cells (odd, so no tile size divides it): 2.3 to 4.6 tiles for each of 760 blocks."""
    return meshes.rotor_mesh(half_width=10.0, n_cart=144, n_hole=54, r_interface=3.0, n_core=33, core_half=1.5,
                             n_ring_in=31, n_ring_out=24)


_ref = {}


def _reference(ssd, mesh, N, rk):
    """The FP64 form's step (kernels of its own: a face pass and k_volume)."""
    if (N, rk) not in _ref:
        prm = FlowParams(omega=0.8, rk_stages=rk)
        dt = stable_dt(mesh, N, prm, 4.0)
        s = ssd.Solver(mesh, N - 1, prm, precision=0)
        Q = s.state_from(lambda x, y: fields.random_smooth_state(x, y, seed=N, amp=0.2, scale=3.0))
        s.sd_set_state(Q)
        s.sd_set_time(0.7)
        R = s.sd_residual()
        s.sd_step(dt, 3)
        s.sd_sync()
        _ref.clear()
        _ref[N, rk] = prm, dt, Q, R, s.sd_get_state()
        s.close()
    return _ref[N, rk]


@pytest.mark.parametrize("N", [3, 4, 5, 6])
@pytest.mark.parametrize("rk", [3, 5])
@pytest.mark.parametrize("precision", [1, 2])
def test_several_tiles_per_block(ssd, mesh, precision, N, rk):
    """What three steps add to the state: good to the residual's FP32 tolerance (5e-5
    relative L2) and, with a float state, to a rounding of 2^-24 of the state at the
    start and in each of the stages."""
    prm, dt, Q, R, q = _reference(ssd, mesh, N, rk)
    assert len(mesh["elem_nodes"]) % 2 == 1
    s = ssd.Solver(mesh, N - 1, prm, precision=precision)
    s.sd_set_state(Q)
    s.sd_set_time(0.7)
    r = s.sd_residual()
    s.sd_step(dt, 1)  # both sets of tables and traces, continued over calls
    s.sd_step(dt, 2)
    s.sd_sync()
    out = s.sd_get_state()
    s.close()
    norm = lambda a: float(np.sqrt((a ** 2).sum()))  # noqa: E731
    # (a residual of a float state is that of the rounded state)
    if precision == 1:
        assert norm(r - R) <= 5e-5 * norm(R)
    tol = 5e-5 + (0.0 if precision == 1 else 2.0 ** -24 * np.sqrt(1 + 3 * rk) * norm(q) / norm(q - Q))
    assert norm(out - q) <= tol * norm(q - Q)


@pytest.mark.parametrize("N", [3, 4, 5, 6])
@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("rk", [3, 5])
def test_more_coupling_blocks_than_blocks(ssd, oracle_mod, precision, N, rk):
    """A row of cells as long as one tile: one block, and its boundary points are two
    coupling blocks (N = 4: 104 points, 96 threads)."""
    n = {3: 16, 4: 12, 5: 12, 6: 8}[N]
    m, prm = meshes.channel_mesh(n, 1, 3.0, 0.25), FlowParams(u_inf=0.3, rk_stages=rk)
    o = oracle_mod.Oracle(m, N, prm)
    Q = o.state_from(lambda x, y: fields.random_smooth_state(x, y, seed=N, amp=0.05, scale=3.0))
    s = ssd.Solver(m, N - 1, prm, precision=precision)
    s.sd_set_state(Q)
    R = s.sd_residual()
    s.sd_step(1e-4, 3)
    s.sd_sync()
    q, _ = o.step(Q, 0.0, 1e-4, 3, rk)
    ref = o.residual(Q, 0.0)
    if precision == 1:
        assert np.sqrt(((R - ref) ** 2).sum() / (ref ** 2).sum()) <= 5e-5
    assert np.sqrt(((s.sd_get_state() - q) ** 2).sum() / (q ** 2).sum()) <= 1e-5
    s.close()
