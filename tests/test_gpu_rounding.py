"""Roundings of the kernels that no tolerance of the parity tests sees."""
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


def _rest_with_density_jumps(ssd, oracle_mod, precision, zone, N, E0):
    """Relative L2 error of the density residual of fluid at rest with total energy E0
    and a density of its own in every cell: only the Rusanov jump term, half the
    sound speed times the jump, is left."""
    SLIP = meshes.BC_SLIP
    m = meshes.channel_mesh(9, 7, 3.0, 2.0, tags=(SLIP,) * 4, zone=zone)
    prm = FlowParams(omega=0.0)
    E = len(m["elem_nodes"])
    Q = np.zeros((E, 4, N, N))
    Q[:, 0] = np.random.Generator(np.random.PCG64(N)).uniform(0.5, 1.5, E)[:, None, None]
    Q[:, 3] = E0
    s = ssd.Solver(m, N - 1, prm, precision=precision)
    s.sd_set_state(Q)
    R = s.sd_residual()[:, 0]
    s.close()
    ref = oracle_mod.Oracle(m, N, prm).residual(Q, 0.0)[:, 0]
    scale = np.abs(ref).max()
    return float(np.sqrt(((R / scale - ref / scale) ** 2).sum() / ((ref / scale) ** 2).sum()))


def _skewed(zone, cubic=False):
    """A channel of cells that are no parallelograms, all in one zone."""
    return meshes.channel_mesh(17, 11, 3.0, 2.0, cubic=cubic, zone=zone,
                               mapping=lambda x, y: (x + 0.07 * x * y, y + 0.05 * x * y + 0.03 * x))


@pytest.mark.parametrize("N", [3, 4, 5, 6])
@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("cubic", [False, True])
def test_stationary_cells_round_as_the_general_form(ssd, precision, N, cubic):
    """FP32 Euler: the branch for cells without rotation and grid velocity against
    the general one on a zone at rest at angle 0.  Every sum rounds the same way in
    both, so residuals and states are equal bit for bit."""
    R, S = [], []
    for zone in (0, 1):
        for rk in (3, 5):
            s = ssd.Solver(_skewed(zone, cubic), N - 1, FlowParams(omega=0.0, u_inf=0.3, rk_stages=rk), precision=precision)
            Q = s.state_from(lambda x, y: fields.random_smooth_state(x, y, seed=N, amp=0.05, scale=3.0))
            s.sd_set_state(Q)
            R.append(s.sd_residual())
            s.sd_step(2e-4, 10)
            s.sd_sync()
            S.append(s.sd_get_state())
            s.close()
    assert np.array_equal(R[0], R[2]) and np.array_equal(R[1], R[3])
    assert np.array_equal(S[0], S[2]) and np.array_equal(S[1], S[3])


@pytest.mark.parametrize("N", [3, 4, 5, 6])
@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("zone", [0, 1])
def test_fp32_sound_speed_of_a_subnormal_square(ssd, oracle_mod, precision, zone, N):
    """gamma p / rho = 5.6e-41, a subnormal float with spacing 1.4e-45 (2.5e-5 of it):
    N roundings of the trace of E, three of p and of the square, each half a
    spacing of values down to 4e-41 (1.8e-5), halved by the root: (N + 3) 0.9e-5
    <= 8.1e-5; twice that is allowed."""
    assert _rest_with_density_jumps(ssd, oracle_mod, precision, zone, N, 1e-40) <= 1.7e-4


@pytest.mark.parametrize("N", [3, 4, 5, 6])
def test_fp64_sound_speed_of_a_subnormal_square(ssd, oracle_mod, N):
    """The same in FP64, E = 1e-310: spacing 4.9e-324, so (N + 3) times
    4.9e-324 / 4e-311 / 4 = 3.1e-14, twice that on each of the two sides compared."""
    assert _rest_with_density_jumps(ssd, oracle_mod, 0, 0, N, 1e-310) <= 1.2e-12


# relative L2 error of the FP64 residual against the extended oracle with every
# contraction a plain chain of FMAs over the weights and the two sides' fluxes
# formed apart, by mesh and N (the cases of _fp64_residual_error)
PLAIN = {("rotor", 3): 2.769e-14, ("rotor", 4): 2.071e-14, ("rotor", 5): 2.743e-14, ("rotor", 6): 2.683e-14,
         ("twin", 3): 1.421e-14, ("twin", 4): 1.01e-14, ("twin", 5): 1.193e-14, ("twin", 6): 1.32e-14}


def _fp64_residual_error(ssd, oracle_mod, kind, N):
    """Root mean square over four smooth states."""
    mesh, prm = (small_rotor(scale=2, shift_R=0.05), FlowParams(omega=0.8)) if kind == "rotor" else \
        (small_twin(n_core2=5), FlowParams(omega=0.6))
    ext = oracle_mod.Oracle(mesh, N, prm, real="long")
    s = ssd.Solver(mesh, N - 1, prm, precision=0)
    e2 = []
    for seed in range(4):
        t = 0.3 + 0.7 * seed
        Q = s.state_from(lambda x, y: fields.random_smooth_state(x, y, seed=10 * N + seed, amp=0.2, scale=3.0))
        s.sd_set_state(Q)
        s.sd_set_time(t)
        ref = ext.residual(Q, t)
        d = s.sd_residual().astype(np.longdouble) - ref
        e2.append(float((d ** 2).sum() / (ref ** 2).sum()))
    s.close()
    return float(np.sqrt(np.mean(e2)))


@pytest.mark.parametrize("N", [3, 4, 5, 6])
@pytest.mark.parametrize("kind", ["rotor", "twin"])
def test_fp64_residual_error_no_larger_than_the_plain_form(ssd, oracle_mod, kind, N):
    """Folded sums and joint fluxes may not round worse than the plain form.  The
    error is a mean over 1e5 values and more, so 1 % is beyond its scatter."""
    e = _fp64_residual_error(ssd, oracle_mod, kind, N)
    print(f"{kind} N={N}: {e:.4g}, plain {PLAIN[kind, N]:.4g}")
    assert e <= 1.01 * PLAIN[kind, N]
