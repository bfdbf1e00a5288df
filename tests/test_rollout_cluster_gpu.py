"""The cluster rollout at the edges of its shapes (columns per block and warp,
ring of one step, parameters up to the padding, one and two row tiles)
against the step kernels."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,L,n_par,width", [(1, 1, 1, 8), (16, 3, 2, 40), (17, 4, 1, 64), (5, 31, 8, 248), (32, 32, 2, 256),
                                             (9, 12, 3, 264)])
def test_rollout_matches_step_kernels(n, L, n_par, width):
    from paper_2506_03127_gb300.surrogate import Surrogate
    rng = np.random.default_rng(n + L)
    s = Surrogate(L=L, width=width, n_par=n_par)
    s.net.init(seed=5, out_gain=0.5)
    T = 4 * L + 9
    a = rng.normal(size=(n, L, 2, 2)) + 1j * rng.normal(size=(n, L, 2, 2))
    rho0 = a @ np.conj(np.swapaxes(a, -1, -2))
    rho0 /= np.trace(rho0, axis1=-2, axis2=-1).real[..., None, None]
    par = rng.uniform(0.1, 2.0, size=(n, n_par))
    rf, rg = s.rollout(rho0, par, T), s.rollout(rho0, par, T, mode="graph")
    # the same rounding points and k order; the update may contract differently (as in the surrogate tests)
    assert np.abs(rf - rg).max() <= 1e-6
    assert np.abs(rf[:, L:]).max() > 0
