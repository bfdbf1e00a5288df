"""The wide expansion's bound on the children's weights at the edge of FP64:
amplitudes whose squares underflow may still have children above the filter."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("amp,eta0", [(1e-154, -14.0), (1e-158, -14.0), (1e-162, -14.0), (1e100, 93.5)])
def test_children_of_amplitudes_with_underflowed_squares(amp, eta0):
    """eta_0 = -14 multiplies off-diagonal children by exp(56): above theta =
    1e-140 from amplitudes of 1e-162 on; eta_0 = 93.5 by exp(-374), whose
    square underflows, above theta from 1e100.  The same paths and rho as on
    the 64-bit keys, which form every child."""
    from paper_2506_03127_gb300 import Propagator, WidePropagator
    hs = np.array([[0.0, 0.7], [0.7, 0.0]])
    out = []
    for cls in (WidePropagator, Propagator):
        p = cls(2, 3, 1.0, (1.0, -1.0), hs, 1e-140, "fp64", max_paths=1 << 10)
        p.set_eta(np.array([eta0, 0.0, 0.0]))
        p.set_mask((0, 1, 2))
        p.set_rho0(np.array([[amp, amp], [amp, amp]]))
        p.step(1)
        out.append((p.rho(0, 2), [(r[1], r[3]) for r in p.stats(1, 1)]))
        p.close()
    assert out[0][1] == out[1][1]
    assert out[1][1][0][1] > 0
    assert np.abs(out[0][0] - out[1][0]).max() <= 1e-12 * np.abs(out[1][0]).max()
