"""Wide keys: masks whose runs start, end and cross at the word boundary of
the key (position 8), windows from one point to sixteen, every number of
states, and filters from none (all M^2 children of 256 groups listed) to
almost everything dropped, against the oracle."""
import numpy as np
import pytest

import workloads as W
from oracle import iquapi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,dkmax,mask,theta,steps", [
    (2, 1, None, 0.0, 6), (2, 2, None, 0.0, 6), (3, 4, (0, 1), 0.0, 7), (8, 2, None, 0.0, 4),
    (2, 9, (0, 1, 2, 3, 8), 0.0, 11), (2, 9, (0, 1, 2, 3, 4, 5, 6, 7, 8), 1e-4, 12),
    (2, 10, (0, 1, 7, 8, 9), 1e-5, 13), (2, 16, (0, 1, 2, 3, 6, 8, 9, 11, 15), 1e-3, 20),
    (5, 8, (0, 1, 2), 4e-4, 11), (6, 9, (0, 1, 2, 8), 1e-3, 12), (8, 10, (0, 1, 2, 8, 9), 4e-3, 13),
    (8, 3, (0, 1), 0.9, 6)])
def test_wide_runs(M, dkmax, mask, theta, steps):
    from paper_2506_03127_gb300 import WidePropagator
    c = W.random_case(80 + dkmax, M, dkmax)
    p = WidePropagator(M, dkmax, c["dt"], c["q"], c["hs"], theta, "fp64", max_paths=1 << 20)
    p.set_eta(c["eta"])
    p.set_mask(range(dkmax) if mask is None else mask)
    p.set_rho0(c["rho0"])
    p.step(steps)
    rho, st = p.rho(0, steps + 1), p.stats(1, steps)
    p.close()
    ref = iquapi.propagate(M, c["q"], c["hs"], c["dt"], c["eta"], dkmax, mask, theta, c["rho0"], steps)
    assert np.abs(rho - ref.rho).max() <= 1e-10 * max(1.0, np.abs(ref.rho).max())
    if not any(s.near_tie or s.near_theta for s in ref.stats):
        assert [(r[1], r[3]) for r in st] == [(o.groups, o.kept) for o in ref.stats]
