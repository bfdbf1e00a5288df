"""The merge table of the wide-key context at its largest load: a first merge
with as many groups as stored paths."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("states,dkmax", [((0, 1, 3, 7), 7), ((1, 2, 5), 9)])
def test_as_many_groups_as_paths(states, dkmax):
    """m of eight states coupled, rho(0) on one element: (m^2)^(dkmax-1) paths
    in as many groups at the first merge, half of the table's slots.  With
    these keys the longest probe sequence is above 64 slots in two orders of
    insertion out of three or more.  Against the m-state problem on the 64-bit
    keys."""
    from paper_2506_03127_gb300 import Propagator, WidePropagator
    states, m = list(states), len(states)
    c = W.random_case(90, m, dkmax)
    q8, h8 = 2.0 + np.arange(8.0), np.zeros((8, 8), dtype=complex)
    q8[states] = c["q"]
    h8[np.ix_(states, states)] = c["hs"]
    rho8, rhom = np.zeros((8, 8)), np.zeros((m, m))
    rho8[states[0], states[0]] = rhom[0, 0] = 1.0
    MM, theta = m * m, 1e-40
    cap = MM ** dkmax // 16 * 16 + 16 * MM
    out = []
    for make, M, rho0, runs in ((lambda: WidePropagator(8, dkmax, c["dt"], q8, h8, theta, "fp64", max_paths=cap,
                                                        max_groups=MM ** (dkmax - 1)), 8, rho8, 4),
                                (lambda: Propagator(m, dkmax, c["dt"], c["q"], c["hs"], theta, "fp64", "stream",
                                                    max_paths=cap), m, rhom, 1)):
        p = make()
        p.set_eta(c["eta"])
        p.set_mask(range(dkmax))
        for _ in range(runs):
            p.set_rho0(rho0)
            p.step(dkmax)
            out.append((p.rho(0, dkmax + 1), [(r[1], r[3]) for r in p.stats(1, dkmax)]))
        p.close()
        del p
    for rho, counts in out:
        assert counts == [(MM ** t, MM ** (t + 1)) for t in range(dkmax)]
    for rho, _ in out[:-1]:
        assert np.abs(rho[:, states][:, :, states] - out[-1][0]).max() <= 1e-10
