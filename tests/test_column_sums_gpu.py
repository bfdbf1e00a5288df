"""rho(t) of complex64 problems with M >= 3 on the tile kernel: columns of the
staged children, and the children past the staging buffer (tiles of more
groups than a third of the tile kernel's size: the filling window)."""
import numpy as np
import pytest

import workloads as W
from oracle import iquapi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,dkmax,T", [(3, 5, 7), (4, 4, 6)])
@pytest.mark.parametrize("tile", [256, 512, 1024])
@pytest.mark.parametrize("theta", [1e-7, 3e-4])
def test_rho_of_every_step(M, dkmax, T, tile, theta):
    from paper_2506_03127_gb300 import Propagator
    c = W.random_case(60 + M, M, dkmax)
    mask = (0, 1, 2)
    p = Propagator(M, dkmax, c["dt"], c["q"], c["hs"], theta, "c64", "stream", max_paths=1 << 19)
    p.set_eta(c["eta"])
    p.set_mask(mask)
    p.set_rho0(c["rho0"])
    p.set_tuning(stream_tile=tile)
    p.step(T)
    rho, st = p.rho(0, T + 1), p.stats(1, T)
    p.close()
    ref = iquapi.propagate(M, c["q"], c["hs"], c["dt"], c["eta"], dkmax, mask, theta, c["rho0"], T)
    # 2^-24 per operation, a few tens of them per step; a child within that of
    # the filter may be kept on one side only (it weighs theta at most)
    flips = sum(abs(a[3] - b.kept) for a, b in zip(st, ref.stats))
    assert flips <= 1e-4 * sum(b.kept for b in ref.stats)
    scale = max(1.0, np.abs(ref.rho).max())
    assert np.abs(rho - ref.rho).max() <= 4e-6 * scale + flips * theta


@pytest.mark.parametrize("tile", [512, 1024])
def test_rho_of_batches(tile):
    """Instances of M = 2 whose filling windows have more groups per tile than
    the staging buffer holds (tiles of 512 at 8e4 paths and more)."""
    from paper_2506_03127_gb300 import Propagator
    n_inst, dkmax, T, theta, mask = 24, 7, 9, 1e-7, (0, 1, 2, 3)
    c = [W.random_case(80 + i, 2, dkmax) for i in range(n_inst)]
    p = Propagator(2, dkmax, c[0]["dt"], c[0]["q"], c[0]["hs"], theta, "c64", "stream", max_paths=1 << 20, n_inst=n_inst)
    p.set_eta(c[0]["eta"])
    for i in range(n_inst):
        p.set_eta_instance(i, c[i]["eta"])
    p.set_mask(mask)
    p.set_rho0(c[0]["rho0"])
    p.set_tuning(stream_tile=tile)
    p.step(T)
    rho, kept = p.rho(0, T + 1), np.array([p.instance_counts(t) for t in range(1, T + 1)])
    p.close()
    for i in range(n_inst):
        ref = iquapi.propagate(2, c[0]["q"], c[0]["hs"], c[0]["dt"], c[i]["eta"], dkmax, mask, theta, c[0]["rho0"], T)
        flips = sum(abs(int(a) - b.kept) for a, b in zip(kept[:, i], ref.stats))
        assert flips <= 1e-4 * sum(b.kept for b in ref.stats) + 1
        assert np.abs(rho[:, i] - ref.rho).max() <= 4e-6 * max(1.0, np.abs(ref.rho).max()) + flips * theta
