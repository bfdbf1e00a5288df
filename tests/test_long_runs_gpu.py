"""Pre-merge groups of many paths on the stream engine: masks that collapse a
filled window onto few positions give runs on both sides of every class of
the tile kernel (one owner thread up to 32 members, a warp up to 512, the
block beyond, runs across several tiles), with and without the sub-groups of
an extra position, and ends of regions inside a run."""
import numpy as np
import pytest

import workloads as W
from oracle import iquapi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,dkmax,mask", [
    (2, 5, (0, 1)), (2, 6, (0, 1)), (2, 8, (0, 1)),            # runs of 64, 256, 4096 members
    (2, 7, (0, 1, 4)), (2, 8, (0, 1, 7)), (2, 8, (0, 1, 2, 5)),   # four sub-groups per run
    (3, 4, (0, 1)), (3, 5, (0, 1)),                            # 81, 729 members
    (4, 3, (0, 1))])
@pytest.mark.parametrize("theta", [0.0, 1e-4])
@pytest.mark.parametrize("precision", ["fp64", "c64"])
@pytest.mark.parametrize("tile", [256, 1024])
def test_long_runs(M, dkmax, mask, theta, precision, tile, monkeypatch):
    from paper_2506_03127_gb300 import Propagator
    c = W.random_case(60 + dkmax, M, dkmax)
    T = dkmax + 3
    p = Propagator(M, dkmax, c["dt"], c["q"], c["hs"], theta, precision, "stream", max_paths=1 << 19)
    p.set_eta(c["eta"])
    p.set_mask(mask)
    p.set_rho0(c["rho0"])
    p.set_tuning(stream_tile=tile)
    p.step(T)
    rho, st = p.rho(0, T + 1), p.stats(1, T)
    p.close()
    if precision == "c64":   # the complex64 tie window
        monkeypatch.setattr(iquapi, "TIE_REL", 1e-6)
    ref = iquapi.propagate(M, c["q"], c["hs"], c["dt"], c["eta"], dkmax, mask, theta, c["rho0"], T)
    scale = max(1.0, np.abs(ref.rho).max())
    if precision == "fp64":
        assert np.abs(rho - ref.rho).max() <= 1e-10 * scale
        if not any(s.near_tie or s.near_theta for s in ref.stats):
            assert [(r[1], r[3]) for r in st] == [(o.groups, o.kept) for o in ref.stats]
    else:   # FP32 children (2^-24 per operation); a child at the filter's edge may fall on either side (theta each)
        assert np.abs(rho - ref.rho).max() <= 4e-6 * scale + 20 * theta * (theta > 0)
