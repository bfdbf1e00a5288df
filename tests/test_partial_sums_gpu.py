"""Sums of the complex64 forms that are kept in FP64 (rounded once where they
are stored): where an FP64 sum is exact in any order, nothing of it may be
lost on the way."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mask", [(0, 1), (0, 1, 2), (0, 1, 5)])
@pytest.mark.parametrize("dkmax,odd", [(10, 5), (11, 7)])
@pytest.mark.parametrize("tile", [256, 1024])
def test_group_sums_of_long_runs(mask, dkmax, odd, tile):
    """Free two-level rotation by x = odd pi / (4 (dkmax - 1)) per step from
    rho(0) = diag(1, -1).  The amplitudes before the first merge are products
    of n = 2 (dkmax - 1) factors cos x and sin x, n log2(cot x) binades apart
    at most (20 and 14), and a group's sum is below (1 + tan x)^n / 2 of the
    largest (9 and 13 bits): with 24 bits of each amplitude a sum needs at most
    53, an FP64 sum is exact in any order.  After dkmax - 1 steps the diagonal
    group sums nearly cancel, and what is left shows every lost bit.  The
    stream engine's runs against the merge table's FP64 atomics, bit for bit."""
    from paper_2506_03127_gb300 import Propagator
    x = odd * np.pi / (4.0 * (dkmax - 1))
    rho0 = np.diag([1.0, -1.0])
    sets = []
    for engine in ("stream", "hash"):
        p = Propagator(2, dkmax, 1.0, (1.0, -1.0), np.array([[0.0, x], [x, 0.0]]), 1e-30, "c64", engine,
                       max_paths=1 << 23)
        p.set_eta(np.zeros(dkmax))
        p.set_mask(mask)
        p.set_rho0(rho0)
        if engine == "stream":
            p.set_tuning(stream_tile=tile)
        p.step(dkmax)
        keys, amps = p.export_paths()
        order = np.argsort(keys)
        sets.append((keys[order], amps[order]))
        p.close()
    assert np.array_equal(sets[0][0], sets[1][0])
    assert np.array_equal(sets[0][1], sets[1][1])
