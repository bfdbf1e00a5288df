"""A launch that fails in the middle of qp_step (injected on the host): the
steps before it stay enqueued and the next qp_step goes on from them, without
a read of the state in between."""
import numpy as np
import pytest

import workloads as W
from oracle import iquapi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,dkmax,mask,theta", [(2, 5, None, 0.0), (2, 5, (0, 1, 2), 0.0), (3, 3, None, 0.0),
                                                (2, 6, (0, 1, 2, 4), 1e-6), (4, 3, (0, 1), 1e-6)])
def test_steps_after_a_failed_launch(M, dkmax, mask, theta):
    from paper_2506_03127_gb300 import Propagator, abi
    c = W.random_case(57, M, dkmax)
    p = Propagator(M, dkmax, c["dt"], c["q"], c["hs"], theta, "fp64", "stream", max_paths=1 << 18)
    p.set_eta(c["eta"])
    p.set_mask(mask)
    p.set_rho0(c["rho0"])
    abi.qp_test_fail_launch(p.ctx, 4)
    with pytest.raises(abi.QPError) as e:
        p.step(7)                                # four steps, then the failure
    assert e.value.status == abi.QP_ERR_CUDA
    p.step(5)
    T = 4 + 5
    rho, st = p.rho(0, T + 1), p.stats(1, T)
    assert p.current()[0] == T
    p.close()
    ref = iquapi.propagate(M, c["q"], c["hs"], c["dt"], c["eta"], dkmax, mask, theta, c["rho0"], T)
    assert np.abs(rho - ref.rho).max() <= 1e-10   # the FP64 bar of the other engine tests
    if not any(s.near_tie or s.near_theta for s in ref.stats):
        assert [(r[1], r[3]) for r in st] == [(o.groups, o.kept) for o in ref.stats]
