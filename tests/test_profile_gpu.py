"""qp_profile_steps reports the time of every kernel that the steps launch, and
none for those that they do not."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,theta,engine,n_inst,mask,kernels", [
    (2, 0.0, "stream", 1, None, (0,)), (3, 0.0, "stream", 1, None, (0,)),      # regular map alone
    (4, 0.0, "stream", 1, None, (2,)), (3, 1e-6, "stream", 1, None, (2,)),     # tile kernel alone
    (2, 1e-6, "stream", 3, None, (2,)),
    (2, 1e-6, "hash", 1, (0, 1, 3), (0, 1, 2)), (2, 1e-6, "hash", 3, (0, 1, 3), (0, 1, 2, 3))])
def test_kernels_of_a_step(M, theta, engine, n_inst, mask, kernels):
    from paper_2506_03127_gb300 import Propagator
    c = W.random_case(59, M, 4)
    p = Propagator(M, 4, c["dt"], c["q"], c["hs"], theta, "fp64", engine, max_paths=1 << 18, n_inst=n_inst)
    p.set_eta(c["eta"])
    p.set_mask(mask)
    p.set_rho0(c["rho0"])
    p.step(6)
    ms = p.profile(5)
    assert p.current()[0] == 11
    p.close()
    assert tuple(np.flatnonzero(ms)) == kernels and (ms[list(kernels)] > 0).all()
