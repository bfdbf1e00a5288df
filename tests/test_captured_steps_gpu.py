"""Steps recorded into a caller's graph (QP_NO_GRAPH: qp_step launches kernels
that read the step index from the device), replayed, and followed by direct
steps without a read of the state in between: the host does not see the
replays, so the direct steps must read the device state too."""
import numpy as np
import pytest

import workloads as W
from oracle import iquapi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,dkmax,mask,theta", [(2, 5, None, 0.0), (2, 5, (0, 1, 2), 0.0), (3, 3, None, 0.0),
                                                (2, 6, (0, 1, 2, 4), 1e-6), (4, 3, (0, 1), 1e-6)])
@pytest.mark.parametrize("precision", ["fp64", "c64"])
def test_capture_replay_step(M, dkmax, mask, theta, precision, monkeypatch):
    import torch
    from paper_2506_03127_gb300 import Propagator
    monkeypatch.setenv("QP_NO_GRAPH", "1")
    c = W.random_case(56, M, dkmax)
    p = Propagator(M, dkmax, c["dt"], c["q"], c["hs"], theta, precision, "stream", max_paths=1 << 18)
    p.set_eta(c["eta"])
    p.set_mask(mask)
    p.set_rho0(c["rho0"])
    p.step(1)
    p.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=p.stream):
        p.step(2)
    with torch.cuda.stream(p.stream):
        for _ in range(3):
            g.replay()
    p.step(3)
    with torch.cuda.stream(p.stream):
        g.replay()
    p.step(1)
    T = 1 + 2 * 3 + 3 + 2 + 1
    assert p.current()[0] == T
    rho, st = p.rho(0, T + 1), p.stats(1, T)
    p.close()
    ref = iquapi.propagate(M, c["q"], c["hs"], c["dt"], c["eta"], dkmax, mask, theta, c["rho0"], T)
    # FP64: the bar of the other engine tests; complex64: 2^-24 per operation, a few tens of them per step
    assert np.abs(rho - ref.rho).max() <= (1e-10 if precision == "fp64" else 1e-5 * max(1.0, np.abs(ref.rho).max()))
    if precision == "fp64" and not any(s.near_tie or s.near_theta for s in ref.stats):
        assert [(r[1], r[3]) for r in st] == [(o.groups, o.kept) for o in ref.stats]


@pytest.mark.parametrize("engine", ["stream", "hash"])
def test_a_start_under_capture_is_refused(engine):
    """qp_set_rho0 on a stream under capture sets nothing: it is refused, the
    capture stays valid and the running propagation goes on."""
    import torch
    from paper_2506_03127_gb300 import Propagator, abi
    M, dkmax, T = 2, 5, 9
    c = W.random_case(58, M, dkmax)
    p = Propagator(M, dkmax, c["dt"], c["q"], c["hs"], 0.0, "fp64", engine, max_paths=1 << 14)
    p.set_eta(c["eta"])
    p.set_mask(None)
    p.set_rho0(c["rho0"])
    p.step(4)
    p.sync()
    x, g = torch.zeros(1, device="cuda"), torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=p.stream):
        x.add_(1)
        with pytest.raises(abi.QPError) as e:
            p.set_rho0(np.eye(2) / 2)
        assert e.value.status == abi.QP_ERR_CUDA
    p.step(T - 4)
    rho = p.rho(0, T + 1)
    p.close()
    ref = iquapi.propagate(M, c["q"], c["hs"], c["dt"], c["eta"], dkmax, None, 0.0, c["rho0"], T)
    assert np.abs(rho - ref.rho).max() <= 1e-10
