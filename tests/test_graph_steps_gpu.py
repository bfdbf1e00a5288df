"""Graphs of several steps (graph_steps > 1) against the oracle, on the paths
that run in graphs: the merge-table engine, batches on the stream engine and
the post-merging order.  Runs shorter than a graph, whole multiples and
remainders, through the fill of the window and past a restart."""
import numpy as np
import pytest

import workloads as W
from oracle import iquapi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("engine,n_inst,scheme", [("hash", 1, "pre"), ("hash", 3, "pre"), ("stream", 3, "pre"),
                                                  ("hash", 1, "post")])
@pytest.mark.parametrize("graph_steps", [2, 4])
def test_graphs_of_several_steps(engine, n_inst, scheme, graph_steps):
    from paper_2506_03127_gb300 import Propagator
    M, dkmax, mask, theta, parts = 2, 5, (0, 1, 2), 1e-6, (1, 4, 9, 2)
    c, T = W.random_case(61, M, dkmax), sum(parts)
    p = Propagator(M, dkmax, c["dt"], c["q"], c["hs"], theta, "fp64", engine, max_paths=1 << 14, n_inst=n_inst,
                   scheme=scheme)
    p.set_eta(c["eta"])
    p.set_mask(mask)
    p.set_tuning(graph_steps=graph_steps)
    ref = iquapi.propagate(M, c["q"], c["hs"], c["dt"], c["eta"], dkmax, mask, theta, c["rho0"], T, scheme=scheme)
    for _ in range(2):
        p.set_rho0(c["rho0"])
        for n in parts:
            p.step(n)
        rho = p.rho(0, T + 1).reshape(T + 1, n_inst, M, M)
        assert p.current()[0] == T
        assert np.abs(rho - ref.rho[:, None]).max() <= 1e-10   # the FP64 bar of the other engine tests
    p.close()
