"""Steps whose surplus blocks start late: a grid above residency and another
stream's kernels on the SMs.  A block that has no work in a step must not take
part in the next one, whose state the step's last block publishes while such a
block may not have started."""
import numpy as np
import pytest

import workloads as W
from oracle import iquapi

pytestmark = pytest.mark.gpu


def _beside_other_work(p, start, steps, runs):
    import torch
    other, a = torch.cuda.Stream(), torch.randn(4096, 4096, device="cuda", dtype=torch.bfloat16)
    torch.cuda.synchronize()
    out = []
    for _ in range(runs):
        with torch.cuda.stream(other):
            for _ in range(6):
                b = a @ a
        start()
        for _ in range(steps):
            p.step(1)
        out.append((p.rho(0, steps + 1), [(r[1], r[3]) for r in p.stats(1, steps)]))
    torch.cuda.synchronize()
    del b
    return out


def _check(out, c, M, dkmax, theta, mask, steps):
    ref = iquapi.propagate(M, c["q"], c["hs"], c["dt"], c["eta"], dkmax, mask, theta, c["rho0"], steps)
    for rho, counts in out:
        assert counts == [(o.groups, o.kept) for o in ref.stats]
        assert np.abs(rho - ref.rho).max() <= 1e-10   # the FP64 bar of the other engine tests


@pytest.mark.parametrize("M,dkmax,mask", [(2, 7, (0, 1, 2, 4, 6)), (3, 4, (0, 1, 3))])
def test_extension_of_the_merge_table(M, dkmax, mask):
    from paper_2506_03127_gb300 import Propagator
    import torch
    c = W.random_case(60 + M, M, dkmax)
    steps = dkmax + 3
    p = Propagator(M, dkmax, c["dt"], c["q"], c["hs"], 0.0, "fp64", "hash", max_paths=1 << 18)
    p.set_eta(c["eta"])
    p.set_mask(mask)
    p.set_rho0(c["rho0"])
    p.set_tuning(expand_blocks_per_sm=2048 // torch.cuda.get_device_properties(0).multi_processor_count)
    out = _beside_other_work(p, lambda: p.set_rho0(c["rho0"]), steps, 20)
    p.close()
    _check(out, c, M, dkmax, 0.0, mask, steps)


@pytest.mark.parametrize("M,dkmax", [(2, 7), (3, 4)])
def test_regular_steps_that_read_the_state(M, dkmax):
    """A mask taken up and dropped again after qp_set_rho0: the counts are no
    longer known on the host, every step reads them from the device."""
    from paper_2506_03127_gb300 import Propagator
    c = W.random_case(60 + M, M, dkmax)
    steps = dkmax + 3
    p = Propagator(M, dkmax, c["dt"], c["q"], c["hs"], 0.0, "fp64", "stream", max_paths=1 << 18)
    p.set_eta(c["eta"])

    def start():
        p.set_mask(None)
        p.set_rho0(c["rho0"])
        p.set_mask((0, 1))
        p.set_mask(None)

    out = _beside_other_work(p, start, steps, 20)
    p.close()
    _check(out, c, M, dkmax, 0.0, None, steps)
