"""Steps whose blocks raise the capacity error while others of the same kernel
are still to start: the step fails as a whole, nothing outside the workspace is
written, and the context propagates again after a restart."""
import numpy as np
import pytest

import workloads as W
from oracle import iquapi

pytestmark = pytest.mark.gpu

GUARD = 1 << 20


def _guarded(nbytes):
    """A workspace between two guards of 1 MiB, all bytes 0xA5."""
    import torch
    buf = torch.full((nbytes + 2 * GUARD + 256,), 0xA5, dtype=torch.uint8, device="cuda")
    off = GUARD + (-(buf.data_ptr() + GUARD)) % 256
    return buf, off


def _untouched(buf, off, nbytes):
    return bool((buf[:off] == 0xA5).all()) and bool((buf[off + nbytes:] == 0xA5).all())


@pytest.mark.parametrize("precision", ["fp64", "c64"])
@pytest.mark.parametrize("max_paths,max_groups", [(40000, 0), (1 << 20, 3000)])
def test_wide(max_paths, max_groups, precision):
    import torch
    from paper_2506_03127_gb300 import abi
    M, dkmax, T = 4, 5, 4
    c = W.random_case(70, M, dkmax)
    full = W.random_density_matrix(np.random.default_rng(3), M)   # 16 paths: 16^(t+1) after t steps
    pure = np.zeros((M, M))
    pure[1, 1] = 1.0                                              # 16^t after t steps
    cfg, keep = abi.make_config(M, dkmax, c["dt"], c["q"], c["hs"], 0.0,
                                abi.QP_FP64 if precision == "fp64" else abi.QP_C64, abi.QP_ENGINE_HASH, max_paths,
                                max_groups)
    stream = torch.cuda.Stream()
    nbytes = abi.qp_wide_workspace_size(cfg)
    buf, off = _guarded(nbytes)
    torch.cuda.synchronize()
    w = abi.qp_wide_create(cfg, buf.data_ptr() + off, nbytes, stream.cuda_stream)
    abi.qp_wide_set_eta(w, c["eta"])
    for _ in range(5):
        abi.qp_wide_set_rho0(w, full)
        abi.qp_wide_step(w, 6)
        with pytest.raises(abi.QPError) as e:
            abi.qp_wide_current(w)
        assert e.value.status == abi.QP_ERR_CAPACITY
        assert _untouched(buf, off, nbytes)
    abi.qp_wide_set_rho0(w, pure)
    abi.qp_wide_step(w, T - 1)
    rho = abi.qp_wide_read_rho(w, 0, T, M)
    stream.synchronize()
    abi.lib.qp_wide_destroy(w)
    ref = iquapi.propagate(M, c["q"], c["hs"], c["dt"], c["eta"], dkmax, None, 0.0, pure, T - 1)
    # FP64: the bar of the other engine tests; complex64: 2^-24 per operation, a few tens of them per step
    assert np.abs(rho - ref.rho).max() <= (1e-10 if precision == "fp64" else 2e-6 * max(1.0, np.abs(ref.rho).max()))
