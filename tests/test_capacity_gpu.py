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


@pytest.mark.parametrize("engine,scheme,n_inst,mode", [
    ("hash", "pre", 1, "graph"), ("hash", "pre", 1, "persistent"), ("hash", "pre", 3, "graph"),
    ("stream", "pre", 1, "graph"), ("stream", "pre", 3, "graph"), ("stream", "pre", 3, "persistent"),
    ("hash", "post", 1, "graph")])
@pytest.mark.parametrize("precision", ["fp64", "c64"])
def test_engines(engine, scheme, n_inst, mode, precision):
    """A filter that keeps (nearly) every child: tile kernels, tables, the sort."""
    import torch
    from paper_2506_03127_gb300 import abi
    M, dkmax, theta, T = 2, 12, 1e-12, 6
    c = W.random_case(71, M, dkmax)
    pure = np.array([[0.0, 0.0], [0.0, 1.0]])
    cfg, keep = abi.make_config(M, dkmax, c["dt"], c["q"], c["hs"], theta,
                                abi.QP_FP64 if precision == "fp64" else abi.QP_C64,
                                abi.QP_ENGINE_HASH if engine == "hash" else abi.QP_ENGINE_STREAM, n_inst * 300000, 0,
                                n_inst=n_inst, scheme=abi.QP_PREMERGE if scheme == "pre" else abi.QP_POSTMERGE)
    stream = torch.cuda.Stream()
    nbytes = abi.qp_workspace_size(cfg)
    buf, off = _guarded(nbytes)
    torch.cuda.synchronize()
    p = abi.qp_create(cfg, buf.data_ptr() + off, nbytes, stream.cuda_stream)
    abi.qp_set_eta(p, c["eta"])
    abi.qp_set_mask(p, (0, 1, 2))
    tune = abi.qp_get_tuning(p)
    if mode == "persistent":
        tune.mode = abi.QP_LAUNCH_PERSISTENT
        abi.qp_set_tuning(p, tune)
    for _ in range(5):
        abi.qp_set_rho0(p, c["rho0"])
        abi.qp_step(p, 11)                       # up to 4^12 paths per instance
        with pytest.raises(abi.QPError) as e:
            abi.qp_sync(p)
        assert e.value.status == abi.QP_ERR_CAPACITY
        assert _untouched(buf, off, nbytes)
    abi.qp_set_rho0(p, pure)
    abi.qp_step(p, T)
    rho = abi.qp_read_rho(p, 0, T + 1, M, n_inst).reshape(T + 1, n_inst, M, M)
    stream.synchronize()
    abi.qp_destroy(p)
    ref = iquapi.propagate(M, c["q"], c["hs"], c["dt"], c["eta"], dkmax, (0, 1, 2), theta, pure, T)
    bar = 1e-10 if precision == "fp64" else 2e-6 * max(1.0, np.abs(ref.rho).max())
    assert np.abs(rho - ref.rho[:, None]).max() <= bar
