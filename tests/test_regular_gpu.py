"""The regular stream kernel (unfiltered steps) against the oracle: M = 2 and
3, every number of nonzero elements of rho(0) (the members of a group at the
first merge), windows from one point up, steps on both sides of the window's
fill, and a mask taken up or dropped in mid-run (the step counts are then no
longer known on the host)."""
import numpy as np
import pytest

import workloads as W
from oracle import iquapi

pytestmark = pytest.mark.gpu


def _rho0(M, nnz, seed):
    rng = np.random.default_rng(seed)
    r = W.random_density_matrix(rng, M)
    keep = np.zeros(M * M, dtype=bool)
    keep[[0] + list(1 + rng.permutation(M * M - 1)[:nnz - 1])] = True
    return np.where(keep.reshape(M, M), r, 0.0)


def _run(c, mask, rho0, parts, precision="fp64"):
    from paper_2506_03127_gb300 import Propagator
    p = Propagator(c["M"], c["dkmax"], c["dt"], c["q"], c["hs"], 0.0, precision, "stream", max_paths=1 << 18)
    p.set_eta(c["eta"])
    p.set_mask(mask)
    p.set_rho0(rho0)
    for n in parts:
        p.step(n)
    T = sum(parts)
    out = p.rho(0, T + 1), p.stats(1, T)
    p.close()
    return out


@pytest.mark.parametrize("M,dkmax,nnz", [(2, d, n) for d in (1, 2, 3, 6) for n in (1, 2, 3, 4)]
                         + [(3, d, n) for d in (1, 2, 4) for n in (1, 2, 5, 9)])
@pytest.mark.parametrize("precision", ["fp64", "c64"])
def test_unfiltered_steps(M, dkmax, nnz, precision):
    c = W.random_case(40 + dkmax, M, dkmax)
    rho0, T = _rho0(M, nnz, 7 * nnz + dkmax), dkmax + 4
    rho, st = _run(c, None, rho0, (1, T - 2, 1), precision)
    ref = iquapi.propagate(M, c["q"], c["hs"], c["dt"], c["eta"], dkmax, None, 0.0, rho0, T)
    # FP64: the bar of the other engine tests; complex64: 2^-24 per operation, a few tens of them per step
    assert np.abs(rho - ref.rho).max() <= (1e-10 if precision == "fp64" else 2e-6 * max(1.0, np.abs(ref.rho).max()))
    assert [(r[1], r[3]) for r in st] == [(o.groups, o.kept) for o in ref.stats]


def test_steps_in_graphs_of_several_match():
    """graph_steps > 1: runs of steps that need different kernels.  The stored
    sets are the same bit for bit; rho(t) of the tile kernel is summed by the
    blocks that drew the tiles, in any order (the engines' parity bar)."""
    from paper_2506_03127_gb300 import Propagator
    c = W.random_case(51, 2, 5)
    rho0 = _rho0(2, 1, 3)
    for mask in (None, (0, 1, 2)):
        out = []
        for gs in (1, 4):
            p = Propagator(2, 5, c["dt"], c["q"], c["hs"], 0.0, "fp64", "stream", max_paths=1 << 14)
            p.set_eta(c["eta"])
            p.set_mask(mask)
            p.set_rho0(rho0)
            p.set_tuning(graph_steps=gs)
            p.step(3)
            p.step(14)
            out.append((p.rho(0, 18), *p.export_paths()))
            p.close()
        assert np.abs(out[0][0] - out[1][0]).max() <= 1e-10
        assert np.array_equal(out[0][1], out[1][1]) and np.array_equal(out[0][2], out[1][2])


@pytest.mark.parametrize("first,then", [(None, (0, 1, 2)), ((0, 1, 2), None)])
def test_mask_changed_in_mid_run(first, then):
    from paper_2506_03127_gb300 import Propagator
    c = W.random_case(53, 2, 5)
    rho0 = _rho0(2, 4, 5)
    out = []
    for engine in ("stream", "hash"):
        p = Propagator(2, 5, c["dt"], c["q"], c["hs"], 0.0, "fp64", engine, max_paths=1 << 14)
        p.set_eta(c["eta"])
        p.set_mask(first)
        p.set_rho0(rho0)
        p.step(7)
        p.set_mask(then)
        p.step(6)
        out.append((p.rho(0, 14), [r[3] for r in p.stats(1, 13)]))
        p.close()
    assert np.abs(out[0][0] - out[1][0]).max() <= 1e-10
    assert out[0][1] == out[1][1]


def test_a_captured_stream_is_refused():
    """The host passes the step index to single steps, so a graph that replayed
    them would repeat it: qp_step refuses, and the propagation goes on after."""
    import torch
    from paper_2506_03127_gb300 import Propagator, abi
    c = W.random_case(54, 2, 5)
    rho0 = _rho0(2, 4, 5)
    p = Propagator(2, 5, c["dt"], c["q"], c["hs"], 0.0, "fp64", "stream", max_paths=1 << 14)
    p.set_eta(c["eta"])
    p.set_mask(None)
    p.set_rho0(rho0)
    p.step(8)
    p.sync()
    x, g = torch.zeros(1, device="cuda"), torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=p.stream):
        x.add_(1)
        with pytest.raises(abi.QPError):
            p.step(1)
    p.step(4)
    rho = p.rho(0, 13)
    p.close()
    ref = iquapi.propagate(2, c["q"], c["hs"], c["dt"], c["eta"], 5, None, 0.0, rho0, 12)
    assert np.abs(rho - ref.rho).max() <= 1e-10


@pytest.mark.parametrize("precision", ["fp64", "c64"])
def test_steps_of_more_chunks_than_warps(precision):
    """59 049 groups (1846 chunks of 32, the last ragged) on at most 1216 warps.
    The counts that the blocks leave with their partials add up to the step's."""
    from paper_2506_03127_gb300 import Propagator
    M, dkmax, T = 3, 6, 8
    c = W.random_case(55, M, dkmax)
    rho0 = _rho0(M, 5, 9)
    p = Propagator(M, dkmax, c["dt"], c["q"], c["hs"], 0.0, precision, "stream", max_paths=1 << 20)
    p.set_eta(c["eta"])
    p.set_mask(None)
    p.set_rho0(rho0)
    p.step(T)
    rho, st = p.rho(0, T + 1), p.stats(1, T)
    kept = [int(np.ravel(p.instance_counts(t))[0]) for t in range(1, T + 1)]
    p.close()
    ref = iquapi.propagate(M, c["q"], c["hs"], c["dt"], c["eta"], dkmax, None, 0.0, rho0, T)
    assert [(r[1], r[3]) for r in st] == [(o.groups, o.kept) for o in ref.stats]
    assert kept == [o.kept for o in ref.stats]
    assert np.abs(rho - ref.rho).max() <= (1e-10 if precision == "fp64" else 2e-6 * max(1.0, np.abs(ref.rho).max()))
