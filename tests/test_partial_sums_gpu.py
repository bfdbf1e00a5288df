"""Sums of the complex64 forms that are kept in FP64 (rounded once where they
are stored): where an FP64 sum is exact in any order, nothing of it may be
lost on the way."""
import math

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


def _rho_of(M, keys, amps):
    """rho from a stored set, the sums correctly rounded."""
    bs = max(1, (M - 1).bit_length())
    mask = np.uint64((1 << bs) - 1)
    a, b = (keys & mask).astype(int), ((keys >> np.uint64(bs)) & mask).astype(int)
    rho = np.zeros((M, M), dtype=complex)
    for i in range(M):
        for j in range(M):
            v = amps[(a == i) & (b == j)]
            rho[i, j] = complex(math.fsum(v.real), math.fsum(v.imag))
    return rho


@pytest.mark.parametrize("dkmax,theta,steps", [(8, 1e-9, 14), (9, 1e-10, 12)])
def test_rho_of_a_batch_of_three_level_chains(dkmax, theta, steps):
    """rho(t) against the exact sum of the stored children.  Its elements are
    below 1 and about two dozen FP64 additions lie between a child and rho (a
    warp, the tiles of a block, the blocks), each rounded by at most 2^-54 of
    either sign: 8 * 2^-54 allows for sqrt(24) of them and half as much again."""
    from paper_2506_03127_gb300 import Propagator, eta_from_bath
    c, n_inst = W.CHAIN3_STRUCTURED_DK12, 3
    p = Propagator(3, dkmax, c.dt, c.q, c.hs_array(), theta, "c64", "stream", max_paths=n_inst << 23, n_inst=n_inst)
    p.set_eta(eta_from_bath(c.bath, c.dt, dkmax))
    p.set_mask(range(5))
    p.set_rho0(c.rho0_array())
    p.step(steps)
    rho = p.rho(steps, 1)[0]
    keys, amps = p.export_paths()
    p.close()
    inst = (keys >> np.uint64(4 * dkmax)).astype(int)
    for i in range(n_inst):
        assert np.abs(rho[i] - _rho_of(3, keys[inst == i], amps[inst == i])).max() <= 8 * 2.0 ** -54


@pytest.mark.parametrize("nvib", [4, 3])
def test_rho_of_wide_keys(nvib):
    """The same for the wide keys.  Some 35 FP64 additions (a block's eight
    warps, 16 threads over the blocks, their sums) of partial sums no larger
    than rho's elements lie behind a block's own sums, each rounded by half a
    unit in the last place of either sign: twice sqrt(35) of these."""
    from paper_2506_03127_gb300 import WidePropagator, eta_from_bath
    steps = 16
    w = W.reaction_coordinate(nvib, 12, (0, 1, 2, 3, 4, 5, 6, 7, 8, 10), 1e-6, steps)
    p = WidePropagator(w.M, w.dkmax, w.dt, w.q, w.hs_array(), w.theta, "c64", max_paths=1 << 24)
    p.set_eta(eta_from_bath(w.bath, w.dt, w.dkmax))
    p.set_mask(w.mask)
    for n in (steps, steps + 1):
        p.set_rho0(w.rho0_array())
        p.step(n)
        rho = p.rho(n, 1)[0]
        keys, amps = p.export_paths()
        lo = keys[:, 0]
        newest = (lo & np.uint64(15)).astype(int), ((lo >> np.uint64(4)) & np.uint64(15)).astype(int)
        exact = np.zeros((w.M, w.M), dtype=complex)
        for i in range(w.M):
            for j in range(w.M):
                v = amps[(newest[0] == i) & (newest[1] == j)]
                exact[i, j] = complex(math.fsum(v.real), math.fsum(v.imag))
        unit = 2.0 ** (np.ceil(np.log2(np.abs(rho).max())) - 54)
        assert np.abs(rho - exact).max() <= 12 * unit
    p.close()


def test_infinite_amplitudes_of_wide_keys():
    """At the second step eta_1 = -1 multiplies the children (0, 1) of (0, 1) by
    exp(4): 54 times 0.58^2 of 6e37 is beyond FP32.  The child, and rho with
    it, is infinite, not undefined (as a plain sum would have it)."""
    from paper_2506_03127_gb300 import WidePropagator
    p = WidePropagator(2, 3, 1.0, (1.0, -1.0), np.array([[0.0, 0.7], [0.7, 0.0]]), 1e-10, "c64", max_paths=1 << 10)
    p.set_eta(np.array([0.0, -1.0, 0.0]))
    p.set_mask((0, 1, 2))
    p.set_rho0(np.array([[0.0, 6e37], [0.0, 0.0]]))
    p.step(2)
    rho = p.rho(2, 1)[0]
    p.close()
    assert np.isposinf(rho[0, 1].real) and np.isfinite(rho[0, 1].imag)
