"""The renormalisation of the positional layout's runs (over the grid, and on one
cluster) against its single steps, whose norm is an FP64 sum: for a norm many
times the target, and for targets far from 1."""
import math

import numpy as np
import pytest

from paper_2303_06890_gb300 import qwalk
from paper_2303_06890_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _matrix(n, s, seed):
    return wl.random_symmetric(n, s, 1, (3 * n * s) // 8, seed)


def _b(n, seed):
    b = np.random.default_rng(seed).standard_normal(n)
    return b / np.linalg.norm(b)


@pytest.mark.parametrize("precision,tol", [(qwalk.QW_FP64, 1e-13), (qwalk.QW_FP32_AMP, 2e-6)])
@pytest.mark.parametrize("count,n", [(64, 200), (16, 30), (3, 40)])
def test_a_batch_imported_and_one_instance_set_again(count, n, precision, tol):
    """Runs and single steps agree whatever the norm is of the target (64 instances:
    12 800 rows on the grid; the others: one cluster).  6 steps: an amplitude takes a
    rounding or two a step, of 2^-53 or 2^-24 of itself, each way."""
    mats = [_matrix(n, 8, 10 + i) for i in range(count)]
    out = []
    for graphs in (True, False):
        sim = qwalk.Sim(mats, s_pad=8, precision=precision, walk_variant=7, renorm=1, graphs=graphs)
        for i in range(count):
            sim.state_init(_b(n, i), inst=i)
        sim.apply_walk_step(2)
        sim.state_import(*sim.state_export())
        sim.state_init(_b(n, 99), inst=1)
        sim.apply_walk_step(6)
        out.append(np.concatenate([sim.measure_register("j", n, inst=i) for i in range(count)]))
        sim.close()
    assert np.isfinite(out[0]).all() and out[0].sum() > 0.0
    assert np.abs(out[0] - out[1]).max() <= tol * np.abs(out[1]).max()


@pytest.mark.parametrize("n,s", [(100, 8), (2000, 16)])
@pytest.mark.parametrize("e", [-60, -300, 200])
def test_complex128_renormalises_at_any_scale(n, s, e):
    """2^e b with the threshold scaled alike: the same bits, scaled."""
    m, b = _matrix(n, s, 1), _b(n, 2)
    out = []
    for c in (1.0, 2.0**e):
        sim = qwalk.Sim(m, s_pad=s, walk_variant=7, renorm=1, prune_tau=2.0**-43 * c)
        sim.state_init(c * b)
        sim.apply_walk_step(20)
        keys, amps = sim.state_export()
        out.append((keys, amps / c))
        sim.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("n,s", [(300, 8), (16384, 16)])
def test_complex64_renormalises_at_small_scale(n, s):
    """2^-50 b against b.  A step's norm is off by at most half the least subnormal
    (2^-150) a branch, 2^-30 of the target; 20 steps of that and of a rounding of
    2^-24 an amplitude: below 1e-5 of a bin.  Branches near the threshold,
    kept on one side only: 2^-48 each."""
    m, b = _matrix(n, s, 3), _b(n, 4)
    out = []
    for c in (1.0, 2.0**-50):
        sim = qwalk.Sim(m, s_pad=s, precision=qwalk.QW_FP32_AMP, walk_variant=7, prune_tau=2.0**-24 * c)
        sim.state_init(c * b)
        sim.apply_walk_step(20)
        out.append(sim.measure_register("j", n) / c**2)
        sim.close()
    assert np.abs(out[0] - out[1]).max() <= 1e-5 * out[0].max() and (np.abs(out[0] - out[1]) <= 1e-5 * out[0] + 1e-9).all()


@pytest.mark.parametrize("n,s", [(100, 8), (900, 8)])
@pytest.mark.parametrize("tau", [3e-5, 1e-4, 3e-4, 1e-3, 3e-3])
def test_complex128_factor_is_fp64(n, s, tau):
    """Steps whose pruning takes 1e-9 to 1e-3 of the norm: the state's norm is the
    target's again to FP64.  A bin is a sum of at most 30 squares (5 roundings
    deep), their sum 10 deep, the norm and the factor 4 roundings, squared: 2^-53 each,
    30 in all at most."""
    m = wl.random_symmetric(n, s, 1, (3 * n * s) // 8, n)
    b = _b(n, 5)
    for graphs in (True, False):
        sim = qwalk.Sim(m, s_pad=s, walk_variant=7, renorm=1, prune_tau=tau, graphs=graphs)
        sim.state_init(b)
        for steps in (3, 4, 5):
            sim.enqueue_walk_steps(steps)
            assert abs(math.fsum(sim.measure_register("j", n)) / math.fsum(b * b) - 1.0) <= 30 * 2.0**-53
        sim.close()


@pytest.mark.parametrize("variant", [7, 4])
def test_a_state_saved_and_resumed_takes_a_new_instance_as_before(variant):
    """Setting one instance of a batch again after an import leaves the same state as
    without the import in between (complex128, FP64 roundings)."""
    mats = [_matrix(n, 8, n) for n in (40, 70, 100)]
    out = []
    for resume in (True, False):
        sim = qwalk.Sim(mats, s_pad=8, walk_variant=variant, renorm=1)
        for i, m in enumerate(mats):
            sim.state_init(_b(m.n, i), inst=i)
        sim.apply_walk_step(2)
        if resume:
            sim.state_import(*sim.state_export())
        sim.state_init(3.0 * _b(70, 9), inst=1)
        sim.apply_walk_step(3)
        out.append([sim.measure_register("j", m.n, inst=i) for i, m in enumerate(mats)])
        sim.close()
    for x, y, norm in zip(*out, (1.0, 9.0, 1.0)):
        assert abs(x.sum() - norm) < 1e-12 and np.abs(x - y).max() < 1e-13
