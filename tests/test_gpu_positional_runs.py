"""The positional layout's runs: many steps (or QLS terms) in one launch, over the
grid or (up to 6144 slots) on one cluster, equal the same ones by single
launches, at the edges of their tables and turns; s = 4, which the autotuner alone chooses; marginals read in place."""
import numpy as np
import pytest

import oracle
from paper_2303_06890_gb300 import qwalk
from paper_2303_06890_gb300 import workloads as wl

from parity import compare, gpu_state, oracle_state

pytestmark = pytest.mark.gpu

# rows a warp, a block of 4 warps, a cluster and the card hold, and one more or less
SHAPES = [(8, 8), (9, 8), (33, 8), (127, 8), (129, 16), (70, 32), (768, 8), (95, 64), (96, 64), (97, 64), (769, 8),
          (1217, 8), (130, 64), (20001, 8)]


def _matrix(n, s):
    return wl.band_positive(n, s // 2 - 1, 15, n) if s >= 32 else wl.random_symmetric(n, s, 1, (3 * n * s) // 8, n)


def _b(n, seed, cplx=False):
    rng = np.random.default_rng(seed)
    b = rng.standard_normal(n) + (1j * rng.standard_normal(n) if cplx else 0.0)
    return b / np.linalg.norm(b)


def _positional(m, s, b, **kw):
    """A simulator on the positional layout, the state T~|b~>."""
    sim = qwalk.Sim(m, s_pad=s, walk_variant=7 if s >= 8 else 0, **kw)
    sim.state_init(b)
    if s < 8:
        v, us = sim.autotune(64)
        # kept: a bucket kernel's step takes three times as long; named: one to create with
        assert 0.0 < us[7] < us[v] and v in (0, 1, 2, 3)
        qwalk.Sim(m, s_pad=s, walk_variant=v, **kw).close()
        sim.state_init(b)
    return sim


@pytest.mark.parametrize("n,s", SHAPES)
def test_a_run_equals_single_steps(n, s):
    """Without renormalisation the arithmetic of a step does not depend on the
    launch it is in: the same bits."""
    m, b = _matrix(n, s), _b(n, 1, cplx=n % 2 == 1)
    runs, single = _positional(m, s, b), _positional(m, s, b, graphs=False)
    for steps in (1, 2, 3, 8):
        for sim in (runs, single):
            sim.enqueue_walk_steps(steps)
        (ka, va), (kb, vb) = runs.state_export(), single.state_export()
        assert np.array_equal(ka, kb) and np.array_equal(va, vb)


@pytest.mark.parametrize("n", [100, 900])
@pytest.mark.parametrize("precision,tol", [(qwalk.QW_FP64, 1e-12), (qwalk.QW_FP32_AMP, 1e-4)])
def test_a_run_over_a_launchs_length(precision, tol, n):
    """1025 steps: two launches, and (complex64) a renormalisation between any two
    steps; against the single steps, whose factor is computed another way.
    complex64: an amplitude takes a rounding of 2^-24 of itself a step from
    the factor's last bit, 1025 steps of it in the worst case 6e-5."""
    m, b = _matrix(n, 8), _b(n, 2)
    out = []
    for graphs in (True, False):
        sim = _positional(m, 8, b, precision=precision, graphs=graphs)
        sim.enqueue_walk_steps(1025)
        out.append([sim.measure_register(r, n) for r in ("j", "k")])
    for x, y in zip(*out):
        assert abs(x.sum() - 1.0) < tol and np.abs(x - y).max() < tol


@pytest.mark.parametrize("n,s", [(16, 4), (40, 4), (257, 4), (1000, 4)])
def test_s4_matches_oracle(n, s):
    m, b = _matrix(n, s), _b(n, 3)
    sim = _positional(m, s, b)
    o = oracle.Oracle(m, s)
    o.init_b(b)
    o.apply("T")
    for steps in (1, 2, 3):
        sim.enqueue_walk_steps(steps)
        for _ in range(steps):
            o.apply("W")
        for reg, length in (("j", n), ("k", n), ("b1", 2), ("b2", 2)):
            assert np.abs(sim.measure_register(reg, length) - o.marginal(reg, length)).max() < 1e-12
        compare(gpu_state(sim), oracle_state(o), 1e-12)


@pytest.mark.parametrize("n,s,terms", [(60, 4, 5), (100, 8, 1), (100, 8, 513), (140, 16, 8), (100, 64, 3),
                                       (900, 8, 3)])
def test_qls_terms_in_one_launch(n, s, terms):
    """Y and every p_j against the Chebyshev sum in numpy (1e-9 relative, the
    bound of the other QLS tests)."""
    m, b = _matrix(n, s), _b(n, 4)
    a = m.dense() / s
    coeffs = np.random.default_rng(5).standard_normal(terms) / terms
    t0, t1, y, p = b, a @ b, np.zeros(n), []
    for c in coeffs:
        y = y + c * t1
        p.append(y @ y)
        for _ in range(2):
            t0, t1 = t1, 2.0 * (a @ t1) - t0
    sim = _positional(m, s, b)
    got_y, got_p = sim.apply_qls(coeffs)
    assert np.abs(got_y - y).max() <= 1e-9 * np.linalg.norm(y)
    assert np.abs(got_p - p).max() <= 1e-9 * max(p)


def test_a_smaller_simulator_leaves_a_larger_ones_launches_alone():
    """The tables of 4000 rows take more shared memory a block than those of
    100: a plan made for the smaller matrix in between changes nothing."""
    big = _positional(_matrix(4000, 16), 16, _b(4000, 6))
    small = _positional(_matrix(100, 16), 16, _b(100, 7))
    for sim, n in ((big, 4000), (small, 100), (big, 4000)):
        sim.enqueue_walk_steps(8)
        assert abs(sim.measure_register("j", n).sum() - 1.0) < 1e-12
