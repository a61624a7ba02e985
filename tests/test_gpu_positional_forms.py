"""Forms of the positional layout's runs beside those of test_gpu_positional_runs.py:
complex64 entries, batches on the cluster and over the grid, tables that do not
fit shared memory, and solves, each against the same steps launched one at a time;
simulators on streams of their own."""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest
import torch

from paper_2303_06890_gb300 import qwalk
from paper_2303_06890_gb300 import workloads as wl

from test_gpu_positional_runs import _b, _matrix, _positional

pytestmark = pytest.mark.gpu


def _pair(make):
    """make(graphs) of a run's simulator and of one that takes single steps"""
    return make(True), make(False)


@pytest.mark.parametrize("n,s", [(9, 8), (33, 8), (129, 16), (70, 32), (97, 64), (40, 4), (1217, 8), (2500, 16), (700, 32),
                                 (130, 64), (3001, 4), (20001, 8)])
def test_a_complex64_run_equals_single_steps(n, s):
    """Without renormalisation the same bits, as in complex128."""
    m, b = _matrix(n, s), _b(n, 1, cplx=n % 2 == 1)
    runs, single = _pair(lambda g: _positional(m, s, b, precision=qwalk.QW_FP32_AMP, renorm=0, graphs=g))
    for steps in (2, 3, 8):
        for sim in (runs, single):
            sim.enqueue_walk_steps(steps)
        (ka, va), (kb, vb) = runs.state_export(), single.state_export()
        assert np.array_equal(ka, kb) and np.array_equal(va, vb)


@pytest.mark.parametrize("precision", [qwalk.QW_FP64, qwalk.QW_FP32_AMP])
@pytest.mark.parametrize("n,s", [(30000, 64)])
def test_a_run_without_tables_equals_single_steps(n, s, precision):
    """198 rows of 64 slots an SM: 20 bytes a slot are 253 KB, more than a block has."""
    m, b = _matrix(n, s), _b(n, 2)
    runs, single = _pair(lambda g: _positional(m, s, b, precision=precision, renorm=0, graphs=g))
    for steps in (2, 3):
        for sim in (runs, single):
            sim.enqueue_walk_steps(steps)
        for reg in ("j", "k"):
            assert np.array_equal(runs.measure_register(reg, n), single.measure_register(reg, n))


# uneven instances of 8 slots a row: 6144 slots in all go to one cluster, more over the grid
@pytest.mark.parametrize("ns", [(16, 100, 33, 401), (300, 17, 451), (300, 17, 452), (900, 16, 2047, 333, 64)])
@pytest.mark.parametrize("precision,renorm,tol", [(qwalk.QW_FP64, 0, 0.0), (qwalk.QW_FP32_AMP, 0, 0.0),
                                                 (qwalk.QW_FP64, 1, 1e-14), (qwalk.QW_FP32_AMP, -1, 2e-6)])
def test_a_batchs_run_equals_single_steps(ns, precision, renorm, tol):
    """The same bits without renormalisation.  With it the factor's last bit can
    differ, a rounding of an amplitude each way in each of 5 steps: 20 of 2^-53 or
    2^-24 of a bin's largest term in all."""
    mats = [_matrix(n, 8) for n in ns]

    def make(graphs):
        sim = qwalk.Sim(mats, s_pad=8, precision=precision, walk_variant=7, renorm=renorm, graphs=graphs)
        for i, n in enumerate(ns):
            sim.state_init(_b(n, i, cplx=i % 2 == 1), inst=i)
        sim.enqueue_walk_steps(5)
        return np.concatenate([sim.measure_register(r, n, inst=i) for i, n in enumerate(ns) for r in ("j", "k")])

    x, y = _pair(make)
    assert y.max() > 0.0 and np.abs(x - y).max() <= tol * y.max()


@pytest.mark.parametrize("n,s", [(60, 4), (100, 8), (700, 8), (900, 8), (140, 16), (97, 64), (2000, 16)])
def test_a_complex64_solve(n, s):
    """Y and every p_j of 8 terms against the Chebyshev sum, and Y against single
    steps without renormalisation (the same state: FP64 roundings of the
    accumulator, two a term).  Before term j's read-out an amplitude has been rounded, at
    2^-24 of itself, twice in each of 2 j + 2 operators, and the 3 n s branches
    lost at most 2^-24 each to pruning; the renormalisation at most doubles that."""
    m, b, terms = _matrix(n, s), _b(n, 4), 8
    a = m.dense() / s
    coeffs = np.random.default_rng(5).standard_normal(terms) / terms
    t0, t1, y, p = b, a @ b, np.zeros(n), []
    for c in coeffs:
        y = y + c * t1
        p.append(y @ y)
        for _ in range(2):
            t0, t1 = t1, 2.0 * (a @ t1) - t0
    err = 2.0 * (2.0 + np.sqrt(3.0 * n * s)) * 2.0**-24 * np.cumsum(np.abs(coeffs) * (2.0 * np.arange(terms) + 2.0))
    got_y, got_p = _positional(m, s, b, precision=qwalk.QW_FP32_AMP).apply_qls(coeffs)
    assert np.linalg.norm(got_y - y) <= err[-1]
    assert (np.abs(got_p - p) <= 2.0 * np.sqrt(p) * err + err**2).all()
    ys = [sim.apply_qls(coeffs)[0] for sim in
          _pair(lambda g: _positional(m, s, b, precision=qwalk.QW_FP32_AMP, renorm=0, graphs=g))]
    assert np.abs(ys[0] - ys[1]).max() <= 16 * 2.0**-53 * np.abs(coeffs).sum()


@pytest.mark.parametrize("n,s", [(300, 8), (5000, 16)])
def test_simulators_on_streams_of_their_own(n, s):
    """Two simulators on two non-blocking streams, each driven by a thread: the bits of
    the same walks one after another."""
    mats, bs = [_matrix(n, s), _matrix(n + 1, s)], [_b(n, 1), _b(n + 1, 2)]
    streams = [torch.cuda.Stream() for _ in mats]

    def walk(i):
        sim = qwalk.Sim(mats[i], s_pad=s, walk_variant=7, stream=streams[i].cuda_stream)
        out = []
        for steps in (1, 40, 41):
            sim.state_init(bs[i])
            sim.enqueue_walk_steps(steps)
            out += [sim.measure_register(r, mats[i].n) for r in ("j", "k")]
        sim.close()
        return out

    with ThreadPoolExecutor(2) as pool:
        together = list(pool.map(walk, range(2)))
    for i in range(2):
        assert all(np.array_equal(x, y) for x, y in zip(together[i], walk(i)))
