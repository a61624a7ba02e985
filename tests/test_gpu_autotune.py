"""The autotuner's choice in a process of its own, where every launch it times is the
first of its kind: the positional layout, two to five times as fast in runs as
any other kernel at these sizes, whatever number of steps is asked for; and the
state it leaves, which the launches whose results it drops do not touch."""
import subprocess
import sys

import numpy as np
import pytest

import oracle
from paper_2303_06890_gb300 import qwalk
from paper_2303_06890_gb300 import workloads as wl

from parity import compare_union, gpu_state, oracle_state

pytestmark = pytest.mark.gpu

CHOICE = """
import numpy as np
from paper_2303_06890_gb300 import qwalk, workloads as wl
n, s = {n}, {s}
b = np.random.default_rng(1).standard_normal(n)
sim = qwalk.Sim(wl.random_symmetric(n, s, 1 if s == 8 else 0, (3 * n * s) // 8, 7), s_pad=s, precision={p}, stream=0)
sim.state_init(b / np.linalg.norm(b))
print(*sim.autotune({steps}))
"""


@pytest.mark.parametrize("steps", [1, 2, 3])
@pytest.mark.parametrize("n,s,p", [(16384, 16, qwalk.QW_FP32_AMP), (16384, 16, qwalk.QW_FP64), (1000, 8, qwalk.QW_FP64)])
def test_few_steps_in_a_fresh_process_choose_the_positional_layout(n, s, p, steps):
    out = subprocess.run([sys.executable, "-c", CHOICE.format(n=n, s=s, p=p, steps=steps)], check=True, capture_output=True,
                         text=True).stdout
    assert out.split()[0] == "7", out


@pytest.mark.parametrize("precision", [qwalk.QW_FP64, qwalk.QW_FP32_AMP])
@pytest.mark.parametrize("n,s,graphs", [(900, 8, True), (900, 8, False), (60, 4, True)])
def test_the_state_advances_by_the_steps_asked_for(n, s, graphs, precision):
    m = wl.random_symmetric(n, s, 1, n, n)
    b = np.random.default_rng(n).standard_normal(n)
    b /= np.linalg.norm(b)
    sim = qwalk.Sim(m, s_pad=s, precision=precision, graphs=graphs)
    sim.state_init(b)
    _, us = sim.autotune(2)
    steps = 2 * sum(u > 0.0 for u in us)
    assert sim.step_stats()["steps"] == steps
    sim.apply_walk_step(3)
    o = oracle.Oracle(m, s)
    o.init_b(b)
    o.apply("T", *["W"] * (steps + 3))
    compare_union(gpu_state(sim), oracle_state(o), *((1e-12, 1e-11) if precision == qwalk.QW_FP64 else (2e-6, 1e-5)))
    sim.close()
