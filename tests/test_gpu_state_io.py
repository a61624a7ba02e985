"""qw_state_import / qw_state_export on the device: any order of the list, key
widths of 1, 2 and 10 words, list lengths about the sort's tile, rows longer
than the buckets, several instances, and every refusal."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qw():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2303_06890_gb300 import qwalk
    return qwalk


def _sim(qw, n=100, s=4, count=1, **kw):
    from paper_2303_06890_gb300 import workloads as wl
    mats = [wl.random_symmetric(n, s, 1, n, 3 + i) for i in range(count)]
    return qw.Sim(mats if count > 1 else mats[0], s_pad=s, **kw)


def _state(sim, m, rng, insts=1, one_row=False):
    """m branches of distinct registers in shuffled order: (registers, amplitudes)."""
    nb = sim.nb
    seen, rows = set(), []
    while len(rows) < m:
        r = (0, 5 if one_row else int(rng.integers(0, 1 << nb)), int(rng.integers(0, 2)),
             int(rng.integers(0, 1 << nb)) if one_row or rng.random() < 0.2 else 0, int(rng.integers(0, 1 << nb)),
             int(rng.integers(0, 2)), 0, int(rng.integers(0, insts)))
        if r not in seen:
            seen.add(r)
            rows.append(r)
    return np.array(rows, dtype=np.uint64), rng.standard_normal(m) + 1j * rng.standard_normal(m)


def _sorted(keys, amps):
    order = np.lexsort(keys.T)  # the last word is the most significant
    return keys[order], amps[order]


@pytest.mark.parametrize("words", [1, 2, 10])
@pytest.mark.parametrize("m", [1, 2, 31, 255, 257, 2047, 2048, 2049, 5000])
def test_round_trip_is_the_sorted_list(qw, words, m):
    sim = _sim(qw, row_capacity=512)  # nb = 7: the layout has 62 bits
    regs, amps = _state(sim, m, np.random.default_rng(m))
    keys = sim.pack(regs, words)
    want_k, want_a = _sorted(keys, amps)
    for k, a in ((keys, amps), (want_k, want_a)):  # shuffled, then as exported
        sim.state_import(k, a)
        got_k, got_a = sim.state_export(key_words=words)
        assert np.array_equal(got_k, want_k)
        assert np.array_equal(got_a, want_a)  # complex128 storage: the same bits


@pytest.mark.parametrize("length", [16, 17, 700])
def test_rows_longer_than_the_buckets_grow_them(qw, length):
    sim = _sim(qw, row_capacity=16)
    regs, amps = _state(sim, length, np.random.default_rng(length), one_row=True)
    keys = sim.pack(regs)
    sim.state_import(keys, amps)
    got_k, got_a = sim.state_export()
    want_k, want_a = _sorted(keys, amps)
    assert np.array_equal(got_k, want_k) and np.array_equal(got_a, want_a)


def test_instances_export_apart(qw):
    sim = _sim(qw, count=3)
    regs, amps = _state(sim, 600, np.random.default_rng(1), insts=3)
    keys = sim.pack(regs)
    sim.state_import(keys, amps)
    for inst in (-1, 0, 1, 2):
        pick = np.ones(len(regs), bool) if inst < 0 else regs[:, 7] == inst
        want_k, want_a = _sorted(keys[pick], amps[pick])
        got_k, got_a = sim.state_export(inst=inst)
        assert np.array_equal(got_k, want_k) and np.array_equal(got_a, want_a)


@pytest.mark.parametrize("words", [2, 10])
def test_refusals_name_the_rule_and_keep_the_state(qw, words):
    sim = _sim(qw)
    regs, amps = _state(sim, 300, np.random.default_rng(2))
    keys = sim.pack(regs, words)
    sim.state_import(keys, amps)
    before = sim.state_export()
    bits = 4 * sim.nb + 34  # 62: the bits above start in word 0

    def refused(change, what):
        bad = keys.copy()
        change(bad)
        for k in (bad, bad[np.lexsort(bad.T)]):
            with pytest.raises(qw.QwError, match=what) as e:
                sim.state_import(k, amps)
            assert e.value.code == -1
        after = sim.state_export()
        assert np.array_equal(before[0], after[0]) and np.array_equal(before[1], after[1])

    def equal(k):
        k[17] = k[211]

    def set_bit(bit):
        def change(k):
            k[100, bit // 64] |= np.uint64(1) << np.uint64(bit % 64)
        return change

    refused(equal, "duplicate key")
    refused(set_bit(bits - 32), "register A must be 0")
    refused(set_bit(bits - 16), "instance out of range")
    refused(set_bit(bits), "bits above the layout")
    refused(set_bit(64 * words - 1), "bits above the layout")

    def both(k):  # equal keys go first
        set_bit(bits)(k)
        equal(k)
    refused(both, "duplicate key")
