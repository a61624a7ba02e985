"""Host side of the C ABI (`qw_api.cpp`) without a GPU: compiled here with the host
C++ compiler against a CUDA runtime and kernel launchers that run on the host
(`fake_cuda/fake_cuda.cpp`), for what a sound device does not show: the autotuner's
choice under given kernel times, and the state of the simulator after a wait
on the device that gave up, an allocation that failed, a refused call."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2303_06890_gb300 import build as native
from paper_2303_06890_gb300 import qwalk
from paper_2303_06890_gb300 import workloads as wl

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2303_06890_gb300", "csrc")
MODE = {0: 0, 1: 3, 2: 4, 3: 5, 4: 6}  # walk_variant -> kernel mode (qw_internal.h)
ROW_OVERFLOW, POS_UNREP, POS_FULL = 1, 64, 256  # device status bits


@pytest.fixture(scope="module")
def fake_path(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    cuda = os.path.join(os.path.dirname(os.path.dirname(native.nvcc())), "include")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    so = str(tmp_path_factory.mktemp("hostapi") / "libfake.so")
    subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", cuda, "-I", CSRC, "-o", so,
                    os.path.join(HERE, "fake_cuda", "fake_cuda.cpp"), os.path.join(CSRC, "qw_api.cpp")], check=True)
    return so


@pytest.fixture
def fake(fake_path, monkeypatch):
    monkeypatch.setattr(native, "LIB", fake_path)
    monkeypatch.setattr(qwalk, "_lib", None)
    lib = qwalk.load(build_if_missing=False)
    for name in ("fake_live", "fake_sync_copies", "fake_map_most", "fake_tinits", "fake_run_steps", "fake_overruns",
                 "fake_pinned_most", "fake_unordered"):
        getattr(lib, name).restype = ctypes.c_int64
    lib.fake_word.restype = lib.fake_epoch.restype = ctypes.c_ulonglong
    lib.fake_target.restype = ctypes.c_double
    lib.fake_room.argtypes = lib.fake_listed.argtypes = [ctypes.c_int64]
    lib.fake_listed.restype = ctypes.c_uint64
    lib.fake_set_step.argtypes = [ctypes.c_int, ctypes.c_double]
    lib.fake_set_times.argtypes = [ctypes.c_double] * 4
    lib.fake_reset()
    yield lib
    lib.fake_reset()


def _b(n):
    b = np.random.default_rng(n).standard_normal(n)
    return b / np.linalg.norm(b)


def _sim(n=64, s=8, **kw):
    return qwalk.Sim(wl.random_symmetric(n, s, 1, n, n), s_pad=s, **kw)


@pytest.mark.parametrize("steps", [1, 2, 3, 8])
@pytest.mark.parametrize("graphs", [True, False])
@pytest.mark.parametrize("slot,run,choice", [(20.0, 8.5, 7), (10.0, 3.5, 7), (6.0, 8.5, 4)])
def test_autotuner_times_steps_not_first_launches(fake, steps, graphs, slot, run, choice):
    """The fastest kernel a step is chosen whatever number of steps is asked for,
    though each kind's first launch takes 60 us more, and a run 15 us beside
    its steps; the state advances by the steps asked for, no more."""
    for v, us in ((0, 40.0), (1, 38.0), (2, 45.0), (3, 44.0), (4, slot)):
        fake.fake_set_step(MODE[v], us)
    fake.fake_set_times(run, run, 15.0 if graphs else 0.0, 60.0)
    with _sim(graphs=graphs) as sim:
        sim.state_init(_b(64))
        v, us = sim.autotune(steps)
        assert v == choice
        assert sim.step_stats()["steps"] == steps  # (the fake counts them for the positional layout)
        tried = sum(u > 0.0 for u in us)
        assert tried == 6 and abs(us[7] - run) <= (15.0 / 32 if graphs else 1e-6) + 1e-6


def test_a_batch_imported_and_one_instance_set_again_keeps_the_target(fake):
    """The renormalisation target is the sum of the instances' norms: of the imported
    list's, and, where one instance is set again, of its new one and the
    others' (which went out of it: the batch was then scaled to one instance's norm)."""
    with qwalk.Sim([wl.random_symmetric(16, 8, 1, 16, i) for i in range(3)], s_pad=8, renorm=1) as sim:
        regs = np.zeros((6, 8), dtype=np.uint64)
        regs[:, 7] = [0, 0, 1, 2, 2, 2]  # inst
        regs[:, 1] = [1, 2, 1, 1, 2, 3]  # j
        amps = np.array([1.0, 2.0j, 3.0, 1.0, 1.0, 1.0 + 1.0j])
        sim.state_import(sim.pack(regs), amps)
        sim.enqueue_walk_steps(1)
        assert fake.fake_target() == 5.0 + 9.0 + 4.0
        sim.state_init(np.full(16, 0.5), inst=1)
        sim.enqueue_walk_steps(1)
        assert fake.fake_target() == 5.0 + 4.0 + 4.0


def test_an_import_that_overflows_after_positional_steps_is_a_capacity_error(fake):
    """The overflow is the import's, not that of the steps enqueued before it (whose
    errors lose the state)."""
    with _sim(walk_variant=7, overflow_fallback=False) as sim:
        sim.state_init(_b(64))
        sim.enqueue_walk_steps(2)
        fake.fake_status(ROW_OVERFLOW)
        regs = np.zeros((1, 8), dtype=np.uint64)
        with pytest.raises(qwalk.QwError) as e:
            sim.state_import(sim.pack(regs), np.ones(1))
        assert e.value.code == qwalk.QW_ERR_CAPACITY


def test_a_bucket_step_that_overflows_in_the_autotuner_is_a_capacity_error(fake):
    """Nor that of the positional steps issued before the call; the state is kept."""
    with _sim(walk_variant=7, overflow_fallback=False) as sim:
        sim.state_init(_b(64))
        sim.enqueue_walk_steps(2)
        fake.fake_status(ROW_OVERFLOW)
        with pytest.raises(qwalk.QwError) as e:
            sim.autotune(2)
        assert e.value.code == qwalk.QW_ERR_CAPACITY
        sim.apply_walk_step(1)


@pytest.mark.parametrize("how", ["init", "init without T", "import", "read", "sync"])
def test_a_run_starts_on_clear_barrier_words_after_one_that_gave_up(fake, how):
    """A launch that gives up its wait leaves words that some blocks arrived at.  They
    are cleared with the status, whether somebody reads it or the state is replaced."""
    with _sim(walk_variant=7) as sim:
        sim.state_init(_b(64))
        fake.fake_give_up(1)
        sim.enqueue_walk_steps(2)
        if how in ("read", "sync"):
            with pytest.raises(qwalk.QwError, match="gave up waiting.*the state is lost") as e:
                sim.measure_register("j", 64) if how == "read" else sim.sync()
            assert e.value.code == qwalk.QW_ERR_DEVICE_STATUS
        if how == "import":
            sim.state_import(sim.pack(np.zeros((1, 8), dtype=np.uint64)), np.ones(1))
        else:
            sim.state_init(_b(64), apply_T=how != "init without T")
        sim.enqueue_walk_steps(2)
        assert [fake.fake_word(i) for i in range(8)] == [0] * 8
        sim.sync()


def test_a_refused_launch_takes_no_turn_of_the_barrier(fake):
    """The words of a run's turns are left clear for it by the runs before: a run that
    was not launched has not passed its turns on."""
    with _sim(walk_variant=7) as sim:
        sim.state_init(_b(64))
        sim.enqueue_walk_steps(3)
        first = fake.fake_epoch()
        fake.fake_refuse(1)
        with pytest.raises(qwalk.QwError) as e:
            sim.enqueue_walk_steps(2)
        assert e.value.code == qwalk.QW_ERR_CUDA
        sim.enqueue_walk_steps(2)
        assert fake.fake_epoch() == first + 3
        sim.sync()
        assert sim.step_stats()["steps"] == 5


@pytest.mark.parametrize("variant", [5, 6])
@pytest.mark.parametrize("nth", range(1, 7))
def test_a_flat_stage_that_gave_up_its_wait_leaves_its_list(fake, variant, nth):
    """What such a stage has written has holes that hold no keys, whose instance and row
    would be looked up: no later kernel is given them (the lists here have 1000
    entries throughout).  The step is reported, the state kept."""
    with _sim(walk_variant=variant) as sim:
        sim.state_init(_b(64))
        fake.fake_flat_wait(nth)
        with pytest.raises(qwalk.QwError, match="gave up waiting.*state kept after 0 clean steps") as e:
            sim.apply_walk_step(1)
        assert e.value.code == qwalk.QW_ERR_DEVICE_STATUS
        assert fake.fake_map_most() == 1000
        sim.apply_walk_step(1)


@pytest.mark.parametrize("after", range(7))
def test_autotuner_at_s4_without_room_for_the_positional_layout(fake, after):
    """Device memory that is out while the layout is built, at its first allocation up
    to its last, leaves the choice among the other kernels, and nothing allocated."""
    for v in (0, 1, 2, 3):
        fake.fake_set_step(MODE[v], 20.0 + v)
    fake.fake_set_times(2.0, 2.0, 0.0, 0.0)
    with _sim(40, 4) as sim:
        sim.state_init(_b(40))
        live = fake.fake_live()
        for _ in range(2):
            fake.fake_fail_malloc(after)
            v, us = sim.autotune(2)
            assert v == 0 and us[7] == 0.0 and fake.fake_live() == live
        sim.apply_walk_step(3)
        fake.fake_fail_malloc(-1)
        assert sim.autotune(2)[1][7] > 0.0


def test_autotuner_at_s4_leaves_a_callers_row_capacity_alone(fake):
    fake.fake_set_times(2.0, 2.0, 0.0, 0.0)
    for v in (0, 1, 2, 3):
        fake.fake_set_step(MODE[v], 20.0 + v)
    with _sim(40, 4, row_capacity=8, overflow_fallback=False) as sim:
        sim.state_init(_b(40))
        live = fake.fake_live()
        assert sim.autotune(2)[0] == 0 and fake.fake_live() == live


@pytest.mark.parametrize("after", range(6))
def test_row_buckets_that_could_not_grow_stay_as_they_were(fake, after):
    """T~ needs rows of 16; the device memory is out at one of the six arrays."""
    with _sim(row_capacity=8) as sim:
        sim.state_init(_b(64), apply_T=False)
        live = fake.fake_live()
        fake.fake_fail_malloc(after)
        with pytest.raises(qwalk.QwError) as e:
            sim.state_init(_b(64))
        assert e.value.code == qwalk.QW_ERR_CUDA and fake.fake_live() == live
        fake.fake_fail_malloc(-1)
        sim.state_init(_b(64), apply_T=False)
        assert fake.fake_overruns() == 0
        sim.state_init(_b(64))
        assert fake.fake_overruns() == 0 and fake.fake_live() == live


@pytest.mark.parametrize("bits", [POS_FULL, POS_UNREP])
def test_the_status_of_a_move_is_cleared_on_the_simulators_stream(fake, bits):
    """A synchronous copy is ordered on the default stream alone, and may still be
    under way when it returns: a step on a non-blocking stream would see the bit and
    do nothing."""
    with _sim(walk_variant=7) as sim:
        sim.state_import(sim.pack(np.zeros((1, 8), dtype=np.uint64)), np.ones(1))
        copies = fake.fake_sync_copies()
        fake.fake_status(bits)
        sim.enqueue_walk_steps(2)
        assert fake.fake_sync_copies() == copies
        sim.sync()


def test_a_state_refused_under_capture_is_not_there(fake):
    """T~|b~> straight into the layout cannot be captured; refused, it leaves nothing
    launched and the simulator without the state it never got."""
    with _sim(walk_variant=7) as sim:
        fake.fake_capture(1)
        with pytest.raises(qwalk.QwError) as e:
            sim.state_init(_b(64))
        assert e.value.code == qwalk.QW_ERR_CUDA and fake.fake_tinits() == 0
        fake.fake_capture(0)
        with pytest.raises(qwalk.QwError) as e:
            sim.measure_register("j", 64)
        assert e.value.code == qwalk.QW_ERR_STATE


@pytest.mark.parametrize("words", [2, 4])
@pytest.mark.parametrize("room", [32, 48, 64, 72])
def test_a_list_is_exported_where_only_itself_fits_the_device(fake, room, words):
    """32 bytes a branch beside the state have always been enough (1000 branches, keys
    from the highest down as the fake gathers them)."""
    with _sim() as sim:
        sim.state_init(_b(64))
        live = fake.fake_live()
        fake.fake_room(1000 * room + 64)
        keys, amps = sim.state_export(key_words=words)
        assert np.array_equal(keys[:, 1] * 7 + keys[:, 0], np.arange(1000)) and not keys[:, 2:].any()
        assert np.array_equal(amps, np.arange(1000) * (1.0 + 2.0j))
        sim.state_init(_b(64))  # no error is left behind
        assert fake.fake_live() == live


@pytest.mark.parametrize("words", [2, 4])
@pytest.mark.parametrize("room", [32, 40, 47])
def test_a_list_is_imported_where_only_itself_fits_the_device(fake, room, words):
    """So too for an import, in any order of its keys; a list that is refused is
    refused for the same reason, and one that does not fit at all leaves no error."""
    with _sim() as sim:
        sim.state_init(_b(64))
        live = fake.fake_live()
        regs = np.zeros((1000, 8), dtype=np.uint64)
        v = np.random.default_rng(3).permutation(1000).astype(np.uint64)
        regs[:, 0], regs[:, 4], regs[:, 5] = v // 32, v // 2 % 16, v % 2  # jc, k, b2
        keys, amps = sim.pack(regs, words), v.astype(float)
        fake.fake_room(1000 * room + 64)
        sim.state_import(keys, amps)
        order = np.lexsort(keys.T)
        for i in (0, 1, 500, 998, 999):
            assert [fake.fake_listed(2 * i), fake.fake_listed(2 * i + 1)] == [int(x) for x in keys[order[i], :2]]
            assert fake.fake_listed(2000 + i) == int(v[order[i]])
        twice, beyond = keys.copy(), keys.copy()
        twice[7] = twice[600]
        beyond[9, -1] |= np.uint64(1 << 63)
        regs[11, 6] = 1  # register A
        for bad, why in ((twice, "duplicate"), (beyond, "above the layout"), (sim.pack(regs, words), "register A")):
            with pytest.raises(qwalk.QwError, match=why) as e:
                sim.state_import(bad, amps)
            assert e.value.code == qwalk.QW_ERR_ARG
        fake.fake_room(1000 * 16)
        with pytest.raises(qwalk.QwError) as e:
            sim.state_import(keys, amps)
        assert e.value.code == qwalk.QW_ERR_CUDA
        sim.state_init(_b(64))
        assert fake.fake_live() == live


def test_an_import_grows_the_rows_before_its_list_takes_the_memory(fake):
    """Row buckets that fit the device, but not beside the scratch of the checks there."""
    with _sim(row_capacity=8) as sim:
        sim.state_init(_b(64), apply_T=False)
        regs = np.zeros((100, 8), dtype=np.uint64)
        regs[:, 3], regs[:, 4] = np.arange(100) % 50, np.arange(100) // 50  # kc, k: one row
        fake.fake_longest(100)
        rows = 3 * 24 * (128 + 256) * 128  # total_buckets, 128 branches a row
        fake.fake_room(rows + 4000)  # the scratch there: 4832 bytes
        sim.state_import(sim.pack(regs), np.ones(100))
        assert fake.fake_overruns() == 0


def test_a_marginal_of_any_length_takes_bounded_pinned_memory(fake):
    """Bins beyond the register's are zeros that the caller asked for; the pinned memory
    that a simulator keeps does not grow with them."""
    with _sim(walk_variant=7) as sim:
        sim.state_init(_b(64))
        for length in (65536, 65537, 1 << 20):
            assert sim.measure_register("j", length).sum() == length  # (the fake writes 1 to each bin)
        assert fake.fake_pinned_most() == 65536 * 8


@pytest.mark.parametrize("kw,tune", [(dict(walk_variant=7), False), (dict(), True)])
def test_the_layouts_tables_are_there_before_the_simulators_stream_goes_on(fake, kw, tune):
    """They are written through the default stream, which another, non-blocking one does
    not wait for; the barrier words of a run among them."""
    with _sim(stream=64, **kw) as sim:
        sim.state_init(_b(64))
        if tune:
            sim.autotune(2)
        sim.state_init(_b(64))
        sim.apply_walk_step(3)
        assert fake.fake_unordered() == 0
