"""The resident step kernel (many steps of a grid in one cooperative launch)
against the streaming kernel and the finalize kernel launched step by step.

Both run the same unit code and sum in the same order, so the states, the
moments, the history and the ledger have to be equal bit for bit, whatever
the launch boundaries: at one plane per unit and at several, with padded
rows, one and several finalize blocks, collisions and reflection, and with an
E_x that changes its sign along x and in time (the planes fetched ahead of a
step were then laid out for the other v1 neighbour)."""
import os
import threading
import time

import numpy as np
import pytest

import oracle
from oracle import ME, QE
from paper_2303_14119_gb300 import fk

from test_gpu_parity import make_pair, rel_l1, strong_physics

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fk.load()


def assert_same(a, b):
    assert np.array_equal(a.get_f(), b.get_f())
    for x, y in zip(a.moments(), b.moments()):
        assert np.array_equal(x, y)
    assert a.surface_charge() == b.surface_charge()
    assert a.ledger() == b.ledger()
    assert a.step_count() == b.step_count()
    n = a.step_count()[0] + 1
    assert np.array_equal(a.history(n), b.history(n))


# thin tiles of one plane, several planes, padded rows, one and more
# finalize blocks (128 planes each), whole-CTA tiles
SHAPES = [(2, 6, 5), (40, 48, 48), (131, 24, 30), (300, 40, 45), (128, 96, 72), (417, 117, 61),
          (9, 3, 1000), (260, 256, 256)]


@pytest.mark.parametrize("prec", [fk.FK_F64, fk.FK_F32])
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("terms", [False, True])
def test_resident_steps_equal_single_launches_bitwise(prec, shape, terms):
    pair = []
    for _ in range(2):
        g, o = make_pair(shape, prec=prec)
        f0, sigma = strong_physics(g, o, shape, seed=7, c1f=0.08)
        if terms:  # ln Lambda such that dt nu_ee is a few percent
            info = g.info()
            n_max = (f0.sum(axis=(1, 2)) * info["dv1"] * info["dv2"]).max()
            g.set_collisions(2.0, 0.03 / (info["dt"] * oracle.nu_ee(n_max, 2.0, 1.0)), True)
            g.set_reflection(0.3)
        g.set_state(f0, sigma)
        pair.append(g)
    a, b = pair
    b.set_kernel_timing(True)  # every step: the streaming kernel, then the finalize kernel
    for n in (1, 2, 131):  # 131: more than one launch
        a.step(n)
        b.step(n)
        a.sync()
        b.sync()
        assert_same(a, b)
    a.close()
    b.close()


@pytest.mark.parametrize("prec", [fk.FK_F64, fk.FK_F32])
def test_field_changing_its_sign_between_steps(prec):
    """The surface charge falls (no secondaries) until E_x at the wall turns
    over, one plane after the other: their c_1 change sign within a launch."""
    shape = (24, 40, 36)
    pair = []
    for _ in range(2):
        g, o = make_pair(shape, prec=prec)
        strong_physics(g, o, shape, seed=9)
        g.set_see(0.0, 400.0, 1.0, 2.0, False)
        f0 = np.full(shape, 1e5)
        g.set_f(f0)
        # in units of E_x's fall over one plane: E_x = 2 - (k + 1/2) at the start
        g.set_surface_charge(4 * QE * g.info()["dx"] * g.moments()[0][0])
        pair.append(g)
    a, b = pair
    b.set_kernel_timing(True)
    a.step(120)
    b.step(120)
    a.sync()
    b.sync()
    ex = a.history(121)[:, 7]
    assert ex[0] > 0 > ex[-1]
    assert_same(a, b)
    a.close()
    b.close()


@pytest.mark.parametrize("prec", [fk.FK_F64, fk.FK_F32])
@pytest.mark.parametrize("shape", [(64, 24, 20), (200, 96, 72)])
def test_wait_that_runs_out_ends_the_launch(prec, shape):
    """The first item's copy withheld: every unit and finalize CTA leaves,
    the state stays, and the GPU steps on afterwards."""
    os.environ["FK_TEST_WAIT_CYCLES"] = "2000000"  # about 1 ms
    os.environ["FK_TEST_WITHHOLD_COPY"] = "0"
    try:
        g, o = make_pair(shape, prec=prec)
    finally:
        del os.environ["FK_TEST_WAIT_CYCLES"]
        del os.environ["FK_TEST_WITHHOLD_COPY"]
    f0, sigma = strong_physics(g, o, shape, seed=31, c1f=0.05)
    g.set_state(f0, sigma)
    start = g.get_f()
    assert fk.fk_step_status(g.h, 40) == fk.FK_OK  # enqueued
    assert fk.fk_sync_status(g.h) == fk.FK_ETIMEOUT
    out = np.empty(shape)
    with pytest.raises(fk.FkError):
        g.get_f(out)
    assert np.array_equal(out, start)
    g.close()
    g, o = make_pair(shape, prec=prec)
    f0, sigma = strong_physics(g, o, shape, seed=31, c1f=0.05)
    g.set_state(f0, sigma)
    o.set_state(g.get_f(), sigma)
    g.step(2)
    o.step(2)
    assert rel_l1(g.get_f(), o.get_f()) <= (2e-12 if prec == fk.FK_F64 else 6e-7)
    g.close()


@pytest.mark.parametrize("prec", [fk.FK_F64, fk.FK_F32])
def test_courant_bound_freezes_at_the_same_step(prec):
    """A field that grows past the Courant bound during a launch: both forms
    stop at the same state."""
    shape = (60, 32, 28)
    pair = []
    for _ in range(2):
        g, o = make_pair(shape, prec=prec)
        f0, sigma = strong_physics(g, o, shape, seed=11)
        g.set_source(5e11, 0.0, 1.0, 300.0)  # charges the gap until |c_1| is too large
        g.set_state(f0, sigma)
        pair.append(g)
    a, b = pair
    b.set_kernel_timing(True)
    for g in pair:
        g.step(400)
        assert fk.fk_sync_status(g.h) == fk.FK_ECFL
    fa, fb = np.empty(shape), np.empty(shape)
    for g, f in ((a, fa), (b, fb)):
        with pytest.raises(fk.FkError):
            g.get_f(f)
    assert np.array_equal(fa, fb)
    for g in pair:
        g.close()


@pytest.mark.parametrize("shape", [(60, 32, 28), (300, 32, 28), (417, 96, 72)])
def test_flag_raised_by_a_unit_during_a_launch(shape):
    """A value below zero reaches the wall in step 38 of a launch: the unit that
    sees it raises the flag, every finalize CTA leaves before that step, and
    the state is that of step 37, as with single launches.  (Courant numbers
    that sum to 1 + 5e-13, within the bound, give the fastest row a weight of
    -5e-13 for its own value: what left plane 37 arrives with weights c_x^37,
    and a step later with the negative one.)"""
    nx, nv1, nv2 = shape
    far, states = 37, []
    for form in ("launches of many steps", "single launches", "the steps before"):
        g = fk.Grid(nx, nv1, nv2, 20e-6, -6e7, 6e7, -3e7, 3e7, cfl=0.5, precision=fk.FK_F64)
        info = g.info()
        c2 = 1.0 - 0.5 * (1.0 - 1.0 / nv1) + 5e-13
        g.set_fields(-c2 * info["dv2"] / info["dt"] * ME / QE, False, 0.0)
        f0 = np.zeros(shape)
        f0[far, 0, 3] = 1.0
        g.set_f(f0)
        if form == "single launches":
            g.set_kernel_timing(True)
        g.step(far if form == "the steps before" else 100)
        ok = form == "the steps before"
        assert fk.fk_sync_status(g.h) == (fk.FK_OK if ok else fk.FK_ENEGATIVE)
        f = np.empty(shape)
        if ok:
            g.get_f(f)
        else:
            with pytest.raises(fk.FkError):
                g.get_f(f)
        states.append(f)
        g.close()
    assert states[2][0, 0, 3] > 0
    assert np.array_equal(states[0], states[1])
    assert np.array_equal(states[0], states[2])


def lower_fields_and_go_on(pair, shape):
    """Fields within the bound clear the error; both forms step on alike."""
    for g in pair:
        g.set_fields(0.0, False, 0.0)
        assert fk.fk_sync_status(g.h) == fk.FK_OK
        g.step(20)
        g.sync()
    assert_same(*pair)


@pytest.mark.parametrize("prec", [fk.FK_F64, fk.FK_F32])
@pytest.mark.parametrize("nx", [131, 300, 417])
@pytest.mark.parametrize("where", ["first block", "last block"])
def test_courant_stop_found_by_one_finalize_block(prec, nx, where):
    """|c_1| grows past the bound in one block's planes only, at the wall (the
    surface charges) or in the last plane (the space charge of a source there
    grows): the other finalize CTAs stop with it at once, the status is the
    Courant one, and lower fields bring the grid back."""
    shape, h = (nx, 32, 28), 20e-6
    pair = []
    for _ in range(2):
        g, o = make_pair(shape, prec=prec)
        f0, sigma = strong_physics(g, o, shape, seed=11)
        if where == "first block":
            g.set_see(9.0, 400.0, 1.0, 400.0)
            sigma *= 2.0
        else:
            g.set_source(1e13 * (nx / 300) ** 2, 0.9 * h, h, 300.0)
            f0[:], sigma = 0.0, 0.0
        g.set_state(f0, sigma)
        pair.append(g)
    a, b = pair
    b.set_kernel_timing(True)
    states = []
    for g in pair:
        g.step(100)
        t = time.perf_counter()
        assert fk.fk_sync_status(g.h) == fk.FK_ECFL
        assert time.perf_counter() - t < 0.5  # no wait ran out
        f = np.empty(shape)
        with pytest.raises(fk.FkError):
            g.get_f(f)
        states.append(f)
    assert np.array_equal(*states)
    lower_fields_and_go_on(pair, shape)
    ex = a.history(200)[:, 7]
    assert 30 < len(ex) - 21 < 70  # the step of the stop, by the oracle 39 to 55
    for g in pair:
        g.close()


@pytest.mark.parametrize("prec", [fk.FK_F64, fk.FK_F32])
@pytest.mark.parametrize("nx", [60, 131, 417])
def test_non_finite_stop_of_several_finalize_blocks(prec, nx):
    """A plane whose sum overflows in the step's partial sums (FP32 sums of FP32
    grids; FP64 grids take values below 2^128): block 0 finds it, and every
    finalize CTA leaves with the non-finite status, not a timeout."""
    shape = (nx, 32, 28)
    f0 = np.zeros(shape)
    f0[nx // 2, :, ::4] = 1e38 if prec == fk.FK_F32 else 1e40
    states = []
    for single in (False, True):
        g = make_pair(shape, prec=prec)[0]
        g.set_fields(-1e5, False, 0.0)
        g.set_f(f0)
        assert fk.fk_sync_status(g.h) == fk.FK_OK
        g.set_kernel_timing(single)
        g.step(40)
        t = time.perf_counter()
        assert fk.fk_sync_status(g.h) == fk.FK_ENUMERIC
        assert time.perf_counter() - t < 0.5
        f = np.empty(shape)
        with pytest.raises(fk.FkError):
            g.get_f(f)
        states.append(f)
        g.close()
    assert np.array_equal(*states)


@pytest.mark.parametrize("prec", [fk.FK_F64, fk.FK_F32])
@pytest.mark.parametrize("nx", [129, 4096, 4225, 8192])
def test_exchange_of_many_finalize_blocks(prec, nx):
    """2, 32, 34 and 64 finalize CTAs, over launches of 1 to 5 and 128 steps (the
    rows of the exchange in every order): the ledger, whose velocity-edge loss
    goes through it after the step, and all the rest equal single launches."""
    shape = (nx, 6, 8)
    pair = []
    for _ in range(2):
        g, o = make_pair(shape, prec=prec)
        f0, sigma = strong_physics(g, o, shape, seed=nx, c1f=0.08)
        g.set_state(f0, sigma)
        pair.append(g)
    a, b = pair
    b.set_kernel_timing(True)
    for n in (1, 2, 3, 4, 5, 128):
        a.step(n)
        b.step(n)
    a.sync()
    b.sync()
    assert a.ledger()["lv"] > 0
    assert_same(a, b)
    a.close()
    b.close()


def stepped_alone(shapes, precs, steps):
    out = []
    for shape, prec in zip(shapes, precs):
        g, o = make_pair(shape, prec=prec)
        f0, sigma = strong_physics(g, o, shape, seed=5, c1f=0.08)
        g.set_state(f0, sigma)
        g.step(steps)
        g.sync()
        out.append(g)
    return out


def test_grids_on_their_own_streams_from_several_threads():
    """Grids of several sizes, each on its own stream and thread, some of them
    beside a batch: whichever form their steps take meanwhile, the states are
    those of each grid stepped alone."""
    shapes = [(321, 117, 61), (64, 48, 48), (200, 96, 72), (300, 40, 45), (64, 48, 48)]
    precs = [fk.FK_F32, fk.FK_F64, fk.FK_F32, fk.FK_F64, fk.FK_F32]
    alone = stepped_alone(shapes, precs, 300)
    grids = stepped_alone(shapes, precs, 0)
    members = stepped_alone([(128, 64, 64)] * 2, [fk.FK_F32] * 2, 0)
    errors = []

    def work(step, sync):
        try:
            for n in (1, 33, 130, 7, 64, 65):  # 300 in all
                step(n)
                sync()
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    with fk.Batch(members) as b:
        threads = [threading.Thread(target=work, args=(x.step, x.sync)) for x in grids + [b]]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
    assert not errors
    for a, g in zip(alone, grids):
        assert_same(a, g)
    for g in alone + grids + members:
        g.close()


def test_grids_on_their_own_streams_share_the_gpu():
    """Four grids that do not fill the GPU's time alone (their steps are bound by
    latency) take less together than one after the other: resident launches,
    which would take turns, give way.  The bound is far from both sides (0.97 of
    the sum when they take turns, about 0.5 side by side)."""
    shape = (321, 117, 117)
    grids = stepped_alone([shape] * 4, [fk.FK_F32] * 4, 0)
    for g in grids:
        g.set_fields(-1e5, False, 0.0)  # the Courant numbers stay what they are
        g.step(64)
        g.sync()

    def best(run):
        times = []
        for _ in range(6):
            t = time.perf_counter()
            run()
            times.append(time.perf_counter() - t)
        return min(times)

    def in_turn():
        for g in grids:
            g.step(256)
            g.sync()

    def together():
        for g in grids:
            g.step(256)
        for g in grids:
            g.sync()

    apart = best(in_turn)
    assert best(together) < 0.75 * apart
    # and back: one after the other again, in the resident form
    assert best(in_turn) < 1.2 * apart
    for g in grids:
        g.close()
