"""Split steps (Lie and Strang) in one march against the FP64 oracle, every
term on, at the sizes where the march can go wrong: one plane per chunk, few
planes, padded rows, rows that leave a tile of two or three, several tiles of
either sign, and rows too wide for it (the steps then run as passes).

Bounds: one step's rounding of FP64 and FP32, those of the tests of the
passes; sums over a plane take the same."""
import time

import numpy as np
import pytest

from paper_2303_14119_gb300 import fk

from test_gpu_strang import rel_l1, setup

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fk.load()


SHAPES = [(2, 12, 10), (3, 40, 33), (5, 8, 1000), (4, 6, 1365), (40, 256, 64), (23, 130, 71),
          (160, 10, 9), (7, 6, 3000)]


@pytest.mark.parametrize("scheme", [fk.FK_SCHEME_LIE, fk.FK_SCHEME_STRANG])
@pytest.mark.parametrize("prec,tol", [(fk.FK_F64, 1e-12), (fk.FK_F32, 5e-7)])
@pytest.mark.parametrize("shape", SHAPES)
def test_split_steps_match_the_oracle(shape, prec, tol, scheme):
    g, o = setup(shape, prec, 91, scheme=scheme)
    for _ in range(3):
        o.set_state(g.get_f(), g.surface_charge())
        g.step(1)
        o.step(1)
        assert rel_l1(g.get_f(), o.get_f()) <= tol
        n, ex, gpe, gsee = g.moments()
        no, exo, gpeo, gseeo = o.moments()
        assert rel_l1(n, no) <= tol
        assert abs(n[0] - no[0]) <= 10 * tol * no[0]  # the plane completed after the march
        assert abs(gpe - gpeo) <= 10 * tol * gpeo and abs(gsee - gseeo) <= 10 * tol * gseeo
        assert abs(g.surface_charge() - o.surface_charge()) <= tol * abs(o.surface_charge())
    g.close()


@pytest.mark.parametrize("scheme", [fk.FK_SCHEME_LIE, fk.FK_SCHEME_STRANG])
@pytest.mark.parametrize("item", [0, 2])
def test_withheld_copy_times_out_and_the_state_stays(scheme, item, monkeypatch):
    monkeypatch.setenv("FK_TEST_WAIT_CYCLES", "2000000")  # about 1 ms
    monkeypatch.setenv("FK_TEST_WITHHOLD_COPY", str(item))
    shape = (1200, 24, 20)  # several planes per chunk
    g, _ = setup(shape, fk.FK_F32, 92, scheme=scheme)
    start = g.get_f()
    assert fk.fk_step_status(g.h, 3) == fk.FK_OK  # enqueued
    assert fk.fk_sync_status(g.h) == fk.FK_ETIMEOUT
    out = np.empty(shape)
    with pytest.raises(fk.FkError):
        g.get_f(out)
    assert np.array_equal(out, start)
    g.close()


# either side of the line between one march and the passes: tiles of two rows,
# thin grids of a few and of many planes per chunk
@pytest.mark.parametrize("scheme", [fk.FK_SCHEME_LIE, fk.FK_SCHEME_STRANG])
@pytest.mark.parametrize("prec,tol", [(fk.FK_F64, 1e-12), (fk.FK_F32, 5e-7)])
@pytest.mark.parametrize("shape", [(40, 8, 1800), (300, 6, 1800), (100, 8, 1000), (1030, 8, 8), (2100, 8, 8),
                                   (2100, 24, 10), (2500, 30, 32)])
def test_split_steps_on_either_side_of_the_march_rule(shape, prec, tol, scheme):
    test_split_steps_match_the_oracle(shape, prec, tol, scheme)


def test_long_chains_of_little_work_run_as_passes():
    """An FP64 Lie step of 8192 planes of 8 x 8 against single launches of the
    unsplit step: two passes take about 1.5 times as long, the march 2.3 times."""
    times = {}
    for scheme in (fk.FK_SCHEME_UNSPLIT, fk.FK_SCHEME_LIE):
        g = fk.Grid(8192, 8, 8, 20e-6, -6e7, 6e7, -3e7, 3e7, cfl=0.4, precision=fk.FK_F64)
        g.set_fields(-1e5, False, 0.0)
        g.set_scheme(scheme)
        g.set_f(np.full((8192, 8, 8), 1e5))
        g.set_kernel_timing(scheme == fk.FK_SCHEME_UNSPLIT)
        best = float("inf")
        for _ in range(6):
            t = time.perf_counter()
            g.step(128)
            g.sync()
            best = min(best, time.perf_counter() - t)
        times[scheme] = best
        g.close()
    assert times[fk.FK_SCHEME_LIE] < 1.9 * times[fk.FK_SCHEME_UNSPLIT]
