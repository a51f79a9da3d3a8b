"""2D passes of two and three steps (csrc/march.cu), which take what calls of few
steps ask for and what passes of four leave over on grids whose populations
outgrow L2, against single steps, bit for bit (the same update in the same
rounding): at the ends of their strips (60 and 56 cells), of the rounds of
sixteen rows and of the row chunks, with the wave, the DFT window and its
staging, a mu_r map and every storage type, and mixed with single steps, passes
of four and a batched run."""
import dataclasses

import numpy as np
import pytest

import workloads as W
from _parity import angles

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_11042_gb300 import lbem
    lbem.lib()


def _wave(mode, nx, ny):
    """Its phase reference lies where the wave comes within a few steps."""
    return dataclasses.replace(W.axis_wave(mode, (nx, ny, 1), 4, 10.0, gap_ntff=2, gap_tf=2), center=(9.0, 9.0, 0.0))


CALLS = (2, 3, 2, 2, 1, 3, 4, 2, 7, 6, 3, 3, 1, 1, 2, 5, 2)


def _run(mode, shape, storage, wave, mu, fuse, calls):
    import torch
    from paper_2510_11042_gb300 import lbem
    nx, ny, _ = shape
    w = 4 if min(nx, ny) >= 40 else 0
    eps = W.random_eps(shape, 1.0, 4.0, 5)
    if wave is not None:
        inside = np.ones_like(eps)
        box = (slice(None), slice(wave.tf_lo[1], wave.tf_hi[1] + 1), slice(wave.tf_lo[0], wave.tf_hi[0] + 1))
        inside[box] = eps[box]
        eps = inside
    s = lbem.Solver(shape, eps, mode, storage, w, 0.3)
    if mu:
        s.set_permeability(W.random_eps(shape, 1.0, 3.0, 9))
    s.set_populations(0.125 * W.random_state_f32(mode, shape, 6))   # within FP16 storage over all steps
    s.set_step_fusion(fuse)
    if wave is not None:
        s.inject(wave)
        s.set_dft_window(9, 1)
    for n in calls:
        if n < 0:
            b = lbem.Batch([s])
            b.run([-n], autotune=False)
            b.close()
        else:
            s.step(n)
    s.sync()
    out = [s.populations()]
    if wave is not None:
        th, ph = angles(mode)
        out += [s.dft(), s.incident_amplitude(), s.far_field(th, ph)]
    s.close()
    torch.cuda.empty_cache()
    return out


def _same(mode, shape, storage, wave=None, mu=False, calls=CALLS):
    a, b = (_run(mode, shape, storage, wave, mu, fuse, calls) for fuse in (1, 2))
    for x, y in zip(a, b):
        assert np.isfinite(x).all() and np.array_equal(x, y)
    return a


@pytest.mark.parametrize("mode", ["ez", "hz"])
@pytest.mark.parametrize("nx,ny", [(2, 29500), (60, 14800), (61, 14801), (57, 14817), (1021, 917), (119, 7300),
                                   (29600, 33), (29601, 32), (240000, 4)])
def test_short_passes_match_single_steps_from_a_random_state(mode, nx, ny):
    _same(mode, (nx, ny, 1), "f32")


@pytest.mark.parametrize("storage,mode,nx,ny,axis,mu", [
    ("f32", "ez", 1000, 990, 0, False), ("f32", "hz", 70, 15001, 1, True), ("f32", "ez", 15003, 70, 0, True),
    ("f16", "ez", 1401, 1400, 1, False), ("f16", "hz", 1390, 1407, 0, True), ("bf16", "ez", 1391, 1402, 0, False)])
def test_short_passes_match_single_steps_with_the_wave(storage, mode, nx, ny, axis, mu):
    wave = _wave(mode, nx, ny)
    if axis == 1:
        wave = dataclasses.replace(wave, direction=(0.0, 1.0, 0.0),
                                   polarization=(0.0, 0.0, 1.0) if mode == "ez" else (1.0, 0.0, 0.0))
    out = _same(mode, (nx, ny, 1), storage, wave, mu)
    assert np.abs(out[1]).max() > 0


def test_short_passes_around_batched_runs():
    _same("ez", (1000, 990, 1), "f32", _wave("ez", 1000, 990), calls=(4, -1, 3, -2, 2, 8, -3, 6, -4, 3, 2))


def test_calls_of_few_steps_take_a_pass():
    from paper_2510_11042_gb300 import lbem
    s = lbem.Solver((1000, 1000, 1), np.ones((1, 1000, 1000), np.float32), "ez", "f32", 4, 0.3)
    for n, launches in ((2, 1), (3, 1), (4, 1), (6, 2), (7, 2), (1, 1)):
        before = s.kernel_launches()
        s.step(n)
        assert s.kernel_launches() - before == launches
    s.sync()
    s.close()
