"""2D passes (csrc/march.cu) against single steps where long runs and large grids
take them: DFT windows longer than the staging area, summed within a call and
across several, checkpoint segments shorter than a pass, and cells whose offsets
exceed 32 bits.  The forward comparisons are equalities (the same update in the
same rounding); the gradient's bound is test_gpu_march.py's, 1e-6."""
import dataclasses

import numpy as np
import pytest

import workloads as W
from _parity import angles, gpu_solver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_11042_gb300 import lbem
    lbem.lib()


@pytest.mark.parametrize("mode,nx,ny,storage,t0,calls", [
    ("ez", 121, 90, "f32", 11, (230,)), ("hz", 120, 91, "f16", 18, (70, 63, 97)), ("ez", 57, 200, "bf16", 9, (205, 25)),
    ("hz", 40000, 20, "f32", 14, (190,))])
def test_windows_longer_than_the_staging_area(mode, nx, ny, storage, t0, calls):
    """Six periods of 30 steps: three staging areas of 64 steps (five of 44 for
    the long faces), starting and ending within a pass."""
    w = 4 if ny >= 40 else 0
    wave = dataclasses.replace(W.axis_wave(mode, (nx, ny, 1), w, 10.0, gap_ntff=2, gap_tf=2), center=(9.0, 9.0, 0.0))
    eps = np.ones((1, ny, nx), np.float32)
    eps[:, wave.tf_lo[1] + 1:wave.tf_hi[1], wave.tf_lo[0] + 2:wave.tf_lo[0] + 20] = 2.25
    p = W.Problem("window", mode, (nx, ny, 1), eps, w, 0.3, wave, 230, 1)
    got = []
    for fuse in (1, 2):
        s = gpu_solver(p, storage=storage, steps=0, dft=False)
        s.set_step_fusion(fuse)
        s.set_dft_window(t0, 6)
        for n in calls:
            s.step(n)
        s.sync()
        got.append([s.populations(), s.dft(), s.incident_amplitude()] +
                   ([s.far_field(*angles(mode))] if nx < 1000 else []))
        s.close()
    for a, b in zip(*got):
        assert np.isfinite(a).all() and np.abs(a).max() > 0 and np.array_equal(a, b)


@pytest.mark.parametrize("K", [1, 2, 3, 5])
def test_adjoint_segments_shorter_than_a_pass(K):
    mode, nx, ny = "ez", 113, 61
    wave = W.axis_wave(mode, (nx, ny, 1), 5, 6.0, gap_ntff=2, gap_tf=2)
    eps = np.ones((1, ny, nx), np.float32)
    eps[0, ny // 2 - 6:ny // 2 + 6, wave.tf_lo[0] + 2:wave.tf_lo[0] + 14] = W.random_eps((12, 12, 1), 1.5, 3.0, 4)[0]
    steps = 3 * nx // 2 + 150
    p = W.Problem("adj_short", mode, (nx, ny, 1), eps, 5, 0.3, wave, steps, 1)
    got = []
    for fuse, k in ((1, 31), (2, K)):
        s = gpu_solver(p, steps=0)
        s.set_step_fusion(fuse)
        s.set_dft_window(steps - 17, 1)
        s.forward_checkpointed(steps, k)
        J, g = s.adjoint([0.0, 1.0], None, [1.0, 0.5])
        got.append((J, g.cpu().numpy()))
        s.close()
    (j0, g0), (j1, g1) = got
    assert j0 > 0 and np.abs(g0).max() > 0
    assert abs(j1 - j0) <= 1e-12 * j0
    assert np.linalg.norm(g1 - g0) <= 1e-6 * np.linalg.norm(g0)


def test_cells_past_32_bit_offsets():
    """32768 x 32900 cells in FP16 (90 GB of populations): the wave at the far
    end of the grid, where a pair group's element offset exceeds 2^31."""
    import torch
    from paper_2510_11042_gb300 import lbem
    nx, ny = 32768, 32900
    assert nx * (ny - 90) * 2 > 2 ** 31
    wave = W.PlaneWave(direction=(1.0, 0.0, 0.0), polarization=(0.0, 0.0, 1.0), wavelength=8.0, ramp_periods=0.5,
                       tf_lo=(10, ny - 80, 0), tf_hi=(nx - 12, ny - 30, 0), ntff_lo=(9, ny - 82, 0),
                       ntff_hi=(nx - 10, ny - 28, 0), center=(12.0, ny - 50.0, 0.0), source_index=8)
    eps = torch.ones((1, ny, nx), device="cuda")
    eps[:, ny - 70:ny - 40, 14:40] = 2.25
    cells = [(x, y, 0) for x in list(range(8, 48, 2)) + [55, 56, 57, 111, 112] for y in range(ny - 84, ny - 24, 2)]
    got = []
    for fuse in (1, 2):
        s = lbem.Solver((nx, ny, 1), eps, "ez", "f16", 8, 0.3)
        s.set_step_fusion(fuse)
        s.inject(wave)
        s.set_dft_window(50, 1)
        s.step(74)
        got.append([s.probe(cells), lbem.lbem_get_dft(s.h)[::7], s.incident_amplitude()])
        s.close()
        del s
        torch.cuda.empty_cache()
    for a, b in zip(*got):
        assert np.isfinite(a).all() and np.abs(a).max() > 0 and np.array_equal(a, b)
