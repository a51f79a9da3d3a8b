"""Single steps on grids of short rows and many of them, which take blocks of one
warp (row_threads, csrc/step_cell.cuh), against 2D passes of four steps, bit for
bit (the same update in the same rounding): the lattice, the incident line, whose
nodes the same blocks update, and the DFT; and in 3D against the FP64 oracle."""
import numpy as np
import pytest

import workloads as W
from _parity import angles, gpu_solver, oracle_to_planes, planes_to_oracle, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_11042_gb300 import lbem
    lbem.lib()


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("mode,nx,ny,axis", [("ez", 8, 5000, 0), ("hz", 31, 6001, 1), ("ez", 32, 4866, 1),
                                             ("hz", 33, 5003, 0)])
def test_short_rows_match_passes(mode, nx, ny, axis, storage):
    pol = (0.0, 0.0, 1.0) if mode == "ez" else ((0.0, 1.0, 0.0) if axis == 0 else (1.0, 0.0, 0.0))
    wave = W.PlaneWave(direction=(1.0, 0.0, 0.0) if axis == 0 else (0.0, 1.0, 0.0), polarization=pol, wavelength=4.0,
                       ramp_periods=0.5, tf_lo=(2, 2, 0), tf_hi=(nx - 3, ny - 3, 0), ntff_lo=(1, 1, 0),
                       ntff_hi=(nx - 2, ny - 2, 0), center=(2.0, 2.0, 0.0), source_index=0)
    eps = W.random_eps((nx, ny, 1), 1.0, 4.0, 5)
    eps[:, :, :2] = eps[:, :, nx - 2:] = eps[:, :2] = eps[:, ny - 2:] = 1.0
    p = W.Problem("thin", mode, (nx, ny, 1), eps, 0, 0.3, wave, 40, 1)
    got = []
    for fuse in (1, 2):
        s = gpu_solver(p, storage=storage, steps=0, dft=False, init=0.125 * W.random_state_f32(mode, p.shape, 6))
        s.set_step_fusion(fuse)
        s.set_dft_window(9, 1)
        s.step(36)
        s.sync()
        got.append([s.populations(), s.dft(), s.incident_amplitude(), s.far_field(*angles(mode))])
        s.close()
    for a, b in zip(*got):
        assert np.isfinite(a).all() and np.abs(a).max() > 0 and np.array_equal(a, b)


@pytest.mark.parametrize("streaming", ["two_buffers", "in_place"])
def test_short_rows_in_3d_against_the_oracle(streaming):
    from oracle import lb
    shape = (17, 80, 61)
    p = W.Problem("thin3d", "3d", shape, W.random_eps(shape, 1.0, 4.0, 5), 2, 0.3, None, 9, 1)
    init = W.random_state_f32("3d", shape, 6)
    s = gpu_solver(p, init=init, streaming=streaming)
    lat = lb.Lattice(shape, p.eps, sponge_w=2, sigma_max=0.3)
    lat.f = planes_to_oracle(init.astype(np.float64), "3d")
    for n in range(9):
        lat.step(n)
    assert rel_l2(s.populations(), oracle_to_planes(lat.f, "3d", shape)) <= 1e-5
    s.close()
