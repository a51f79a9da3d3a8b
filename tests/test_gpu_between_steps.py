"""Calls that change what the steps read, taken between two of them: the step
kernels of one call are chained (a kernel may start before the one before it has
finished), and what the changing call enqueued has to be complete all the same.
Both sides of each comparison run the same kernels on the same values, so the
tolerance is equality."""
import dataclasses

import numpy as np
import pytest

import workloads as W
from _parity import gpu_solver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_11042_gb300 import lbem
    lbem.lib()


@pytest.mark.parametrize("mode,shape,analytic", [("ez", (200, 200, 1), True), ("hz", (131, 77, 1), True),
                                                 ("ez", (200, 200, 1), False), ("3d", (48, 40, 36), False)])
def test_maps_changed_between_steps(mode, shape, analytic):
    """eps_r and mu_r maps set and followed at once by steps, against the same
    calls with the stream synchronised after each."""
    import torch
    wave = W.axis_wave(mode, shape, 6, 10.0, gap_ntff=2, gap_tf=2)
    if analytic:
        wave = dataclasses.replace(wave, analytic=True, origin=(20.0, 20.0, 0.0))
    eps = [torch.from_numpy(W.random_eps(shape, 1.0, 4.0, k)).cuda() for k in range(4)]
    mu = torch.from_numpy(W.random_eps(shape, 1.0, 2.0, 9)).cuda()
    p = W.Problem("maps", mode, shape, eps[0].cpu().numpy(), 6, 0.3, wave, 60, 1)
    got = []
    for wait in (True, False):
        s = gpu_solver(p, steps=0, dft=False, init=W.random_state_f32(mode, shape, 6))
        s.step(40)
        for k in range(24):
            s.set_permittivity(eps[k % 4])
            if wait:
                torch.cuda.synchronize()
            s.step(2)
            if k % 4 == 3:
                s.set_permeability(mu if k % 8 == 3 else None)
                if wait:
                    torch.cuda.synchronize()
                s.step(5)
        s.sync()
        got.append(s.populations())
        s.close()
    assert np.isfinite(got[0]).all() and np.abs(got[0]).max() > 0
    assert np.array_equal(got[0], got[1])


@pytest.mark.parametrize("t", [7, 8, 9, 10])
@pytest.mark.parametrize("mode,shape", [("ez", (90, 70, 1)), ("3d", (40, 36, 34))])
def test_a_wave_injected_again_starts_from_an_empty_line(mode, shape, t):
    """At any time, after another wave has filled the line's buffers: as on a
    handle that never had one, in a workspace of zeros."""
    wave = W.axis_wave(mode, shape, 4, 10.0, gap_ntff=2, gap_tf=2)
    first = dataclasses.replace(wave, wavelength=8.0, amplitude=3.0, ramp_periods=0.0)
    p = W.Problem("again", mode, shape, W.random_eps(shape, 1.0, 4.0, 5), 4, 0.3, None, 60, 1)
    init = W.random_state_f32(mode, shape, 6)
    got = []
    for again in (False, True):
        s = gpu_solver(p, steps=0)
        if again:
            s.inject(first)
        else:
            s.workspace.zero_()          # and what the handle keeps there, anew
            s.set_permittivity(p.eps)
            s.set_permeability(None)
        s.step(t)
        s.inject(wave)
        s.set_populations(init)
        s.set_dft_window(t + 3, 1)
        s.step(38)
        s.sync()
        got.append([s.populations(), s.dft(), s.incident_amplitude()])
        s.close()
    for a, b in zip(*got):
        assert np.isfinite(a).all() and np.array_equal(a, b)


def test_two_step_passes_outside_the_window_of_faces_too_large_to_stage():
    """A flat 3D grid whose NTFF faces (46 million cells) exceed what a pass can
    stage takes single steps in the DFT window only: the kernels that run, and
    the state and sums of a run through the window against single steps."""
    import torch
    from paper_2510_11042_gb300 import lbem
    nx, ny, nz = 4800, 4800, 5
    wave = W.PlaneWave(direction=(1.0, 0.0, 0.0), polarization=(0.0, 0.0, 1.0), wavelength=4.0, amplitude=1.0,
                       ramp_periods=0.5, tf_lo=(6, 2, 1), tf_hi=(nx - 4, ny - 3, 3), ntff_lo=(5, 1, 0),
                       ntff_hi=(nx - 3, ny - 2, 4), center=(nx / 2, ny / 2, 2.0), source_index=0)
    eps = torch.ones((nz, ny, nx), device="cuda")
    eps[:, :, 10:30] = 2.25
    cells = [(x, y, z) for x in (4, 5, 6, 9, 12, 20) for y in (0, 1, 2, 77, 4799) for z in range(5)]
    got = []
    for fuse in (1, 2):
        s = lbem.Solver((nx, ny, nz), eps, "3d", "f16")
        s.set_step_fusion(fuse)
        s.inject(wave)
        s.set_dft_window(21, 1)
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
            s.step(20)
            s.sync()
        names = [e.key for e in prof.key_averages()]
        assert any("step2_kernel" in k for k in names) == (fuse == 2), names
        s.step(15)
        s.sync()
        got.append([s.probe(cells), lbem.lbem_get_dft(s.h)[::97], s.incident_amplitude()])
        s.close()
        del s
        torch.cuda.empty_cache()
    assert np.abs(got[0][0]).max() > 0 and np.abs(got[0][1]).max() > 0
    for a, b in zip(*got):
        assert np.array_equal(a, b)
