"""Four steps per pass in 2D (csrc/march.cu) against single steps, bit for bit:
populations, DFT accumulators, incident amplitude and far field, at the sizes
where the strips of 56 cells, the rounds of sixteen rows and the row chunks
end, over step counts that leave single steps before, between and after the
passes (both are the same update in the same rounding, so the tolerance is
equality)."""
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


def _compare(mode, shape, storage, wave, mu=False, width=None, axis=0):
    nx, ny, _ = shape
    w = (6 if wave else 2 if min(nx, ny) > 5 else 0) if width is None else width
    eps = W.random_eps(shape, 1.0, 4.0, 5)
    wv = None
    if wave:
        wv = W.axis_wave(mode, shape, w, 10.0, gap_ntff=2, gap_tf=2)
        if axis == 1:
            wv = dataclasses.replace(wv, direction=(0.0, 1.0, 0.0),
                                     polarization=(0.0, 0.0, 1.0) if mode == "ez" else (1.0, 0.0, 0.0))
        inside = np.ones_like(eps)
        box = (slice(None), slice(wv.tf_lo[1], wv.tf_hi[1] + 1), slice(wv.tf_lo[0], wv.tf_hi[0] + 1))
        inside[box] = eps[box]
        eps = inside
    p = W.Problem("march", mode, shape, eps, w, 0.3, wv, 45, 1, mu=W.random_eps(shape, 1.0, 3.0, 9) if mu else None)
    init = W.random_state_f32(mode, shape, 6)
    got = []
    for fuse in (1, 2):
        s = gpu_solver(p, storage=storage, init=init, steps=0)
        s.set_step_fusion(fuse)
        assert s.step_fusion() == fuse
        if wave:
            s.set_dft_window(8, 1)
        for n in (38, 1, 6):
            s.step(n)
        s.sync()
        out = [s.populations()]
        if wave:
            th, ph = angles(mode)
            out += [s.dft(), s.incident_amplitude(), s.far_field(th, ph)]
        got.append(out)
        s.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)
    return got[1]


@pytest.mark.parametrize("mode", ["ez", "hz"])
@pytest.mark.parametrize("nx,ny", [(2, 2), (3, 40), (56, 4), (57, 5), (64, 17), (113, 300), (2001, 33), (700, 2050)])
def test_passes_match_single_steps_from_a_random_state(mode, nx, ny):
    _compare(mode, (nx, ny, 1), "f32", wave=False)


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("mode,nx,ny,axis,mu", [("ez", 121, 90, 0, False), ("hz", 120, 91, 1, False),
                                                ("ez", 168, 61, 1, True), ("hz", 57, 333, 0, True)])
def test_passes_match_single_steps_with_the_wave(mode, nx, ny, axis, mu, storage):
    out = _compare(mode, (nx, ny, 1), storage, wave=True, axis=axis, mu=mu)
    assert np.abs(out[1]).max() > 0


def test_line_restarts_after_a_snapshot():
    """The passes keep the incident line ahead of the state; loading a snapshot
    of an earlier time starts it again from the snapshot's own line."""
    from paper_2510_11042_gb300 import lbem
    p = W.cylinder_problem(n=96, x=2.0, wavelength=10.0, eps_in=2.25, w=6, mode="ez", periods=8)
    s = gpu_solver(p, steps=0)
    s.step(41)
    snap = lbem.lbem_save_state(s.h)
    s.step(60)
    ref = s.populations()
    lbem.lbem_load_state(s.h, snap)
    s.step(60)
    assert np.array_equal(s.populations(), ref)


@pytest.mark.parametrize("mode", ["ez", "hz"])
@pytest.mark.parametrize("nx,ny,K", [(57, 61, 23), (113, 300, 31), (168, 50, 20), (600, 53, 25)])
def test_adjoint_passes_match_single_steps(mode, nx, ny, K):
    """Replay and backward sweep in passes of four steps (with the single steps
    that K leaves over) against one launch a step.  The arithmetic is the same
    but for the FP64 phase products of the DFT source, whose contraction the
    compiler chooses: a difference of 2^-52 there can move its FP32 rounding by
    one unit (6e-8), and the sweep is linear in it; 1e-6 allows sixteen of them."""
    from paper_2510_11042_gb300 import lbem
    import torch
    w = 5
    wv = W.axis_wave(mode, (nx, ny, 1), w, 6.0, gap_ntff=2, gap_tf=2)
    eps = np.ones((1, ny, nx), np.float32)
    eps[0, ny // 2 - 6:ny // 2 + 6, wv.tf_lo[0] + 2:wv.tf_lo[0] + 14] = W.random_eps((12, 12, 1), 1.5, 3.0, 4)[0]
    steps = 3 * nx // 2 + 150
    p = W.Problem("adj_march", mode, (nx, ny, 1), eps, w, 0.3, wv, steps, 1)
    got = []
    for fuse in (1, 2):
        s = gpu_solver(p, steps=0)
        s.set_step_fusion(fuse)
        s.set_dft_window(steps - 17, 1)
        s.forward_checkpointed(steps, K)
        J, g = s.adjoint([0.0, 1.0], None, [1.0, 0.5])
        got.append((J, g.cpu().numpy()))
        torch.cuda.synchronize()
        s.close()
    (j0, g0), (j1, g1) = got
    assert j0 > 0 and np.abs(g0).max() > 0
    assert abs(j1 - j0) <= 1e-12 * j0
    assert np.linalg.norm(g1 - g0) <= 1e-6 * np.linalg.norm(g0)
