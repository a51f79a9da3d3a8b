"""The FP64 projection where its phase tables reach the 48 KB of shared memory
that a kernel gets without asking for more: long thin 3D boxes of 3000, 3001,
3008 and 3009 table entries (16 B each, beside the kernel's static part).  Each
box in a process of its own, where no larger table has raised the limit before.

Tolerance as in test_gpu_far_field_f64.py: both sides are FP64; a phase is at most
2 pi / 8 * 1410 = 1110, known to 1110 * 2^-53 = 1.2e-13, and a sum of n = 51,000
cells adds at most n 2^-53 = 6e-12 of its absolute sum: 1e-10 in relative L2."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 1e-10
LO = (1, 1, 1)


def _inputs(nz):
    rng = np.random.default_rng(nz)
    shape, hi = (6, 7, nz + 2), (4, 5, nz)
    grid = rng.standard_normal((*shape[::-1], 6)) + 1j * rng.standard_normal((*shape[::-1], 6))
    box = grid[1:nz + 1, 1:6, 1:5]
    parts = []
    for ax in range(3):
        for side in (0, -1):
            face = np.take(box, side, axis=2 - ax)
            for c in range(6):
                parts += [face[..., c].real.ravel(), face[..., c].imag.ravel()]
    centre = tuple((n - 1) / 2 + 0.25 for n in shape)
    n = 37
    return grid, shape, hi, np.concatenate(parts), centre, rng.uniform(0, np.pi, n), rng.uniform(0, 2 * np.pi, n)


def _project(nz, path):
    import torch
    from paper_2510_11042_gb300 import lbem
    _, shape, hi, dft, centre, theta, phi = _inputs(nz)
    dev = torch.device("cuda", torch.cuda.current_device())
    desc = lbem.NtffDesc(lbem.MODE["3d"], *shape, LO, hi, 8.0, centre, 1.5)
    out = torch.full((theta.size,), float("nan"), dtype=torch.float64, device=dev)
    stream = torch.cuda.current_stream(dev)
    lbem.lbem_far_field_noalloc(desc, torch.from_numpy(dft).to(dev), torch.from_numpy(theta).to(dev),
                                torch.from_numpy(phi).to(dev), out, stream=stream.cuda_stream)
    stream.synchronize()
    np.save(path, out.cpu().numpy())


@pytest.mark.parametrize("nz", [2805, 2806, 2813, 2814])
def test_tables_at_the_shared_memory_limit(nz, tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import ntff
    path = str(tmp_path / "s2.npy")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, PYTHONPATH=root + os.pathsep + os.environ.get("PYTHONPATH", ""))
    r = subprocess.run([sys.executable, os.path.abspath(__file__), str(nz), path], env=env, cwd=root,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    grid, _, hi, _, centre, theta, phi = _inputs(nz)
    want = ntff.far_field(grid, LO, hi, 2 * np.pi / 8.0, centre, 1.5, "3d", theta, phi)
    got = np.load(path)
    assert np.linalg.norm(got - want) <= TOL * np.linalg.norm(want)


if __name__ == "__main__":
    _project(int(sys.argv[1]), sys.argv[2])
