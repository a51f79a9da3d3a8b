"""The FP64 projection (far_field_columns, through lbem_far_field_noalloc) on
random phasors against the FP64 oracle, on boxes of every way it gets its
phases: few and many fine offsets per coarse entry, ragged last entries, faces
of three cells, boxes shorter than a block's columns and longer.

Both sides are FP64 and differ in the order of the sums and in how the phases
are formed.  A phase k r.(p - c) is at most 2 pi / 8 * 700 = 550 here, known to
550 * 2^-53 = 6e-14 on either side; as products, with two factors' errors; a sum
of n terms adds at most n 2^-53 = 1e-12 of its absolute sum for 10^4 cells.  The
bar is 1e-10 in relative L2 over the angles."""
import numpy as np
import pytest

from _parity import rel_l2

pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.mark.parametrize("mode,shape,lo,hi", [
    ("ez", (7, 9, 1), (2, 3, 0), (4, 6, 0)),
    ("hz", (48, 320, 1), (5, 4, 0), (40, 300, 0)),
    ("ez", (1200, 70, 1), (3, 4, 0), (1190, 65, 0)),
    ("hz", (513, 514, 1), (0, 1, 0), (511, 513, 0)),
    ("3d", (12, 20, 9), (2, 3, 1), (9, 16, 5)),
    ("3d", (40, 24, 70), (3, 2, 2), (35, 20, 66)),
])
def test_projection_of_random_phasors(mode, shape, lo, hi):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import ntff
    from paper_2510_11042_gb300 import lbem
    rng = np.random.default_rng(sum(shape))
    held = {"ez": (2, 3, 4), "hz": (0, 1, 5), "3d": range(6)}[mode]   # of Ex Ey Ez Hx Hy Hz
    grid = np.zeros((shape[2], shape[1], shape[0], 6), complex)
    for c in held:
        grid[..., c] = rng.standard_normal(grid.shape[:3]) + 1j * rng.standard_normal(grid.shape[:3])
    box = grid[tuple(slice(lo[a], hi[a] + 1) for a in (2, 1, 0))]
    parts = []
    for ax in range(3):
        if shape[ax] == 1:
            continue
        for side in (0, -1):
            face = np.take(box, side, axis=2 - ax)        # [u][v][6]
            for c in held:
                parts += [face[..., c].real.ravel(), face[..., c].imag.ravel()]
    centre = tuple((n - 1) / 2 + 0.25 for n in shape)
    desc = lbem.NtffDesc(lbem.MODE[mode], *shape, lo, hi, 8.0, centre, 1.5)
    n = 37
    theta = rng.uniform(0.0, np.pi, n)
    phi = rng.uniform(0.0, 2.0 * np.pi, n) if mode == "3d" else None
    dev = torch.device("cuda", torch.cuda.current_device())
    dft = torch.from_numpy(np.concatenate(parts)).to(dev)
    assert dft.numel() == lbem.ntff_dft_doubles(desc)
    out = torch.full((n,), float("nan"), dtype=torch.float64, device=dev)
    stream = torch.cuda.current_stream(dev)
    lbem.lbem_far_field_noalloc(desc, dft, torch.from_numpy(theta).to(dev),
                                torch.from_numpy(phi).to(dev) if phi is not None else None, out,
                                stream=stream.cuda_stream)
    stream.synchronize()
    want = ntff.far_field(grid, lo, hi, 2 * np.pi / 8.0, centre, 1.5, mode, theta, phi)
    assert rel_l2(out.cpu().numpy(), want) <= TOL
