"""The FP32 line stages with two inner points per lane, at the edges of their tiling.

Inner extents of one and two whole tiles of 64 and of a partly filled one, axes
of odd length, and output rows that do not fill a group of four.  The training step runs against the FP64
oracle with the FP32 bound of the block tests.
"""
import numpy as np
import pytest

import oracle
from oracle import Dims
from paper_2211_12709_gb300 import inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

CASES = [
    Dims(1, 20, 20, 16, 15, 16, 16, 2, 2, 4, 8),   # inner 64 on y
    Dims(1, 20, 20, 17, 12, 16, 12, 3, 3, 5, 6),   # inner 60 on y, 6 rows of a group of four
    Dims(2, 13, 11, 16, 9, 20, 18, 3, 1, 6, 5),    # inner 60, odd channels, 2 rows
    Dims(1, 20, 20, 15, 16, 16, 16, 3, 4, 8, 8),   # inner 128 on y, 1024 on x
]


def relerr(a, b):
    a = np.asarray(a.detach().cpu().numpy(), dtype=np.float64)
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(np.asarray(b).ravel()))


@pytest.mark.parametrize("d", CASES, ids=[f"{d.B}x{d.Ci}-{d.Co}x{d.Nx}x{d.Ny}x{d.Nz}x{d.Nt}" for d in CASES])
def test_paired_lines_match_the_oracle(d):
    from paper_2211_12709_gb300 import ops
    modes = (d.mx, d.my, d.mz, d.mt)
    x = inputs.normal((d.B, d.Ci) + d.grid, 601)
    w = inputs.spectral_weights(d.Ci, d.Co, d.modes, 602)
    wl, b = inputs.linear_params(d.Ci, d.Co, 603)
    dz = inputs.normal((d.B, d.Co) + d.grid, 604)
    X, W, WL, Bb, DZ = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (x, w, wl, b, dz))
    z = ops.block_fwd(X, W, WL, Bb, modes, "fp32")
    got = ops.block_bwd(X, W, WL, Bb, DZ, modes, "fp32")
    rz, _ = oracle.block_fwd(d, x, w, wl, b)
    rg = oracle.block_bwd(d, x, w, dz, wl, b)
    errs = {"z": relerr(z, rz), **{k: relerr(v, rg[k]) for k, v in zip(("dx", "dw", "dwl", "db"), got)}}
    print(errs)
    assert all(v <= 1e-5 for v in errs.values()), errs
