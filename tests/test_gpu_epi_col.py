"""The column epilogue (inverse z, t + 1x1 + GELU, and dX) at the edges of its tiling.

Sixteen-plane tiles with a remainder of one and of fifteen planes, eight-point t
sub-tiles with remainders of two to six points on 8- and 16-byte rows, one kept
kz more or less than a k-step of eight, odd and single channels, one to four
t items a warp, and the channel bounds of its register arrays.  Every case runs
the training forward, the plain forward and the backward against the FP64
oracle with the precisions' bounds of the block tests (split BF16 1e-5, BF16
2e-2: the stages are the same ones, with the same operand types).
"""
import numpy as np
import pytest

import oracle
from oracle import Dims
from paper_2211_12709_gb300 import inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

TOL = {"bf16x3": 1e-5, "bf16": 2e-2}

CASES = [
    Dims(1, 5, 5, 6, 6, 17, 36, 2, 2, 5, 5),      # one plane past a tile, 16-byte rows, 4 points past a tile
    Dims(1, 6, 6, 7, 5, 31, 20, 2, 2, 4, 8),      # fifteen planes past a tile, 2mz = 8: one whole k-step
    Dims(2, 3, 5, 4, 8, 18, 10, 1, 2, 9, 6),      # Nt <= 16: one sub-tile; 2mz = 18
    Dims(1, 12, 12, 6, 6, 16, 34, 2, 2, 3, 7),    # 8-byte rows, a t tile of two points
    Dims(1, 20, 20, 6, 6, 16, 16, 2, 2, 7, 4),    # Nt = 16
    Dims(1, 13, 20, 5, 7, 32, 32, 2, 3, 6, 8),    # 13 -> 20 channels, Nt = 32
    Dims(1, 20, 17, 4, 9, 16, 96, 2, 2, 2, 8),    # 20 -> 17 channels, three items a warp
    Dims(1, 24, 22, 6, 6, 16, 32, 2, 2, 4, 5),    # the 24-channel bound
    Dims(1, 32, 31, 6, 6, 18, 126, 2, 2, 4, 8),   # 32 -> 31 channels, four items a warp, 8-byte rows
    Dims(1, 32, 32, 6, 6, 16, 8, 2, 2, 8, 5),     # 32 channels, Nt = 8, 2mz = Nz
    Dims(1, 1, 2, 8, 8, 16, 32, 2, 2, 8, 8),      # a single input channel
    Dims(3, 2, 1, 4, 8, 20, 128, 2, 2, 4, 8),     # a single output channel, the largest Nt
]


def relerr(a, b):
    a = np.asarray(a.detach().cpu().numpy(), dtype=np.float64)
    return float(np.linalg.norm((a - b).ravel()) / max(np.linalg.norm(np.asarray(b).ravel()), 1e-300))


@pytest.mark.parametrize("precision", ["bf16x3", "bf16"])
@pytest.mark.parametrize("d", CASES, ids=[f"{d.B}x{d.Ci}-{d.Co}x{d.Nx}x{d.Ny}x{d.Nz}x{d.Nt}" for d in CASES])
def test_column_epilogue_matches_the_oracle(d, precision):
    from paper_2211_12709_gb300 import _lib, ops
    modes = (d.mx, d.my, d.mz, d.mt)
    x = inputs.normal((d.B, d.Ci) + d.grid, 501)
    w = inputs.spectral_weights(d.Ci, d.Co, d.modes, 502)
    wl, b = inputs.linear_params(d.Ci, d.Co, 503)
    dz = inputs.normal((d.B, d.Co) + d.grid, 504)
    X, W, WL, Bb, DZ = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (x, w, wl, b, dz))
    ws = ops.workspace(ops.dims_of(X, d.Co, modes), precision, ops.OP_BLOCK_TRAIN, X.device)
    _lib.fno_profile_start()
    z = ops.block_fwd(X, W, WL, Bb, modes, precision)
    zt = ops.block_fwd(X, W, WL, Bb, modes, precision, ws=ws, train=True)
    dx, dw, dwl, db = ops.block_bwd(X, W, WL, Bb, DZ, modes, precision, ws=ws, saved=True)
    y = ops.spectral_fwd(X, W, modes, precision)
    torch.cuda.synchronize()
    names = _lib.fno_profile_stop()
    wanted = ["dx", "spectral", "fwd"]
    if precision == "bf16":  # the grids of the mma.sync epilogue, and not the forward
        fused = d.Nt in (16, 32) and d.Nz % (128 // d.Nt) == 0
        wanted = ["dx", "spectral"] if fused else []
    assert all(f"fno_epi_{m}_cmma_{precision}" in names for m in wanted), sorted(names)
    assert torch.equal(z, zt)
    rz, _ = oracle.block_fwd(d, x, w, wl, b)
    ry, _ = oracle.block_fwd(d, x, w)
    rg = oracle.block_bwd(d, x, w, dz, wl, b)
    errs = {"z": relerr(z, rz), "y": relerr(y, ry), "dx": relerr(dx, rg["dx"]), "dw": relerr(dw, rg["dw"]),
            "dwl": relerr(dwl, rg["dwl"]), "db": relerr(db, rg["db"])}
    print(precision, errs)
    assert all(v <= TOL[precision] for v in errs.values()), errs
