"""The channel mixing and its adjoint with few channels on one side.

One to sixteen input or output channels (fewer than a CTA has groups, a number
that does not divide them, and one more than divides them evenly), batches of one
to several chunks, and mode counts that do not fill the last tile of 16; and 22 to
24 channels on tiles that fill the chip.  Forward
and backward of the FP32 spectral layer against the FP64 oracle with the bound of
the layer tests (1e-5); dW alone has the same bits as with dX.
"""
import numpy as np
import pytest

import oracle
from oracle import Dims
from paper_2211_12709_gb300 import inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

CASES = [
    Dims(5, 1, 20, 6, 5, 6, 6, 3, 1, 3, 3),
    Dims(9, 20, 1, 6, 4, 6, 8, 1, 2, 3, 5),
    Dims(3, 2, 17, 5, 4, 6, 10, 2, 2, 1, 3),
    Dims(2, 5, 3, 4, 4, 4, 6, 2, 1, 2, 4),
    Dims(1, 7, 33, 4, 5, 4, 4, 1, 2, 2, 3),
    Dims(2, 15, 16, 4, 4, 5, 6, 2, 2, 1, 1),
    Dims(1, 16, 15, 4, 4, 5, 6, 2, 2, 1, 3),
    Dims(4, 33, 2, 4, 4, 4, 6, 1, 2, 2, 3),
    Dims(2, 23, 22, 16, 16, 8, 10, 8, 8, 4, 5),   # 640 tiles: two channels in turn
    Dims(5, 22, 24, 16, 16, 8, 10, 8, 8, 4, 5),   # eight entries at a time: the adjoint one each
]


def relerr(a, b):
    a = np.asarray(a.detach().cpu().numpy(), dtype=np.float64)
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(np.asarray(b).ravel()))


@pytest.mark.parametrize("d", CASES, ids=[f"{d.B}x{d.Ci}-{d.Co}" for d in CASES])
def test_mixing_with_few_channels_matches_the_oracle(d):
    from paper_2211_12709_gb300 import ops
    modes = (d.mx, d.my, d.mz, d.mt)
    x = inputs.normal((d.B, d.Ci) + d.grid, 711)
    w = inputs.spectral_weights(d.Ci, d.Co, d.modes, 712)
    dy = inputs.normal((d.B, d.Co) + d.grid, 713)
    X, W, DY = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (x, w, dy))
    y = ops.spectral_fwd(X, W, modes, "fp32")
    dx, dw = ops.spectral_bwd(X, W, DY, modes, precision="fp32")
    _, dw1 = ops.spectral_bwd(X, W, DY, modes, need_dx=False, precision="fp32")
    dx1, _ = ops.spectral_bwd(X, W, DY, modes, need_dw=False, precision="fp32")
    torch.cuda.synchronize()
    assert torch.equal(dw, dw1) and torch.equal(dx, dx1)
    ry, _ = oracle.block_fwd(d, x, w)
    rg = oracle.block_bwd(d, x, w, dy)
    errs = {"y": relerr(y, ry), "dx": relerr(dx, rg["dx"]), "dw": relerr(dw, rg["dw"])}
    assert all(v <= 1e-5 for v in errs.values()), errs
