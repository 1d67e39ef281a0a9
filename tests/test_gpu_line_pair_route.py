"""The rule that gives the FP32 line stages two inner points per lane, on both sides.

The paired kernel has a launch name of its own: calls well above the line (many
tiles of 64 that are hardly emptier than those of 32) launch it for the y stages or
for all, calls below do not launch it, and both match the FP64 oracle with the FP32
bound of the layer tests (1e-5).
"""
import numpy as np
import pytest

import oracle
from oracle import Dims
from paper_2211_12709_gb300 import inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

PAIR, ONE = "fno_line_pair_f32", "fno_line_f32"
CASES = [
    (Dims(4, 16, 16, 16, 15, 16, 16, 2, 2, 4, 8), {PAIR, ONE}),   # inner 64 on y (1024 tiles), x: 128 tiles
    (Dims(4, 20, 18, 17, 12, 16, 12, 3, 3, 5, 6), {PAIR}),        # inner 60 and 360, 6 rows in groups of four
    (Dims(2, 8, 8, 16, 16, 12, 6, 2, 2, 6, 4), {ONE}),            # inner 48: tiles of 64 a quarter empty
    (Dims(1, 2, 2, 16, 16, 16, 16, 3, 4, 8, 8), {ONE}),           # two tiles of 64 on y, 32 columns: too few
]


def relerr(a, b):
    a = np.asarray(a.detach().cpu().numpy(), dtype=np.float64)
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(np.asarray(b).ravel()))


@pytest.mark.parametrize("d,names", CASES, ids=[f"{d.B}x{d.Ci}-{d.Co}x{d.Nx}x{d.Ny}x{2 * d.mz * d.mt}" for d, _ in CASES])
def test_the_rule_names_the_kernel_and_it_matches_the_oracle(d, names):
    from paper_2211_12709_gb300 import _lib, ops
    modes = (d.mx, d.my, d.mz, d.mt)
    x = inputs.normal((d.B, d.Ci) + d.grid, 741)
    w = inputs.spectral_weights(d.Ci, d.Co, d.modes, 742)
    dy = inputs.normal((d.B, d.Co) + d.grid, 743)
    X, W, DY = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (x, w, dy))
    torch.cuda.synchronize()
    _lib.fno_profile_start()
    y = ops.spectral_fwd(X, W, modes, "fp32")
    dx, dw = ops.spectral_bwd(X, W, DY, modes, precision="fp32")
    torch.cuda.synchronize()
    launched = {n for n in _lib.fno_profile_stop() if n.startswith("fno_line")}
    assert launched == names, launched
    ry, _ = oracle.block_fwd(d, x, w)
    rg = oracle.block_bwd(d, x, w, dy)
    errs = {"y": relerr(y, ry), "dx": relerr(dx, rg["dx"]), "dw": relerr(dw, rg["dw"])}
    assert all(v <= 1e-5 for v in errs.values()), errs
