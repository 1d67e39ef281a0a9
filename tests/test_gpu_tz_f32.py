"""The FP32 t, z DFT in each of its forms: every size that is accepted has one.

Long z and t axes whose warp-per-column plan does not fit shared memory, the
edges of the rules between the forms (16-byte rows, copied rows, rows read in
place, a CTA per column), both row counts of a lane and more than one group of
eight kt.  Forward and backward of the spectral layer against the FP64 oracle with
the FP32 bound of the other layer tests (1e-5).
"""
import numpy as np
import pytest

import oracle
from oracle import Dims
from paper_2211_12709_gb300 import inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

WARP, CTA = "fno_fwd_tz_f32", "fno_fwd_tz_cta_f32"
CASES = [
    (Dims(1, 2, 2, 4, 4, 32, 1450, 1, 1, 4, 8), WARP),   # copied rows of 32 x 1450 floats do not fit
    (Dims(1, 2, 1, 4, 4, 2600, 8, 1, 1, 2, 2), CTA),     # P of 2600 rows does not fit
    (Dims(1, 1, 2, 4, 2, 2601, 6, 1, 1, 2, 2), CTA),     # nor with 8-byte rows
    (Dims(1, 1, 1, 2, 2, 6, 9002, 1, 1, 2, 2), CTA),     # nor a t table padded to eight kt
    (Dims(1, 2, 3, 4, 4, 1030, 18, 1, 1, 5, 4), CTA),    # one warp on an SM
    (Dims(1, 1, 2, 3, 4, 100, 1022, 1, 1, 4, 8), CTA),   # long rows, more than 48 planes
    (Dims(1, 2, 2, 4, 4, 262, 22, 2, 2, 6, 10), WARP),   # rows in place, 64 at a time, two groups of kt
    (Dims(1, 2, 3, 4, 5, 46, 254, 2, 2, 5, 8), WARP),    # rows in place, few planes and long rows
    (Dims(1, 3, 2, 4, 6, 45, 22, 2, 3, 5, 8), WARP),     # copied rows, 64 at a time
    (Dims(1, 2, 2, 6, 4, 20, 30, 2, 2, 4, 12), WARP),    # copied rows, two groups of kt
]


def relerr(a, b):
    a = np.asarray(a.detach().cpu().numpy(), dtype=np.float64)
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(np.asarray(b).ravel()))


@pytest.mark.parametrize("d,kernel", CASES, ids=[f"{d.Nz}x{d.Nt}-mt{d.mt}" for d, _ in CASES])
def test_spectral_layer_matches_the_oracle_on_long_columns(d, kernel):
    from paper_2211_12709_gb300 import _lib, ops
    modes = (d.mx, d.my, d.mz, d.mt)
    x = inputs.normal((d.B, d.Ci) + d.grid, 701)
    w = inputs.spectral_weights(d.Ci, d.Co, d.modes, 702)
    dy = inputs.normal((d.B, d.Co) + d.grid, 703)
    X, W, DY = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (x, w, dy))
    torch.cuda.synchronize()
    _lib.fno_profile_start()
    y = ops.spectral_fwd(X, W, modes, "fp32")
    dx, dw = ops.spectral_bwd(X, W, DY, modes, precision="fp32")
    torch.cuda.synchronize()
    names = _lib.fno_profile_stop()
    assert {n for n in names if n.startswith("fno_fwd_tz")} == {kernel}, sorted(names)
    ry, _ = oracle.block_fwd(d, x, w)
    rg = oracle.block_bwd(d, x, w, dy)
    errs = {"y": relerr(y, ry), "dx": relerr(dx, rg["dx"]), "dw": relerr(dw, rg["dw"])}
    print(errs)
    assert all(v <= 1e-5 for v in errs.values()), errs
