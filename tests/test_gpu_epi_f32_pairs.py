"""The FP32 epilogue on both sides of its rule for two time points a thread.

Columns of 128 points (one point a thread) and a little more (two), one row of
two points, and rows of an odd number of pairs with tiles half as many and not.
The training step against the FP64 oracle (FP32 bound, 1e-5); the dA mode of the
recomputing backward forms the forward's A bit for bit, whichever form it takes.
"""
import numpy as np
import pytest

import oracle
from oracle import Dims
from paper_2211_12709_gb300 import inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

CASES = [
    Dims(1, 8, 8, 6, 5, 16, 8, 2, 2, 4, 4),
    Dims(2, 5, 7, 4, 6, 17, 8, 2, 2, 4, 5),
    Dims(1, 3, 4, 8, 4, 64, 2, 2, 1, 6, 2),
    Dims(1, 6, 6, 5, 4, 65, 2, 2, 1, 6, 2),
    Dims(1, 20, 20, 4, 5, 48, 14, 2, 2, 6, 8),
    Dims(1, 20, 12, 4, 5, 64, 14, 2, 2, 6, 8),
    Dims(2, 4, 5, 6, 4, 64, 10, 1, 2, 5, 6),
]


def relerr(a, b):
    a = np.asarray(a.detach().cpu().numpy(), dtype=np.float64)
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(np.asarray(b).ravel()))


@pytest.mark.parametrize("d", CASES, ids=[f"{d.Ci}-{d.Co}x{d.Nz}x{d.Nt}" for d in CASES])
def test_both_forms_match_the_oracle(d):
    from paper_2211_12709_gb300 import ops
    modes = (d.mx, d.my, d.mz, d.mt)
    x = inputs.normal((d.B, d.Ci) + d.grid, 721)
    w = inputs.spectral_weights(d.Ci, d.Co, d.modes, 722)
    wl, b = inputs.linear_params(d.Ci, d.Co, 723)
    dz = inputs.normal((d.B, d.Co) + d.grid, 724)
    X, W, WL, Bb, DZ = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (x, w, wl, b, dz))
    ws = ops.workspace(ops.dims_of(X, d.Co, modes), "fp32", ops.OP_BLOCK_TRAIN, X.device)
    z = ops.block_fwd(X, W, WL, Bb, modes, "fp32", ws=ws, train=True)
    got = ops.block_bwd(X, W, WL, Bb, DZ, modes, "fp32", ws=ws, saved=True)
    ref = ops.block_bwd(X, W, WL, Bb, DZ, modes, "fp32")
    torch.cuda.synchronize()
    assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
    rz, _ = oracle.block_fwd(d, x, w, wl, b)
    rg = oracle.block_bwd(d, x, w, dz, wl, b)
    errs = {"z": relerr(z, rz), **{k: relerr(v, rg[k]) for k, v in zip(("dx", "dw", "dwl", "db"), got)}}
    assert all(v <= 1e-5 for v in errs.values()), errs
