"""dW_lin and db of a training step beyond the two-CTA dA pass (25 to 32 outputs, 32 inputs and more).

FP32, and the tensor-core precisions on grids that the tensor-core dA epilogue does
not tile, form them in FP32 but at 32 -> 29..32: with one nonzero dA = 1 per output
channel dW_lin is a value of x, all 24 bits of it.  (w = 0, w_lin = 0 and bias = 50
make A exactly 50, where GELU' is exactly 1 in every form.)  Split BF16 on the other
grids, and every precision at 32 -> 29..32, take the wide tensor-core pass, whose
error there is the smaller one: its channel bounds, both counts of m-tiles, a partly filled tile of points and
more than one batch entry against the FP64 oracle, with the bound of the block tests
(1e-5).
"""
import numpy as np
import pytest

import oracle
from oracle import Dims
from paper_2211_12709_gb300 import inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

EXACT = [("fp32", 28, 28, 16), ("fp32", 32, 28, 16), ("fp32", 33, 25, 10), ("fp32", 40, 28, 16), ("fp32", 47, 32, 7),
         ("bf16x3", 28, 28, 20), ("bf16x3", 31, 32, 20), ("bf16x3", 40, 28, 16), ("tf32", 32, 28, 20),
         ("bf16", 30, 32, 20)]


@pytest.mark.parametrize("precision,ci,co,nt", EXACT, ids=["-".join(map(str, c)) for c in EXACT])
def test_dw_lin_keeps_every_bit_of_fp32_operands(precision, ci, co, nt):
    from paper_2211_12709_gb300 import ops
    grid, modes = (4, 6, 8, nt), (1, 2, 2, 4)
    n = int(np.prod(grid))
    rng = np.random.default_rng(801)
    x = rng.standard_normal((1, ci) + grid).astype(np.float32)
    dz = np.zeros((1, co, n), np.float32)
    at = rng.permutation(n)[:co]
    dz[0, np.arange(co), at] = 1.0
    X, DZ = (torch.from_numpy(a).cuda() for a in (x, dz.reshape((1, co) + grid)))
    W = torch.zeros(ops._wshape(ci, co, modes), device="cuda")
    WL, Bb = torch.zeros((ci, co), device="cuda"), torch.full((co,), 50.0, device="cuda")
    ws = ops.workspace(ops.dims_of(X, co, modes), precision, ops.OP_BLOCK_TRAIN, X.device)
    z = ops.block_fwd(X, W, WL, Bb, modes, precision, ws=ws, train=True)
    _, _, dwl, db = ops.block_bwd(X, W, WL, Bb, DZ, modes, precision, ws=ws, saved=True)
    torch.cuda.synchronize()
    assert torch.all(z == 50.0)
    assert torch.all(db == 1.0)
    assert np.array_equal(dwl.cpu().numpy(), x.reshape(ci, n)[:, at])


WIDE = [
    Dims(1, 32, 32, 4, 5, 16, 16, 2, 2, 4, 6),
    Dims(2, 31, 25, 5, 3, 24, 16, 2, 1, 4, 6),
    Dims(1, 32, 24, 4, 4, 12, 32, 2, 2, 4, 8),
    Dims(2, 9, 32, 3, 5, 16, 32, 1, 2, 4, 8),
    Dims(1, 1, 27, 3, 3, 8, 16, 1, 1, 4, 5),
    Dims(1, 32, 32, 5, 4, 12, 20, 2, 1, 4, 6),
    Dims(2, 32, 29, 3, 4, 10, 34, 1, 2, 3, 8),
]


def relerr(a, b):
    a = np.asarray(a.detach().cpu().numpy(), dtype=np.float64)
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(np.asarray(b).ravel()))


CHAIN = [("fp32", d) for d in (Dims(1, 32, 32, 4, 5, 16, 16, 2, 2, 4, 6), Dims(2, 32, 29, 3, 4, 9, 7, 1, 2, 3, 4))]
RUNS = [("bf16x3", d) for d in WIDE] + CHAIN


@pytest.mark.parametrize("precision,d", RUNS, ids=[f"{p}-{d.B}x{d.Ci}-{d.Co}x{d.Nz}x{d.Nt}" for p, d in RUNS])
def test_wide_tensor_core_pass_matches_the_oracle(precision, d):
    from paper_2211_12709_gb300 import _lib, ops
    modes = (d.mx, d.my, d.mz, d.mt)
    x = inputs.normal((d.B, d.Ci) + d.grid, 811)
    w = inputs.spectral_weights(d.Ci, d.Co, d.modes, 812)
    wl, b = inputs.linear_params(d.Ci, d.Co, 813)
    dz = inputs.normal((d.B, d.Co) + d.grid, 814)
    X, W, WL, Bb, DZ = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (x, w, wl, b, dz))
    ws = ops.workspace(ops.dims_of(X, d.Co, modes), precision, ops.OP_BLOCK_TRAIN, X.device)
    _lib.fno_profile_start()
    z = ops.block_fwd(X, W, WL, Bb, modes, precision, ws=ws, train=True)
    got = ops.block_bwd(X, W, WL, Bb, DZ, modes, precision, ws=ws, saved=True)
    torch.cuda.synchronize()
    names = _lib.fno_profile_stop()
    assert "fno_da_saved" in names, sorted(names)
    rz, _ = oracle.block_fwd(d, x, w, wl, b)
    rg = oracle.block_bwd(d, x, w, dz, wl, b)
    errs = {"z": relerr(z, rz), **{k: relerr(v, rg[k]) for k, v in zip(("dx", "dw", "dwl", "db"), got)}}
    print(errs)
    assert all(v <= 1e-5 for v in errs.values()), errs
