"""The column epilogue with many kept z modes, and the block function without kept state.

2 mz of 26 and 32 (four k-steps of the z phase), and beyond, where no tensor-core line
takes the inverse z stage and the FP32 epilogue runs, at the channel bounds, against the FP64 oracle with the bound of the block tests (split BF16 1e-5);
and the autograd function called with train=False under grad, whose backward
recomputes everything.
"""
import numpy as np
import pytest

import oracle
from oracle import Dims
from paper_2211_12709_gb300 import inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

F32, COL = "f32", "cmma_bf16x3"
CASES = [
    (Dims(1, 32, 32, 4, 4, 64, 20, 2, 2, 32, 8), F32),
    (Dims(1, 20, 20, 5, 4, 50, 30, 2, 2, 25, 7), F32),
    (Dims(2, 8, 12, 3, 6, 28, 16, 1, 2, 13, 6), COL),
    (Dims(1, 24, 17, 4, 4, 66, 34, 2, 2, 29, 8), F32),
    (Dims(1, 32, 32, 4, 4, 64, 20, 2, 2, 16, 8), COL),
    (Dims(1, 20, 20, 5, 4, 50, 30, 2, 2, 16, 7), COL),
    (Dims(1, 24, 17, 4, 4, 66, 34, 2, 2, 16, 8), COL),
]


def relerr(a, b):
    a = np.asarray(a.detach().cpu().numpy(), dtype=np.float64)
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(np.asarray(b).ravel()))


def make(d):
    x = inputs.normal((d.B, d.Ci) + d.grid, 751)
    w = inputs.spectral_weights(d.Ci, d.Co, d.modes, 752)
    wl, b = inputs.linear_params(d.Ci, d.Co, 753)
    dz = inputs.normal((d.B, d.Co) + d.grid, 754)
    return x, w, wl, b, dz


@pytest.mark.parametrize("d,kernel", CASES, ids=[f"{d.Ci}-{d.Co}x{d.Nz}x{d.Nt}-2mz{2 * d.mz}" for d, _ in CASES])
def test_many_z_modes_match_the_oracle(d, kernel):
    from paper_2211_12709_gb300 import _lib, ops
    modes = (d.mx, d.my, d.mz, d.mt)
    x, w, wl, b, dz = make(d)
    X, W, WL, Bb, DZ = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (x, w, wl, b, dz))
    ws = ops.workspace(ops.dims_of(X, d.Co, modes), "bf16x3", ops.OP_BLOCK_TRAIN, X.device)
    _lib.fno_profile_start()
    z = ops.block_fwd(X, W, WL, Bb, modes, "bf16x3", ws=ws, train=True)
    got = ops.block_bwd(X, W, WL, Bb, DZ, modes, "bf16x3", ws=ws, saved=True)
    y = ops.spectral_fwd(X, W, modes, "bf16x3")
    torch.cuda.synchronize()
    names = _lib.fno_profile_stop()
    assert {f"fno_epi_{m}_{kernel}" for m in ("fwd_train", "dx", "spectral")} <= set(names), sorted(names)
    rz, _ = oracle.block_fwd(d, x, w, wl, b)
    ry, _ = oracle.block_fwd(d, x, w)
    rg = oracle.block_bwd(d, x, w, dz, wl, b)
    errs = {"z": relerr(z, rz), "y": relerr(y, ry),
            **{k: relerr(v, rg[k]) for k, v in zip(("dx", "dw", "dwl", "db"), got)}}
    print(errs)
    assert all(v <= 1e-5 for v in errs.values()), errs


@pytest.mark.parametrize("precision", ["fp32", "bf16x3"])
def test_function_without_kept_state_recomputes_in_its_backward(precision):
    from paper_2211_12709_gb300 import ops
    d = Dims(1, 4, 5, 6, 5, 16, 8, 2, 2, 4, 4)
    modes = (d.mx, d.my, d.mz, d.mt)
    x, w, wl, b, dz = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in make(d))
    leaves = [t.clone().requires_grad_(True) for t in (x, w, wl, b)]
    z = ops.FNOBlock4dFn.apply(*leaves, modes, precision, False)
    z.backward(dz)
    ref = ops.block_bwd(x, w, wl, b, dz, modes, precision)
    torch.cuda.synchronize()
    assert torch.equal(z, ops.block_fwd(x, w, wl, b, modes, precision))
    for t, r in zip(leaves, ref):
        assert torch.equal(t.grad, r)
