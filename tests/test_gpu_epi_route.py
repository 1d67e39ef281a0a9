"""Which epilogue kernels run where tiles of 16 planes are partly empty, and above 24 channels.

Both sides of each line: the training step launches the kernel that the dispatch's
rule names, and matches the FP64 oracle with the bound of the block tests (split
BF16 1e-5, BF16 2e-2).
"""
import numpy as np
import pytest

import oracle
from oracle import Dims
from paper_2211_12709_gb300 import inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

TOL = {"bf16x3": 1e-5, "bf16": 2e-2}
FORMER, COL = "mma", "cmma"
CASES = [
    ("bf16x3", Dims(1, 20, 20, 6, 5, 4, 32, 2, 2, 2, 8), COL, COL),
    ("bf16x3", Dims(1, 24, 21, 6, 5, 4, 32, 2, 2, 2, 8), FORMER, FORMER),
    ("bf16x3", Dims(1, 28, 28, 6, 5, 8, 16, 2, 2, 4, 6), FORMER, FORMER),
    ("bf16x3", Dims(1, 28, 25, 5, 5, 20, 32, 2, 2, 4, 6), FORMER, FORMER),
    ("bf16x3", Dims(1, 28, 28, 5, 5, 24, 16, 2, 2, 4, 6), COL, COL),
    ("bf16x3", Dims(1, 28, 26, 32, 32, 4, 20, 2, 2, 2, 6), "synth", "synth"),
    ("bf16x3", Dims(1, 28, 26, 16, 16, 4, 20, 2, 2, 2, 6), COL, COL),
    ("bf16", Dims(1, 24, 24, 6, 5, 16, 16, 2, 2, 4, 6), FORMER, COL),
    ("bf16", Dims(1, 25, 24, 6, 5, 16, 16, 2, 2, 4, 6), FORMER, FORMER),
    ("bf16", Dims(1, 12, 12, 6, 5, 4, 32, 2, 2, 2, 6), FORMER, COL),
    ("bf16", Dims(1, 12, 13, 6, 5, 4, 32, 2, 2, 2, 6), FORMER, FORMER),
]


def relerr(a, b):
    a = np.asarray(a.detach().cpu().numpy(), dtype=np.float64)
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(np.asarray(b).ravel()))


def name(mode, kind, precision):
    return f"fno_synth_t_{precision}" if kind == "synth" else f"fno_epi_{mode}_{kind}_{precision}"


@pytest.mark.parametrize("precision,d,fwd,dxk", CASES,
                         ids=[f"{p}-{d.Ci}-{d.Co}x{d.Nx}x{d.Nz}x{d.Nt}" for p, d, _, _ in CASES])
def test_the_rule_names_the_kernel_and_it_matches_the_oracle(precision, d, fwd, dxk):
    from paper_2211_12709_gb300 import _lib, ops
    modes = (d.mx, d.my, d.mz, d.mt)
    x = inputs.normal((d.B, d.Ci) + d.grid, 731)
    w = inputs.spectral_weights(d.Ci, d.Co, d.modes, 732)
    wl, b = inputs.linear_params(d.Ci, d.Co, 733)
    dz = inputs.normal((d.B, d.Co) + d.grid, 734)
    X, W, WL, Bb, DZ = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (x, w, wl, b, dz))
    torch.cuda.synchronize()
    _lib.fno_profile_start()
    z = ops.block_fwd(X, W, WL, Bb, modes, precision)
    torch.cuda.synchronize()
    names = set(_lib.fno_profile_stop())
    assert name("fwd", fwd, precision) in names, sorted(names)
    _lib.fno_profile_start()
    got = ops.block_bwd(X, W, WL, Bb, DZ, modes, precision)
    torch.cuda.synchronize()
    names = set(_lib.fno_profile_stop())
    assert name("dx", dxk, precision) in names, sorted(names)
    rz, _ = oracle.block_fwd(d, x, w, wl, b)
    rg = oracle.block_bwd(d, x, w, dz, wl, b)
    errs = {"z": relerr(z, rz), **{k: relerr(v, rg[k]) for k, v in zip(("dx", "dw", "dwl", "db"), got)}}
    print(errs)
    assert all(v <= TOL[precision] for v in errs.values()), errs
