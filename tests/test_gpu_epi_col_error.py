"""Rounding of the column epilogue's 1x1 on the grids that tcgen05 does not tile.

There its FP32 sums stand in for six products of BF16 parts, whose sums were
short, and run in four chains instead of one.  With w = 0 and A of at least 6, GELU
is the identity in FP32 and z is the 1x1 alone: its rms error has to be at most
three quarters of the one that a single chain of the same products makes on the
same inputs, formed here in numpy (four chains make 0.49 to 0.6 of it).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

# channels and (Nz, Nt): no multiple of 512 points of whole planes, or too wide for tcgen05
CASES = [(32, 32, 16), (28, 32, 16), (24, 8, 16), (20, 8, 16), (20, 4, 32), (24, 20, 32)]


@pytest.mark.parametrize("c,nz,nt", CASES, ids=["x".join(map(str, c)) for c in CASES])
def test_sums_of_the_1x1_run_in_short_chains(c, nz, nt):
    from paper_2211_12709_gb300 import _lib, ops
    grid, modes = (16, 16, nz, nt), (2, 2, min(4, nz // 2), 6)
    n = int(np.prod(grid))
    rng = np.random.default_rng(901)
    x = (1 + rng.random((c, n))).astype(np.float32)
    wl = (0.5 + 0.5 * rng.random((c, c))).astype(np.float32)
    args = (torch.from_numpy(x.reshape((1, c) + grid)).cuda(), torch.zeros(ops._wshape(c, c, modes), device="cuda"),
            torch.from_numpy(wl).cuda(), torch.zeros(c, device="cuda"))
    torch.cuda.synchronize()
    _lib.fno_profile_start()
    z = ops.block_fwd(*args, modes, "bf16x3")
    torch.cuda.synchronize()
    names = _lib.fno_profile_stop()
    assert "fno_epi_fwd_cmma_bf16x3" in names, sorted(names)
    x64, w64 = x.astype(np.float64), wl.astype(np.float64)
    exact = np.einsum("ip,io->op", x64, w64)
    assert exact.min() >= 6
    one = np.zeros((c, n), np.float32)
    for i in range(c):  # fused multiply-adds: products exact in 64 bits, one rounding to 32
        one = (x64[i][None, :] * w64[i][:, None] + one).astype(np.float32)

    def rms(a):
        return float(np.sqrt(np.mean(((a - exact) / exact) ** 2)))

    got, chain = rms(z.cpu().numpy().reshape(c, n).astype(np.float64)), rms(one.astype(np.float64))
    print(got, chain)
    assert got <= 0.75 * chain
