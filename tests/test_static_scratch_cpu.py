"""The sizes that the allocation-free entry takes, checked on the host.

Its limit is FNO_STATIC_SCRATCH_BYTES of the workspace that the call needs; the
basis fragments of the column epilogue (tensor-core precisions, even Nt up to 128)
come on top and are bounded.  No pointer is passed: a call that is not refused for
its size stops at the missing weights, or at the missing GPU.
"""
import ctypes
import random

import pytest

from paper_2211_12709_gb300 import _lib

SCRATCH = 16 << 20
FWD = _lib.FNO_OP_SPECTRAL_FWD
PREC = {"fp32": _lib.FNO_FP32, "tf32": _lib.FNO_TF32, "bf16": _lib.FNO_BF16, "bf16x3": _lib.FNO_BF16X3}


def ws(d, p):
    return _lib.load().fno_workspace_bytes(ctypes.byref(d), p, FWD)


def static_rc(d, p):
    return _lib.load().fno_spectral_fwd_static(ctypes.byref(d), p, None, None, None, None)


@pytest.mark.parametrize("nt", [348, 349, 512, 4096])
def test_long_t_axes_in_fp32_are_taken_and_carry_no_fragments(nt):
    def dims(n):
        return _lib.make_dims(1, 2, 2, 8, 8, 8, n, 2, 2, 2, 4)

    def t_tables(n):  # the four tables of Jt x Nt values
        return 4 * ((8 * 4 * n + 255) // 256 * 256)

    # nothing else of a spectral forward's workspace grows with Nt beyond 128
    assert ws(dims(nt), 0) - ws(dims(200), 0) == t_tables(nt) - t_tables(200)
    assert ws(dims(nt), 0) < SCRATCH
    assert static_rc(dims(nt), 0) in (-1, -4), _lib.fno_last_error()


def test_fragments_are_bounded_and_only_in_the_precisions_that_use_them():
    rng = random.Random(7)
    seen = 0
    for _ in range(3000):
        nz, nt = rng.randint(2, 300), rng.choice([2, 6, 8, 16, 18, 30, 32, 86, 96, 128])
        if nz * nt % 4:
            continue
        d = _lib.make_dims(1, rng.randint(1, 40), rng.randint(1, 40), 4, 4, nz, nt, 1, 1,
                           rng.randint(1, min(32, nz // 2)), rng.randint(1, min(8, nt // 2 + 1)))
        n = {k: ws(d, p) for k, p in PREC.items()}
        if not n["bf16x3"]:
            continue
        assert n["fp32"] == n["tf32"] and n["bf16"] == n["bf16x3"]
        assert 0 <= n["bf16x3"] - n["fp32"] <= 36 << 10
        for k, p in PREC.items():
            assert (static_rc(d, p) == -2) == (n["fp32"] > SCRATCH), (k, n)
        seen += 1
    assert seen > 500
