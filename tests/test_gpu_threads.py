"""Calls of several host threads, each with its own stream, workspace and size.

Kernels that need more than 48 KB of shared memory have their limit raised before
the launch, per kernel and not per thread: a call of one size must not fail or
change because another thread calls with a smaller one.
"""
import threading

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

# (Nz, Nt) pairs whose kernels are the same and whose shared memory differs
SIZES = {"fp32": [(130, 16), (240, 16), (180, 16), (64, 16)], "bf16x3": [(128, 32), (16, 32), (64, 32), (32, 32)]}


@pytest.mark.parametrize("precision", sorted(SIZES))
def test_threads_with_different_sizes_do_not_disturb_each_other(precision):
    from paper_2211_12709_gb300 import ops
    c, rounds = 12, 1500
    jobs = []
    for n, (nz, nt) in enumerate(SIZES[precision]):
        g = torch.Generator(device="cuda")
        g.manual_seed(n)
        modes = (1, 1, 8, 8)
        x = torch.randn((1, c, 2, 2, nz, nt), device="cuda", generator=g)
        w = torch.randn(ops._wshape(c, c, modes), device="cuda", generator=g)
        wl = torch.randn((c, c), device="cuda", generator=g)
        b = torch.randn((c,), device="cuda", generator=g)
        ws = ops.workspace(ops.dims_of(x, c, modes), precision, ops.OP_BLOCK_FWD, x.device)
        jobs.append((x, w, wl, b, modes, ws, ops.block_fwd(x, w, wl, b, modes, precision)))
    torch.cuda.synchronize()
    start, errors, outs = threading.Barrier(len(jobs)), [], [None] * len(jobs)

    def work(n):
        x, w, wl, b, modes, ws, _ = jobs[n]
        stream = torch.cuda.Stream()
        try:
            with torch.cuda.stream(stream):
                start.wait(60)
                for _ in range(rounds):
                    outs[n] = ops.block_fwd(x, w, wl, b, modes, precision, ws=ws)
            stream.synchronize()
        except Exception as e:  # noqa: BLE001 - reported below
            errors.append(f"{SIZES[precision][n]}: {e}")

    threads = [threading.Thread(target=work, args=(n,)) for n in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for job, out in zip(jobs, outs):
        assert torch.equal(job[-1], out)
