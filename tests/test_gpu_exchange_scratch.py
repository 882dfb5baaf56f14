"""The FP32 exchange in a context whose HBM budget holds one field per pair of a symmetric application, N (N + 1)/2 of them,
and little else: it runs, on smaller tiles, and with less it is refused."""
import numpy as np
import pytest

from paper_2501_03061_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KERNEL = {"type": 1, "mu": synth.SCREENED_MU}


@pytest.mark.parametrize("n,nz,N", [(24, 24, 40), (24, 20, 21), (64, 64, 5), (16, 16, 2), (16, 16, 1)])
def test_budget_of_one_field_per_pair(n, nz, N):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_03061_gb300 import api
    cell = synth.Cell((n, n, nz), (0.3 * n, 0.3 * n, 0.3 * nz))
    rng = np.random.default_rng(N)
    src = torch.from_numpy((rng.standard_normal((N, nz, n, n)) + 1j * rng.standard_normal((N, nz, n, n))).astype(np.complex64)).cuda()
    occ = torch.linspace(1, 0, N + 1, dtype=torch.float64)[:N].cuda()

    def run(budget, batched=False):
        ctx = api.Context(0, budget)
        try:
            if batched:
                call = [{"src": src, "occ": occ, "cell": cell, "kernel": KERNEL, "out": torch.empty_like(src)}]
                for _ in range(2):
                    out = ctx.apply_exchange_batched(call, precision="fp32")[0][0]
                return out
            for _ in range(2):
                out = ctx.apply_exchange(src, occ, cell=cell, kernel=KERNEL, precision="fp32")
            return out
        finally:
            ctx.close()

    pairs = N * (N + 1) // 2 * cell.ng * 8
    ref = run(0)
    for batched in (False, True):
        out = run(pairs + 4096, batched)
        # the same pair fields, summed tile by tile
        assert torch.linalg.norm(out - ref) <= 1e-6 * torch.linalg.norm(ref)
    with pytest.raises(api.PtimError, match="PT_OOM"):
        run(pairs - 4096)


def test_budget_of_a_batch():
    """Four branches, each with the fields of its largest item's pairs: every branch finds its room."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_03061_gb300 import api
    rng = np.random.default_rng(8)
    calls, pairs = [], 0
    for n, N in ((24, 40), (30, 30), (32, 28), (20, 50)):
        src = torch.from_numpy((rng.standard_normal((N, n, n, n)) + 1j * rng.standard_normal((N, n, n, n))).astype(np.complex64)).cuda()
        calls.append({"src": src, "occ": torch.linspace(1, 0.1, N, dtype=torch.float64).cuda(), "cell": synth.cubic(n, 0.3 * n),
                      "kernel": KERNEL, "out": torch.empty_like(src)})
        pairs += N * (N + 1) // 2 * n ** 3 * 8
    got = []
    for budget in (0, pairs + (64 << 10)):
        ctx = api.Context(0, budget)
        try:
            for _ in range(2):
                outs = ctx.apply_exchange_batched(calls, precision="fp32")[0]
            got.append([o.clone() for o in outs])
        finally:
            ctx.close()
    for a, b in zip(*got):
        assert torch.linalg.norm(a - b) <= 1e-6 * torch.linalg.norm(a)
