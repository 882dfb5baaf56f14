"""Batched exchange after its workspace has grown: a captured graph holds the addresses of the workspace it was recorded
with, so it is recorded anew once a larger call has replaced a buffer."""
import numpy as np
import pytest

from paper_2501_03061_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KERNEL = {"type": 1, "mu": synth.SCREENED_MU}


@pytest.fixture()
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_03061_gb300 import api
    c = api.Context(0)
    yield c
    c.close()


def item(n, N, seed):
    rng = np.random.default_rng(seed)
    src = torch.from_numpy((rng.standard_normal((N, n, n, n)) + 1j * rng.standard_normal((N, n, n, n))).astype(np.complex64)).cuda()
    return {"src": src, "occ": torch.linspace(1, 0.1, N, dtype=torch.float64).cuda(), "cell": synth.cubic(n, 0.3 * n),
            "kernel": KERNEL, "out": torch.empty_like(src)}


@pytest.mark.parametrize("streams", [1, 4])
@pytest.mark.parametrize("larger", ["batch", "single"])
def test_small_batch_after_a_larger_call(ctx, streams, larger):
    ctx.set_option("batch_streams", streams)
    small = [item(24, 6, 1), item(20, 5, 2)]
    big = [item(30, 40, 3 + k) for k in range(2)]
    first = [o.clone() for o in ctx.apply_exchange_batched(small, precision="fp32")[0]]
    again, _, nodes = ctx.apply_exchange_batched(small, precision="fp32")
    assert nodes > 0 and all(torch.equal(a, b) for a, b in zip(first, again))
    held = ctx.workspace_bytes()
    if larger == "batch":
        ctx.apply_exchange_batched(big, precision="fp32")
    else:
        ctx.apply_exchange(big[0]["src"], big[0]["occ"], cell=big[0]["cell"], kernel=KERNEL, precision="fp32")
    assert ctx.workspace_bytes() > held
    other = torch.zeros(64 << 20, dtype=torch.uint8, device="cuda")  # takes what the context gave back, if anything did
    for _ in range(2):
        for it in small:
            it["out"].zero_()
        outs, _, nodes = ctx.apply_exchange_batched(small, precision="fp32")
        torch.cuda.synchronize()
        assert nodes > 0 and all(torch.equal(a, b) for a, b in zip(first, outs))
    assert not other.any()
