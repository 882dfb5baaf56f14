"""pt_rotate in the default FP32 form works on the caller's buffers alone: it holds no workspace, so calls of one context
on different streams are independent and the first call can be captured.  Its B operand is rounded to FP32 as a
conversion does."""
import numpy as np
import pytest

from paper_2501_03061_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture()
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_03061_gb300 import api
    c = api.Context(0)
    yield c
    c.close()


def inputs(n1, n2, seed, n=12):
    g = torch.Generator(device="cuda").manual_seed(seed)
    A = torch.randn(n1, n, n, n, 2, generator=g, device="cuda")
    B = torch.randn(n1, n2, 2, generator=g, device="cuda", dtype=torch.float64)
    return torch.view_as_complex(A), torch.view_as_complex(B)


def test_no_workspace_and_rounding_of_b(ctx):
    """A one-orbital block of ones copies B out: bit for bit the FP32 rounding of its FP64 values, ties, denormal
    results, zeros and values next to the ends of the FP32 range among them."""
    one = np.float64(1.0)
    rng = np.random.default_rng(1)
    edge = [0.0, -0.0, one + 2.0 ** -24, one + 3 * 2.0 ** -24, one + 2.0 ** -24 + 2.0 ** -52, 2 - 2.0 ** -24, 3.4028234e38,
            2.0 ** -126, 2.0 ** -126 * (1 - 2.0 ** -24), 2.0 ** -127, 2.0 ** -149, 2.0 ** -150, 3 * 2.0 ** -150, 1e-300,
            5e-324]
    v = np.concatenate([edge, np.negative(edge), rng.standard_normal(4000) * 10.0 ** rng.uniform(-44, 37, 4000)])
    cell = synth.cubic(2, 1.0)
    A = torch.ones(1, 2, 2, 2, dtype=torch.complex64).cuda()
    for part in (1.0, 1j):
        B = torch.from_numpy((part * v).astype(np.complex128).reshape(1, -1)).cuda()
        out = ctx.rotate(A, B, cell=cell, precision="fp32")
        got = out[:, 1, 0, 1].cpu().numpy()
        want = v.astype(np.float32)
        assert np.array_equal(got.real if part == 1.0 else got.imag, want)
    assert ctx.workspace_bytes() == 0


@pytest.mark.parametrize("n1,n2", [(1, 1), (15, 31), (16, 32), (17, 33), (75, 75), (40, 61), (200, 70)])
def test_matches_torch(ctx, n1, n2):
    """Edges of the tile in both orbital counts; FP32 sums of n1 products against FP64."""
    A, B = inputs(n1, n2, 10 * n1 + n2)
    cell = synth.cubic(12, 5.0)
    out = ctx.rotate(A, B, cell=cell, precision="fp32").reshape(n2, -1)
    a = A.reshape(n1, -1).to(torch.complex128)
    bound = 2.0 ** -23 * (n1 + 4) * (B.abs().T @ a.abs())
    assert ((out - B.T @ a).abs() <= bound).all()
    assert ctx.workspace_bytes() == 0


@pytest.mark.parametrize("n1", [128, 129])
def test_prepared_operand(ctx, n1):
    """Inside an ACE application B comes converted from 129 terms on: -xi (xi^* psi) with xi = phi for W = -phi."""
    cell = synth.cubic(12, 5.0)
    q = torch.linalg.qr(inputs(cell.ng, n1, n1)[1])[0].T / np.sqrt(cell.dV)
    phi = q.reshape(n1, 12, 12, 12).to(torch.complex64).contiguous()
    psi = inputs(33, 1, 5)[0].contiguous()
    ace = ctx.build_ace_from(-phi, phi, cell=cell, precision="fp32")
    out = ctx.apply_ace(ace, psi).reshape(33, -1)
    ace.close()
    p = psi.reshape(33, -1).to(torch.complex128)
    ref = -cell.dV * (q.conj() @ p.T).T @ q
    # FP32 phi, xi (a triangular solve of the identity to 1e-7) and two contractions of n1 and ng terms
    assert torch.linalg.norm(out - ref) <= 1e-5 * torch.linalg.norm(ref)


def test_first_call_under_capture(ctx):
    cell = synth.cubic(12, 5.0)
    A, B = inputs(20, 30, 3)
    out = torch.empty(30, 12, 12, 12, dtype=torch.complex64, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ctx.rotate(A, B, cell=cell, precision="fp32", out=out)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, ctx.rotate(A, B, cell=cell, precision="fp32"))


def test_two_streams(ctx):
    """Rotations of one context in flight on two streams give what each gives alone."""
    n = 32
    cell = synth.cubic(n, 10.0)
    pairs = [inputs(48, 48, s, n) for s in (1, 2)]
    alone = [ctx.rotate(A, B, cell=cell, precision="fp32") for A, B in pairs]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in pairs]
    outs = [[torch.empty_like(a) for _ in range(20)] for a in alone]
    torch.cuda.synchronize()
    for k in range(20):
        for s, (A, B), o in zip(streams, pairs, outs):
            ctx.rotate(A, B, cell=cell, precision="fp32", out=o[k], stream=s)
    torch.cuda.synchronize()
    for a, o in zip(alone, outs):
        assert all(torch.equal(a, x) for x in o)
