"""The 64 x 128 Gram tiles of the tensor-core overlap at the edges of their rings: from one K stage of 32 floats up to more
than the rings hold, a partial last stage, partial and single rows and column halves, an absent second half, and
the Hermitian form's mirrored blocks.

FP32 by three TF32 products: 1e-5 of dV sum_r |a_i| |b_j| an entry (the bound of the other overlap tests)."""
import numpy as np
import pytest

from paper_2501_03061_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_03061_gb300 import api
    c = api.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("n1,n2", [(1, 65), (64, 128), (65, 129), (130, 200), (70, 0), (193, 0)])
@pytest.mark.parametrize("shape", [(2, 2, 4), (3, 5, 6), (4, 6, 9), (20, 20, 18), (36, 36, 36)])
def test_gram_stages(ctx, n1, n2, shape):
    """n2 = 0: the Hermitian overlap of A with itself."""
    cell = synth.Cell(shape, (6.0, 6.5, 7.0))
    gen = np.random.default_rng(1000 * n1 + n2)

    def fields(n):
        return (gen.standard_normal((n, cell.ng)) + 1j * gen.standard_normal((n, cell.ng))).astype(np.complex64)

    A = fields(n1)
    B = fields(n2) if n2 else A
    a = torch.from_numpy(A.reshape(n1, *shape)).cuda()
    b = torch.from_numpy(B.reshape(-1, *shape)).cuda() if n2 else a
    ctx.set_option("tc_gram", 1)
    try:
        got = ctx.overlap(a, b, cell=cell, precision="fp32").cpu().numpy()
    finally:
        ctx.set_option("tc_gram", 0)
    A, B = A.astype(np.complex128), B.astype(np.complex128)
    ref = cell.dV * (A.conj() @ B.T)
    assert np.all(np.abs(got - ref) <= 1e-5 * cell.dV * (np.abs(A) @ np.abs(B).T))
