"""The tensor-core rotation's operand rings: few stages (fewer than the rings are deep), a partial last
stage, one column up to a partial second column tile, and enough point tiles that a CTA walks several.
FP32 inputs with TF32 triple products: 1e-5 of sum_k |A_k| |B_kj| per point (the bound of the dropped
lo * lo terms, 2^-22 a product, with FP32 accumulation over at most 2 x 49 terms)."""
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


@pytest.mark.parametrize("n1,n2", [(1, 1), (16, 64), (17, 65), (33, 3), (49, 130)])
@pytest.mark.parametrize("shape", [(8, 9, 10), (36, 36, 36)])
def test_rotate_stages(ctx, n1, n2, shape):
    cell = synth.Cell(shape, (6.0, 6.5, 7.0))
    gen = np.random.default_rng(1000 * n1 + n2)
    A = gen.standard_normal((n1, cell.ng)) + 1j * gen.standard_normal((n1, cell.ng))
    B = gen.standard_normal((n1, n2)) + 1j * gen.standard_normal((n1, n2))
    A = A.astype(np.complex64)
    a = torch.from_numpy(A.reshape(n1, *shape)).cuda()
    ctx.set_option("tc_gram", 1)
    try:
        got = ctx.rotate(a, torch.from_numpy(B).cuda(), cell=cell, precision="fp32").cpu().numpy().reshape(n2, -1)
    finally:
        ctx.set_option("tc_gram", 0)
    ref = B.T @ A.astype(np.complex128)
    scale = np.abs(B).T @ np.abs(A.astype(np.complex128))
    assert np.all(np.abs(got - ref) <= 1e-5 * scale)
