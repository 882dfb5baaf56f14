"""FP32 overlaps on CUDA cores over the orbital counts that take each tile (64, 48 or 32 orbitals: one tile, several with a
ragged last one, the Hermitian form's mirrored tiles) and ragged ranges of grid points.

Bound: FP32 products with compensated sums, 1e-5 of dV sum_r |a_i| |b_j| an entry (as for the other overlaps)."""
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


@pytest.mark.parametrize("n1,n2", [(30, 0), (49, 0), (75, 0), (97, 0), (150, 0), (200, 0), (300, 0), (400, 0), (75, 20), (33, 150), (200, 70),
                                   (400, 390)])
@pytest.mark.parametrize("shape", [(12, 12, 12), (15, 16, 18)])
def test_gram_tiles(ctx, n1, n2, shape):
    """n2 = 0: the Hermitian overlap of A with itself, which is exactly Hermitian."""
    cell = synth.Cell(shape[::-1], (6.0, 6.5, 7.0))
    gen = torch.Generator(device="cuda").manual_seed(1000 * n1 + n2)

    def fields(n):
        return torch.view_as_complex(torch.randn(n, *shape, 2, generator=gen, device="cuda"))

    A = fields(n1)
    B = fields(n2) if n2 else A
    got = ctx.overlap(A, B, cell=cell, precision="fp32")
    a, b = A.reshape(n1, -1).to(torch.complex128), B.reshape(B.shape[0], -1).to(torch.complex128)
    assert ((got - cell.dV * (a.conj() @ b.T)).abs() <= 1e-5 * cell.dV * (a.abs() @ b.abs().T)).all()
