"""The FP32 density where a partial sum of its products leaves the FP32 range: the sums are those of FP64."""
import numpy as np
import pytest

from paper_2501_03061_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [3, 8, 21])
def test_sums_beyond_fp32(N):
    """|phi|^2 = 1.96e38 an orbital: two of them exceed 3.4e38.  A few points also hold a negative weight, so that a sum
    leaves the range and comes back; bound: the FP32 rounding of each product, twice 2^-24 of sum |terms|."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_03061_gb300 import api
    cell = synth.Cell((6, 5, 4), (2.0, 2.0, 2.0))
    rng = np.random.default_rng(N)
    phi = (1.4e19 * np.exp(2j * np.pi * rng.uniform(size=(N, cell.ng)))).astype(np.complex64)
    phi[:, ::3] *= 1e-19  # ordinary points among them
    w = np.where(rng.uniform(size=N) < 0.3, -1.0, 1.0)
    ctx = api.Context(0)
    try:
        rho = ctx.density(torch.from_numpy(phi.reshape(N, 4, 5, 6)).cuda(), torch.from_numpy(np.diag(w).astype(np.complex128)).cuda(),
                          cell=cell, precision="fp32", spin=2.0).cpu().numpy().reshape(-1)
    finally:
        ctx.close()
    terms = 2.0 * w[:, None] * np.abs(phi.astype(np.complex128)) ** 2
    assert np.isfinite(rho).all()
    assert np.all(np.abs(rho - terms.sum(0)) <= 2 * 2.0 ** -24 * np.abs(terms).sum(0))
