"""stats.eig_sweeps of the FP32-form PT-IM step counts all Jacobi sweeps of its sigma eigensolves, the FP32 passes' and
the FP64 ones'."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [24, 48, 95, 97, 110])
def test_sweeps_of_a_step(N):
    """A full random matrix takes more than two sweeps to diagonalise by any cyclic Jacobi method.  Of the passes: cyclic
    Jacobi takes log2 N + 1 or 2 sweeps to FP32 rounding (8 at these sizes), a second pass from off-diagonals of 1e-6 at most
    4, and the FP64 sweeps are left one or two, so 16 a solve at most; a pass that does not converge runs
    to its cap of 12 and leaves the FP64 sweeps the whole work (8 or more: 20)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_03061_gb300 import api, synth
    w = synth.small_cell(700 + N, 16, 5.12, N, kT=0.05)
    rng = np.random.default_rng(N)
    q, _ = np.linalg.qr(rng.standard_normal((N, N)) + 1j * rng.standard_normal((N, N)))
    s = (q / (1.0 + np.exp(np.linspace(-6, 6, N)))) @ q.conj().T
    ctx = api.Context(0)
    try:
        st = ctx.ptim_step(torch.from_numpy(w.phi.astype(np.complex64)).cuda(), torch.from_numpy(0.5 * (s + s.conj().T)).cuda(),
                           torch.from_numpy(w.vloc).cuda(), cell=w.cell, kernel=w.kernel, precision="fp32", dt=0.2, tol=2e-6)
    finally:
        ctx.close()
    assert st["converged"] and st["exchange_calls"] > 0
    assert 3 <= st["eig_sweeps"] <= 16 * st["exchange_calls"]
