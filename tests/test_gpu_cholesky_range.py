"""The blocked Cholesky factorisation behind the ACE build at the ends of its range: pivots that fail after the first, and
matrices scaled far from one."""
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


def system(N, seed=5):
    """phi, and a matrix A = -<phi|W> that is positive definite, with W = -phi A^T for orthonormal phi."""
    cell = synth.cubic(12, 8.0)
    rng = np.random.default_rng(seed)
    q, _ = np.linalg.qr(rng.standard_normal((cell.ng, N)) + 1j * rng.standard_normal((cell.ng, N)))
    phi = np.ascontiguousarray(q.T) / np.sqrt(cell.dV)
    b = rng.standard_normal((N, N)) + 1j * rng.standard_normal((N, N))
    A = b @ b.conj().T / N + np.eye(N)
    return cell, phi, A


def build(ctx, cell, phi, A):
    W = -(A.T @ phi)  # <phi_i|W_j> = -A_ij
    shape = (-1, 12, 12, 12)
    return ctx.build_ace_from(torch.from_numpy(W.reshape(shape)).cuda(), torch.from_numpy(phi.reshape(shape)).cuda(),
                              cell=cell, precision="fp64")


@pytest.mark.parametrize("scale", [2.0 ** -664, 2.0 ** -400, 2.0 ** 600])
@pytest.mark.parametrize("N", [2, 33])
def test_scaled_matrix(ctx, N, scale):
    """xi of scale W is sqrt(scale) times xi of W: the squares of its columns (2^-1328 and 2^1200) stay
    out of the arithmetic.  A scale that is an even power of two changes no significand; the bound is FP64 rounding
    over N columns of a matrix of condition below 30."""
    cell, phi, A = system(N)
    one = build(ctx, cell, phi, A)
    got = build(ctx, cell, phi, A * scale)
    a, b = one.xi().cpu().numpy(), got.xi().cpu().numpy() / np.sqrt(scale)
    one.close()
    got.close()
    assert np.linalg.norm(a - b) <= 1e-13 * N * np.linalg.norm(a)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("N,p", [(2, 1), (24, 7), (32, 31), (33, 32), (70, 20), (70, 40), (70, 69)])
def test_pivot_after_the_first_fails(ctx, N, p, precision):
    """A = diag(1, .., 1, -1 at p, 1, ..): the factorisation reports pivot p + 1 of whichever block, and the context goes on."""
    from paper_2501_03061_gb300 import api
    cell, phi, _ = system(N)
    d = np.ones(N)
    d[p] = -1.0
    dt = np.complex128 if precision == "fp64" else np.complex64
    shape = (N, 12, 12, 12)
    W = torch.from_numpy((-d[:, None] * phi).astype(dt).reshape(shape)).cuda()
    f = torch.from_numpy(phi.astype(dt).reshape(shape)).cuda()
    with pytest.raises(api.PtimError, match=rf"PT_NOT_PD.*\(pivot {p + 1}\)"):
        ctx.build_ace_from(W, f, cell=cell, precision=precision)
    ok = ctx.build_ace_from(-f, f, cell=cell, precision=precision)
    assert torch.isfinite(torch.view_as_real(ok.xi())).all()
    ok.close()
