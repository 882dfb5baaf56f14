"""The FP32 Jacobi passes in front of the FP64 sweeps of the step's sigma eigensolve (csrc/dense.cu), through FP32-form
steps whose orbital counts take each form of them: one CTA (N <= 96), the whole GPU (N > 96), odd counts with a
padding player, and the boundary between them; and occupation matrices with degenerate and empty clusters.

The FP32 form against the FP64 form of the same step (pinned to the oracle elsewhere), at the bar of the other FP32 steps
(5e-5 on phi and sigma): an eigenbasis that missed its tolerance of 1e-9 by even 1e-4 would change the exchange by
more than that."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2501_03061_gb300 import api
    c = api.Context(0)
    yield c
    c.close()


def sigma_of(kind, N, rng):
    q, _ = np.linalg.qr(rng.standard_normal((N, N)) + 1j * rng.standard_normal((N, N)))
    if kind == "fermi":
        d = 1.0 / (1.0 + np.exp(np.linspace(-6, 6, N)))
    elif kind == "clusters":  # half full to 1e-9 of one another, a quarter empty, the rest spread
        d = np.concatenate([1.0 - 1e-9 * rng.uniform(size=N // 2), np.zeros(N // 4), rng.uniform(0.2, 0.8, N - N // 2 - N // 4)])
    else:  # nearly diagonal already
        return np.diag(np.linspace(1.0, 0.1, N)).astype(np.complex128) + 1e-7 * (lambda m: m + m.conj().T)(
            rng.standard_normal((N, N)) + 1j * rng.standard_normal((N, N)))
    s = (q * d) @ q.conj().T
    return 0.5 * (s + s.conj().T)


@pytest.mark.parametrize("N,kind", [(2, "fermi"), (7, "clusters"), (48, "fermi"), (95, "clusters"), (96, "near"), (97, "fermi"),
                                    (110, "clusters")])
def test_fp32_step_matches_fp64_step(ctx, N, kind):
    import torch
    from paper_2501_03061_gb300 import synth
    w = synth.small_cell(300 + N, 16, 5.12, N, kT=0.05)
    sig = sigma_of(kind, N, np.random.default_rng(N))
    got = {}
    for prec, tol in (("fp32", 2e-6), ("fp64", 1e-9)):
        phi = torch.from_numpy(w.phi.astype(np.complex64 if prec == "fp32" else np.complex128)).cuda()
        s = torch.from_numpy(sig.copy()).cuda()
        st = ctx.ptim_step(phi, s, torch.from_numpy(w.vloc).cuda(), cell=w.cell, kernel=w.kernel, precision=prec, dt=0.2, tol=tol)
        assert st["converged"]
        got[prec] = phi.cpu().numpy().astype(np.complex128), s.cpu().numpy()
    (p32, s32), (p64, s64) = got["fp32"], got["fp64"]
    assert np.linalg.norm(p32 - p64) <= 5e-5 * np.linalg.norm(p64)
    assert np.abs(s32 - s64).max() <= 5e-5
