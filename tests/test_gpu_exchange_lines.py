"""The FP32 line kernels of the exchange (csrc/exchange_lines.cu) against the oracle on every cubic side:
ragged pair tiles, separate targets, empty occupations, a cell with three different side lengths, and
both forms of the last pass (one and four groups of threads per column).

Tolerance (relative Frobenius): six line transforms of at most 64 points and the products around them
round each value at most 6 * 6 + 4 times by 2^-24, 2.4e-6."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIDES = [16, 20, 24, 30, 32, 36, 40, 48, 54, 60, 64]
TOL = 40 * 2.0 ** -24


@pytest.fixture(scope="module")
def ctx():
    from paper_2501_03061_gb300 import api
    c = api.Context(0)
    yield c
    c.close()


def run(ctx, cell, src, occ, tgt, tile, kernel):
    import torch

    def dev(a):
        return torch.from_numpy(np.ascontiguousarray(a)).cuda()

    for key in ("scratch_bytes", "exchange64_scratch_bytes"):
        ctx.set_option(key, tile * tile * cell.ng * 8)
    try:
        out = ctx.apply_exchange(dev(src.astype(np.complex64)), dev(occ), None if tgt is None else dev(tgt.astype(np.complex64)),
                                 cell=cell, kernel=kernel, precision="fp32")
    finally:
        for key in ("scratch_bytes", "exchange64_scratch_bytes"):
            ctx.set_option(key, 512 << 20)
    return out.cpu().numpy().astype(np.complex128)


@pytest.mark.parametrize("N,M,tile", [(1, 0, 1), (5, 0, 2), (7, 3, 3), (6, 0, 8)])
@pytest.mark.parametrize("n", SIDES)
def test_lines_match_oracle(ctx, n, N, M, tile):
    from oracle import ptim_oracle as O
    from paper_2501_03061_gb300 import synth
    rng = np.random.default_rng(40 + 7 * n + N)
    cell = synth.Cell((n, n, n), (0.32 * n, 0.29 * n, 0.35 * n))
    src = rng.standard_normal((N, n, n, n)) + 1j * rng.standard_normal((N, n, n, n))
    tgt = rng.standard_normal((M, n, n, n)) + 1j * rng.standard_normal((M, n, n, n)) if M else None
    src = src.astype(np.complex64).astype(np.complex128)
    tgt = tgt.astype(np.complex64).astype(np.complex128) if M else None
    occ = np.linspace(1.0, 0.1, N)
    if N > 4:
        occ[[1, 4]] = 0.0
    kernel = {"type": 0} if tile == 3 else {"type": 1, "mu": synth.SCREENED_MU}
    K = O.exchange_kernel(O.grid_of(cell), kernel["type"], synth.SCREENED_MU)
    ref = O.apply_exchange(src, occ, src if tgt is None else tgt, K)
    out = run(ctx, cell, src, occ, tgt, tile, kernel)
    assert np.linalg.norm(out - ref) <= TOL * np.linalg.norm(ref)


LENGTHS = [16, 18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64]


@pytest.mark.parametrize("k", range(len(LENGTHS)))
@pytest.mark.parametrize("N,M,tile", [(4, 0, 3), (3, 5, 8)])
def test_axes_match_oracle(ctx, k, N, M, tile):
    """Grids that are not cubic: every length on every axis, odd products among them."""
    from oracle import ptim_oracle as O
    from paper_2501_03061_gb300 import synth
    rng = np.random.default_rng(900 + k)
    nx, ny, nz = LENGTHS[k], LENGTHS[(k + 5) % 16], LENGTHS[(k + 11) % 16]
    cell = synth.Cell((nx, ny, nz), (0.3 * nx, 0.34 * ny, 0.32 * nz))
    src = rng.standard_normal((N, nz, ny, nx)) + 1j * rng.standard_normal((N, nz, ny, nx))
    tgt = rng.standard_normal((M, nz, ny, nx)) + 1j * rng.standard_normal((M, nz, ny, nx)) if M else None
    src = src.astype(np.complex64).astype(np.complex128)
    tgt = tgt.astype(np.complex64).astype(np.complex128) if M else None
    occ = np.linspace(1.0, 0.0, N)
    kernel = {"type": 1, "mu": synth.SCREENED_MU}
    K = O.exchange_kernel(O.grid_of(cell), 1, synth.SCREENED_MU)
    ref = O.apply_exchange(src, occ, src if tgt is None else tgt, K)
    out = run(ctx, cell, src, occ, tgt, tile, kernel)
    assert np.linalg.norm(out - ref) <= TOL * np.linalg.norm(ref)


@pytest.mark.parametrize("n,N", [(16, 70), (24, 40), (36, 30), (48, 18), (60, 14)])
def test_one_group_per_column(ctx, n, N):
    """Enough targets that the last pass runs one group of threads per column; the tile kernels
    (exchange64_engine 1), pinned to the oracle elsewhere, give the reference: both round as above."""
    from paper_2501_03061_gb300 import synth
    rng = np.random.default_rng(n)
    cell = synth.cubic(n, 0.32 * n)
    src = rng.standard_normal((N, n, n, n)) + 1j * rng.standard_normal((N, n, n, n))
    occ = rng.uniform(0.1, 1.0, N)
    occ[::9] = 0.0
    kernel = {"type": 1, "mu": synth.SCREENED_MU}
    out = run(ctx, cell, src, occ, None, 1 << 10, kernel)
    ctx.set_option("exchange64_engine", 1)
    try:
        ref = run(ctx, cell, src, occ, None, 1 << 10, kernel)
    finally:
        ctx.set_option("exchange64_engine", 0)
    assert np.linalg.norm(out - ref) <= 2 * TOL * np.linalg.norm(ref)


def test_empty_occupations_and_nonfinite_empty_orbital(ctx):
    """All occupations zero give zero; an orbital that is exactly empty contributes nothing even where it
    is not finite and is not its own target."""
    from paper_2501_03061_gb300 import synth
    n = 24
    rng = np.random.default_rng(5)
    cell = synth.cubic(n, 0.32 * n)
    src = (rng.standard_normal((4, n, n, n)) + 1j * rng.standard_normal((4, n, n, n))).astype(np.complex64)
    tgt = src[:2].copy()
    kernel = {"type": 1, "mu": synth.SCREENED_MU}
    assert not run(ctx, cell, src, np.zeros(4), None, 8, kernel).any()
    occ = np.array([1.0, 0.0, 0.5, 0.0])
    ref = run(ctx, cell, src, occ, tgt, 8, kernel)
    src[1] = np.nan
    src[3] = np.inf
    assert np.array_equal(run(ctx, cell, src, occ, tgt, 8, kernel), ref)
