"""Occupations that are not ordinary numbers in the FP32 exchange: a NaN belongs to the result, an exactly empty orbital
does not, whatever form the accumulate pass takes (sums in registers, shared memory and tensor memory, one and
four groups per column, cubic and other grids, one tile of pairs and several)."""
import numpy as np
import pytest

from paper_2501_03061_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KERNEL = {"type": 1, "mu": synth.SCREENED_MU}


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_03061_gb300 import api
    c = api.Context(0)
    yield c
    c.close()


def block(n, shape, seed):
    rng = np.random.default_rng(seed)
    a = rng.standard_normal((n, *shape)) + 1j * rng.standard_normal((n, *shape))
    return torch.from_numpy(a.astype(np.complex64)).cuda()


@pytest.mark.parametrize("targets", [0, 3])
@pytest.mark.parametrize("nx,ny,nz,N", [(16, 16, 16, 5), (16, 16, 16, 130), (24, 24, 24, 5), (24, 24, 24, 60), (64, 64, 64, 3),
                                        (64, 64, 64, 9), (16, 20, 64, 4), (24, 20, 18, 4)])
def test_nan_occupation_reaches_every_target(ctx, nx, ny, nz, N, targets):
    """d_i = NaN makes every term d_i src_i v_ij NaN, so every point of every target."""
    cell = synth.Cell((nx, ny, nz), (0.3 * nx, 0.3 * ny, 0.3 * nz))
    src = block(N, (nz, ny, nx), N)
    tgt = block(targets, (nz, ny, nx), 77) if targets else None
    occ = np.linspace(1.0, 0.2, N)
    occ[0] = 0.0
    ref = ctx.apply_exchange(src, torch.from_numpy(occ).cuda(), tgt, cell=cell, kernel=KERNEL, precision="fp32")
    assert torch.isfinite(torch.view_as_real(ref)).all()
    occ[1] = np.nan
    for tile in (256, 2):
        ctx.set_option("scratch_bytes", tile * tile * cell.ng * 8)
        ctx.set_option("exchange64_scratch_bytes", tile * tile * cell.ng * 8)
        try:
            out = ctx.apply_exchange(src, torch.from_numpy(occ).cuda(), tgt, cell=cell, kernel=KERNEL, precision="fp32")
        finally:
            ctx.set_option("scratch_bytes", 512 << 20)
            ctx.set_option("exchange64_scratch_bytes", 512 << 20)
        assert torch.isnan(torch.view_as_real(out)).all()


def test_nan_occupation_fails_the_ace_build(ctx):
    from paper_2501_03061_gb300 import api
    cell = synth.cubic(24, 8.0)
    occ = torch.tensor([1.0, float("nan"), 0.5, 0.2], dtype=torch.float64).cuda()
    with pytest.raises(api.PtimError, match="PT_NOT_PD"):
        ctx.build_ace(block(4, (24, 24, 24), 3), occ, cell=cell, kernel=KERNEL, precision="fp32")


@pytest.mark.parametrize("n", [16, 24, 64])
@pytest.mark.parametrize("empty", [0.0, -0.0, 1e-60])
def test_empty_orbital_is_left_out(ctx, n, empty):
    """An occupation that is zero, or zero in FP32, contributes nothing even where its orbital is not finite."""
    cell = synth.cubic(n, 0.3 * n)
    src, tgt = block(3, (n, n, n), n), block(2, (n, n, n), n + 1)
    occ = torch.tensor([1.0, 0.0, 0.5], dtype=torch.float64).cuda()
    ref = ctx.apply_exchange(src, occ, tgt, cell=cell, kernel=KERNEL, precision="fp32")
    src[1] = float("inf")
    occ[1] = empty
    assert torch.equal(ctx.apply_exchange(src, occ, tgt, cell=cell, kernel=KERNEL, precision="fp32"), ref)
