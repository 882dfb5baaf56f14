"""The half-spectrum Hartree transforms of V_Hxc (csrc/hxc.cu) on grids with odd sides, sides shorter than a tile
and a last row without a partner, against the oracle; and the FP32 density's running sums.

Tolerances: 1e-11 relative for FP64 transforms, as in test_gpu_hxc; the FP32 density's products round by 3 * 2^-24
of the sum of their magnitudes and the running sums add 2^-40 of it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2501_03061_gb300 import api
    c = api.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("dims", [(2, 3, 5), (15, 25, 27), (27, 9, 2), (3, 64, 8), (45, 10, 16), (64, 5, 3), (48, 50, 54)])
def test_potential_and_energies(ctx, dims):
    import torch
    from oracle import ptim_oracle as O
    from paper_2501_03061_gb300 import synth
    nx, ny, nz = dims
    rng = np.random.default_rng(sum(dims))
    cell = synth.Cell(dims, (0.4 * nx, 0.3 * ny, 0.35 * nz))
    g = O.grid_of(cell)
    rho = 10.0 ** rng.uniform(-4, 1.5, (nz, ny, nx))
    rho[0, 0, 0] = 0.0
    rho[-1, -1, -1] = -1e-18
    vloc = rng.standard_normal((nz, ny, nx))
    out, (eh, exc) = ctx.hxc_potential(torch.from_numpy(rho).cuda(), torch.from_numpy(vloc).cuda(), cell=cell, energies=True)
    ref = vloc + O.hxc_potential(rho, g)
    reh, rexc = O.hxc_energy(rho, g)
    assert np.abs(out.cpu().numpy() - ref).max() <= 1e-11 * np.abs(ref).max()
    assert abs(eh - reh) <= 1e-11 * abs(reh) and abs(exc - rexc) <= 1e-11 * abs(rexc)


@pytest.mark.parametrize("N", [1, 3, 4, 9, 70])
def test_fp32_density_sums(ctx, N):
    import torch
    from paper_2501_03061_gb300 import synth
    rng = np.random.default_rng(N)
    cell = synth.Cell((6, 5, 9), (2.0, 2.0, 3.0))
    phi = (rng.standard_normal((N, 9, 5, 6)) + 1j * rng.standard_normal((N, 9, 5, 6))).astype(np.complex64)
    d = rng.uniform(0.1, 1.0, N)
    rho = ctx.density(torch.from_numpy(phi).cuda(), torch.from_numpy(np.diag(d).astype(np.complex128)).cuda(), cell=cell,
                      precision="fp32").cpu().numpy()
    p = np.abs(phi.astype(np.complex128)) ** 2
    ref = 2.0 * np.einsum("j,jzyx->zyx", d, p)
    # chi = phi d rounds the product and d itself: two roundings more
    assert (np.abs(rho - ref) <= (5 * 2.0 ** -24 + 2.0 ** -40) * ref).all()
