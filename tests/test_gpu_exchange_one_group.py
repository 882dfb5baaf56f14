"""The accumulate pass of the FP32 exchange with one group of threads per column, in every place its sums live (registers for
z lines up to 20 points, shared memory, tensor memory at 64) and with a last CTA that is partly past the grid's columns.

The pass takes four groups while a tile's warps, 2 per 64 columns and target, are fewer than 6 to an SM; the cases have more,
which the test asserts from the SM count.  A few targets are compared with the oracle: FP32 to 1e-5."""
import numpy as np
import pytest

from oracle import ptim_oracle as O
from paper_2501_03061_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_03061_gb300 import api
    c = api.Context(0)
    c.set_option("scratch_bytes", 2 << 30)  # one tile of pairs in every case
    yield c
    c.close()


# registers; shared memory; tensor memory; the same on grids that are not cubic, 300 to 540 columns
CASES = [(16, 16, 16, 118), (20, 20, 20, 68), (24, 24, 24, 53), (64, 64, 64, 9), (16, 20, 18, 95), (20, 27, 20, 53), (20, 16, 24, 95),
         (18, 25, 45, 60), (20, 24, 60, 60), (18, 18, 64, 80), (20, 25, 64, 60)]


@pytest.mark.parametrize("symmetric", [True, False])
@pytest.mark.parametrize("nx,ny,nz,N", CASES)
def test_one_group(ctx, nx, ny, nz, N, symmetric):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert N * ((nx * ny + 63) // 64) * 2 >= 6 * sms
    cell = synth.Cell((nx, ny, nz), (0.3 * nx, 0.34 * ny, 0.32 * nz))
    rng = np.random.default_rng(N + nz)
    targets = (rng.standard_normal((N, nz, ny, nx)) + 1j * rng.standard_normal((N, nz, ny, nx))).astype(np.complex64)
    src = targets if symmetric else targets[:4].copy()
    occ = rng.uniform(0.1, 1.0, src.shape[0])
    occ[1] = 0.0
    kernel = {"type": 1, "mu": synth.SCREENED_MU}
    dev = torch.from_numpy(targets).cuda()
    out = ctx.apply_exchange(dev if symmetric else torch.from_numpy(src).cuda(), torch.from_numpy(occ).cuda(),
                             None if symmetric else dev, cell=cell, kernel=kernel, precision="fp32").cpu().numpy()
    some = [0, 1, N // 2, N - 1]
    ref = O.apply_exchange(src.astype(np.complex128), occ, targets[some].astype(np.complex128),
                           O.exchange_kernel(O.grid_of(cell), 1, synth.SCREENED_MU))
    assert np.linalg.norm(out[some] - ref) <= 1e-5 * np.linalg.norm(ref)
