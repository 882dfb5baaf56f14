"""V_Hxc under stream capture and back to back: its passes are launched dependent on one another, inside a graph too, and
calls that follow each other at once on one stream, on small grids, give what each gives alone."""
import pytest

from paper_2501_03061_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(5, 5, 5), (60, 3, 4), (24, 20, 18), (64, 64, 32), (64, 64, 64)])
def test_captured_and_back_to_back(shape):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_03061_gb300 import api
    cell = synth.Cell(shape, (6.0, 6.5, 7.0))
    gen = torch.Generator(device="cuda").manual_seed(1)
    rho = [torch.rand(*shape[::-1], generator=gen, device="cuda", dtype=torch.float64) for _ in range(6)]
    ctx = api.Context(0)
    try:
        alone = []
        for r in rho:
            alone.append(ctx.hxc_potential(r, None, cell=cell))
            torch.cuda.synchronize()
        row = [ctx.hxc_potential(r, None, cell=cell) for r in rho]
        outs = [torch.zeros_like(r) for r in rho]
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            for r, o in zip(rho, outs):
                ctx.hxc_potential(r, None, cell=cell, out=o)
        g.replay()
        torch.cuda.synchronize()
        for a, b, c in zip(alone, row, outs):
            assert torch.equal(a, b) and torch.equal(a, c)
    finally:
        ctx.close()
