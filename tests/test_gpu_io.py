"""psatd_scatter_global and psatd_gather_global against index arithmetic in
torch, exactly: widths that are and are not multiples of 16 bytes, boxes that
wrap in x and y, boxes wider than the block of threads, guards wider than the
grid, arrays that start off a 16-byte boundary, both precisions."""

import pytest
import torch

from paper_1707_08500_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_08500_gb300 import build
    build.build()
    from paper_1707_08500_gb300 import psatd
    return psatd


CASES = {
    "aligned": (((24, 40), (16, 32), (5, 4)), 8),
    "odd": (((24, 36), (18, 9), (6,)), 3),
    "guards_off_16_bytes": (((24, 40), (16,), (4,)), 6),
    "wide": (((1096,), (3,), (2,)), 2),
    "rows_of_130_or_260_pieces": (((516,), (9,), (3,)), 2),
    "guards_wider_than_grid": (((4,), (4,), (2,)), 8),
    "one_row": (((32, 32), (1,), (1,)), 0),
}


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("name", list(CASES))
def test_scatter_and_gather(P, name, shift, precision):
    cuts, ng = CASES[name]
    wl = I.custom(name, tuple(sum(c) for c in cuts), cuts, ng, 2, precision=precision)
    sol = P.Solver(wl)
    nx, ny, nz = wl.global_n
    cells = nx * ny * nz

    def array():        # `shift` elements off the allocation's alignment
        return torch.empty(cells + 4, dtype=sol.dtype, device="cuda")[shift:shift + cells].view(nz, ny, nx)

    src = [array().copy_(torch.rand((nz, ny, nx), dtype=torch.float64)) for _ in range(2)]
    P.psatd_scatter_global(sol.plan, src, [sol.arenas["Ex"], sol.arenas["rho"]])
    torch.cuda.synchronize()
    for g, a in zip(src, ("Ex", "rho")):
        for s, sd in enumerate(wl.subs):
            ix, iy, iz = ((torch.arange(sd.local[k], device="cuda") + sd.lo[k] - ng) % wl.global_n[k] for k in range(3))
            assert torch.equal(sol.box(a, s), g[iz][:, iy][:, :, ix]), (a, s)
    out = [array().fill_(-1) for _ in range(2)]
    P.psatd_gather_global(sol.plan, [sol.arenas["Ex"], sol.arenas["rho"]], out)
    torch.cuda.synchronize()
    for g, o in zip(src, out):
        assert torch.equal(g, o)
