"""FP32 stages with one axis length compiled in -- the row and column launches of
the split-plane schedule and the z stage of long axes -- against the FP64 oracle:
every compiled length, row blocks and column blocks with remainders, chunks with
a ragged end, guards, a length that is not compiled beside one that is.
Tolerances: one FP32 step, 2e-6 relative L2 (measured 2.6e-7); Gauss sums 1e-5
(measured 5.5e-7; squares of i[k].E - rho, whose terms carry the transforms' few
1e-7)."""
import numpy as np
import pytest
import torch

from oracle import psatd_oracle as O
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


@pytest.mark.parametrize("local,ng,split", [
    ((128, 20, 6), 2, True), ((192, 9, 5), 0, True), ((256, 33, 3), 0, True), ((384, 18, 4), 1, True), ((512, 7, 3), 0, True),
    ((40, 128, 4), 1, True), ((36, 192, 5), 2, True), ((64, 256, 3), 0, True),
    ((12, 10, 128), 2, False), ((14, 9, 192), 0, False), ((10, 13, 256), 3, False), ((128, 128, 128), 0, True),
])
def test_compiled_axis_lengths(P, local, ng, split):
    n = tuple(v - 2 * ng for v in local)
    wl = I.custom("long", n, tuple((v,) for v in n), ng, 8, fields="wavepacket", precision="f32", c_dt=0.6)
    glob = I.global_fields(wl)
    sol = P.Solver(wl, gauss=True, extra_flags=P.PSATD_SPLIT_PLANES if split else 0)
    want = P.PSATD_KERNEL_Z_LONG if local[2] >= 128 else 0
    if split:
        want |= P.PSATD_KERNEL_SPLIT | (P.PSATD_KERNEL_ROWS_X if local[0] >= 128 else 0) | \
            (P.PSATD_KERNEL_COLS_Y if local[1] >= 128 else 0)
    assert P.psatd_stage_kernels(sol.plan)[0] & ~P.PSATD_KERNEL_PLANES == want
    sol.load_global(glob, guards=True)
    sol.push()
    torch.cuda.synchronize()
    assert P.psatd_check(sol.plan) == 0
    gs = []
    ref = O.step({k: v.numpy() for k, v in glob.items()}, wl, gauss_out=gs)
    assert O.rel_l2({k: v.numpy() for k, v in sol.gather_global().items()}, ref) < 2e-6
    np.testing.assert_allclose(sol.gauss_sums(), np.array(gs), rtol=1e-5)
