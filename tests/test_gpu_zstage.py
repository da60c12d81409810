"""The FP32 z stage with a mode's block of four positions in registers
(psatd_zpass.cuh) against the FP64 oracle: every compiled z length, planes with
an odd number of modes and a ragged last chunk, the Gauss sums; staggered fields
and mixed lengths (PSATD_PACKED_Z); the heat equation.  Tolerances: one FP32
step, 2e-6 relative L2 (measured 2.5e-7); Gauss sums 1e-5 (measured 1.7e-6): a
sum of squares of i[k].E - rho, whose terms carry the transforms' few 1e-7."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import heat_oracle as H
from oracle import psatd_oracle as O
from paper_1707_08500_gb300 import inputs as I

pytestmark = pytest.mark.gpu
NG = 4


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_08500_gb300 import build
    build.build()
    from paper_1707_08500_gb300 import psatd
    return psatd


def _wl(ycuts, zlens, staggered=False):
    zc = tuple(v - 2 * NG for v in zlens)
    wl = I.custom("z", (14, sum(ycuts), sum(zc)), ((14,), ycuts, zc), NG, 8, fields="wavepacket", c_dt=0.6,
                  precision="f32")
    return dataclasses.replace(wl, staggered=staggered)


def _step(P, wl, flags=0, tuning=None):
    glob = I.global_fields(wl)
    sol = P.Solver(wl, gauss=True, extra_flags=flags, tuning=tuning)
    assert P.psatd_stage_kernels(sol.plan)[0] & (P.PSATD_KERNEL_Z_FLAT if wl.two_d else P.PSATD_KERNEL_Z)
    sol.load_global(glob, guards=True)
    sol.push()
    torch.cuda.synchronize()
    assert P.psatd_check(sol.plan) == 0
    gs = []
    ref = O.step({k: v.numpy() for k, v in glob.items()}, wl, gauss_out=gs)
    assert O.rel_l2({k: v.numpy() for k, v in sol.gather_global().items()}, ref) < 2e-6
    np.testing.assert_allclose(sol.gauss_sums(), np.array(gs), rtol=1e-5)


# local x 22 (12 columns), y 15: 180 modes per plane, 4 in the last chunk of 8
@pytest.mark.parametrize("lz", [32, 48, 64, 80, 96])
@pytest.mark.parametrize("ycuts", [(7,), (8, 5)])
def test_z_lengths(P, lz, ycuts):
    # few items: the flag, which an even number of modes per plane needs
    _step(P, _wl(ycuts, (lz,)), P.PSATD_PACKED_Z)


# odd numbers of modes per plane (117 x 97 and 63 x 61), enough items for the
# stage to be chosen without the flag
@pytest.mark.parametrize("local", [(192, 117, 32), (120, 63, 96)])
def test_odd_modes_per_plane(P, local):
    n = tuple(v - 2 * NG for v in local)
    wl = I.custom("zodd", n, tuple((v,) for v in n), NG, 8, fields="wavepacket", precision="f32")
    assert local[1] * (local[0] // 2 + 1) % 2 == 1
    _step(P, wl)


@pytest.mark.parametrize("zlens,staggered", [((32, 80), False), ((48,), True), ((64, 96), True)])
def test_mixed_lengths_and_stagger(P, zlens, staggered):
    wl = _wl((8,), zlens, staggered)
    assert P.psatd_plane_engine(P.Solver(wl, extra_flags=P.PSATD_PACKED_Z).plan) & 2
    _step(P, wl, P.PSATD_PACKED_Z)


# six modes per item asked for: 14 x 11 and 16 x 11 modes per plane, 4 and 2 of
# them in the last chunk
@pytest.mark.parametrize("zlens,staggered", [((32,), False), ((96,), False), ((48, 80), False), ((64, 96), True)])
def test_six_modes_per_item(P, zlens, staggered):
    zc = tuple(v - 2 * NG for v in zlens)
    wl = I.custom("z6", (12, 14, sum(zc)), ((12,), (6, 8), zc), NG, 8, fields="wavepacket", c_dt=0.6, precision="f32")
    wl = dataclasses.replace(wl, staggered=staggered)
    tuning = {"chunk_b": 6}
    assert P.psatd_stage_kernels(P.Solver(wl, extra_flags=P.PSATD_PACKED_Z, tuning=tuning).plan) == (P.PSATD_KERNEL_Z, 6)
    _step(P, wl, P.PSATD_PACKED_Z, tuning)


@pytest.mark.parametrize("zlens", [(32,), (48, 64), (80, 96)])
@pytest.mark.parametrize("source", [False, True])
@pytest.mark.parametrize("ycuts", [(5,), (8, 7)])
def test_heat(P, zlens, source, ycuts):
    wl = _wl(ycuts, zlens)
    g = I.random_fields(wl.global_n, 3, names=("Jx", "Jy"))
    names = ("T", "S") if source else ("T",)
    hs = P.HeatSolver(wl, 0.4, source=source)
    assert P.psatd_stage_kernels(hs.plan)[0] & P.PSATD_KERNEL_Z
    hs.load_global({"T": g["Jx"], "S": g["Jy"]}, names=names, guards=True)
    hs.push()
    torch.cuda.synchronize()
    ref = H.heat_step({"T": g["Jx"].numpy(), **({"S": g["Jy"].numpy()} if source else {})}, wl, 0.4)["T"]
    assert H.rel_l2(hs.gather_global(names=("T",))["T"].numpy(), ref) < 2e-6


@pytest.mark.parametrize("staggered", [False, True])
@pytest.mark.parametrize("cuts", [((14,), (5,)), ((24, 56), (16, 34, 7))])
def test_one_cell_deep(P, staggered, cuts):
    # 2D problems: Eq. 1 without a z transform; 143 modes in one chunk, then
    # several chunks of 512 and ragged ones
    wl = I.custom("flat", (sum(cuts[0]), sum(cuts[1]), 1), cuts + ((1,),), NG, 8, fields="wavepacket", precision="f32",
                  two_d=True)
    _step(P, dataclasses.replace(wl, staggered=staggered))
