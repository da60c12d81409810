"""psatd_stage_kernels reports the kernels that a plan's push launches (host
only): the z stages that are chosen without a flag, and the lengths compiled in
for the split-plane schedule."""
import pytest

from paper_1707_08500_gb300 import build, inputs as I


@pytest.fixture(scope="module")
def P():
    build.build()
    from paper_1707_08500_gb300 import psatd
    return psatd


def boxes(P, count, local, flags, ng=4, tuning=None, two_d=False):
    """stage_kernels of `count` boxes along x of the given local lengths."""
    n = [v - 2 * ng for v in local[:2]] + [1 if two_d else local[2] - 2 * ng]
    wl = I.custom("k", (n[0] * count, n[1], n[2]), ((n[0],) * count, (n[1],), (n[2],)), ng, 8, two_d=two_d)
    h = P.psatd_plan_create(wl.global_n, wl.subs, flags | (P.PSATD_2D if two_d else 0), tuning)
    try:
        return P.psatd_stage_kernels(h)
    finally:
        P.psatd_destroy(h)


def test_z_stage(P):
    F, K = P.PSATD_F32, P
    assert boxes(P, 8, (96, 96, 96), F) == (K.PSATD_KERNEL_PLANES | K.PSATD_KERNEL_Z, 8)
    assert boxes(P, 8, (96, 96, 96), F | P.PSATD_GENERIC_PLANES) == (0, 8)
    assert boxes(P, 8, (48, 48, 48), P.PSATD_F64) == (0, 4)
    # one box of 64^3 is too few items for k_pass_z, unless asked for it
    assert boxes(P, 1, (64, 64, 64), F) == (K.PSATD_KERNEL_PLANES, 8)
    assert boxes(P, 1, (64, 64, 64), F | P.PSATD_PACKED_Z) == (K.PSATD_KERNEL_PLANES | K.PSATD_KERNEL_Z, 8)
    # a chunk width asked for is the one that runs
    assert boxes(P, 1, (64, 64, 64), F | P.PSATD_PACKED_Z, tuning={"chunk_b": 6}) == (K.PSATD_KERNEL_PLANES | K.PSATD_KERNEL_Z, 6)
    assert boxes(P, 8, (96, 96, 96), F, tuning={"chunk_b": 8}) == (K.PSATD_KERNEL_PLANES | K.PSATD_KERNEL_Z, 8)
    assert boxes(P, 8, (96, 96, 96), F, tuning={"chunk_b": 6}) == (K.PSATD_KERNEL_PLANES, 6)
    # not for staggered fields, other lengths or chunks; the heat equation always
    assert boxes(P, 8, (96, 96, 96), F | P.PSATD_STAGGERED)[0] == K.PSATD_KERNEL_PLANES
    assert boxes(P, 8, (96, 96, 88), F)[0] == K.PSATD_KERNEL_PLANES
    assert boxes(P, 8, (96, 96, 96), F, tuning={"chunk_b": 4}) == (K.PSATD_KERNEL_PLANES, 4)
    assert boxes(P, 1, (30, 30, 32), F | P.PSATD_HEAT) == (K.PSATD_KERNEL_Z, 16)
    assert boxes(P, 1, (30, 30, 36), F | P.PSATD_HEAT)[0] == 0
    assert boxes(P, 2, (30, 30, 1), F, two_d=True)[0] == K.PSATD_KERNEL_Z_FLAT
    assert boxes(P, 1, (30, 30, 192), F) == (K.PSATD_KERNEL_Z_LONG, 4)


def test_few_items_are_counted_per_launch(P):
    """Eight boxes of 64^3 are enough items for k_pass_z in one launch; in the
    plain schedule, one launch a box, they are not, while boxes of 96^3 are."""
    F = P.PSATD_F32
    for size, flags, z in ((64, 0, True), (64, P.PSATD_PLAIN, False), (80, P.PSATD_PLAIN, False), (96, P.PSATD_PLAIN, True)):
        k = boxes(P, 8, (size,) * 3, F | flags)[0]
        assert bool(k & P.PSATD_KERNEL_Z) == z, (size, flags)
    assert boxes(P, 8, (64,) * 3, F | P.PSATD_PLAIN | P.PSATD_PACKED_Z)[0] & P.PSATD_KERNEL_Z


def test_split_planes(P):
    F, K, S = P.PSATD_F32, P, P.PSATD_KERNEL_SPLIT
    assert boxes(P, 1, (256, 256, 256), F, ng=0)[0] == S | K.PSATD_KERNEL_ROWS_X | K.PSATD_KERNEL_COLS_Y | K.PSATD_KERNEL_Z_LONG
    assert boxes(P, 1, (128, 60, 30), F | P.PSATD_SPLIT_PLANES)[0] == S | K.PSATD_KERNEL_ROWS_X
    assert boxes(P, 1, (60, 192, 30), F | P.PSATD_SPLIT_PLANES)[0] == S | K.PSATD_KERNEL_COLS_Y
    assert boxes(P, 1, (256, 256, 30), P.PSATD_F64)[0] == S
