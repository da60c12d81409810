"""Launches that overlap at their ends (psatd_launch.cuh): what the kernel ahead
may still be writing is not read through the non-coherent path, and calls queued
back to back on one stream give bit for bit what the same calls give with the
device synchronised after each.  Yee steps queued back to back are no slower
than steps that each find the device idle."""
import os
import re

import pytest
import torch

from paper_1707_08500_gb300 import inputs as I

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1707_08500_gb300", "csrc")


def _function(file, head):
    """A function's text, from its head to the closing brace in column 0."""
    text = open(os.path.join(CSRC, file)).read()
    return text[text.index(head):].split("\n}\n")[0]


@pytest.mark.parametrize("file,head,data", [
    ("psatd_io.cu", "void copy_rows(", ("in", "src")),
    ("psatd_kernels.cuh", "void k_gauss_reduce(", ("part",)),
])
def test_data_of_the_kernel_ahead_is_read_coherently(file, head, data):
    body = _function(file, head)
    for name in data:
        assert not re.search(r"__restrict__\s+%s\b" % name, body), (head, name)
        assert not re.search(r"__ldg\(\s*&?%s\b" % name, body), (head, name)


@pytest.mark.gpu
@pytest.mark.parametrize("n,ng,precision", [((32, 32), 8, "f32"), ((24, 18), 3, "f32"), ((16, 16), 8, "f64")])
def test_queued_calls_equal_synchronised_ones(n, ng, precision):
    """Scatter J and rho, push with the Gauss sums, gather E and B, four times
    over: brief launches (eight boxes of 48^3 and smaller), all of them
    overlapped."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_08500_gb300 import build
    build.build()
    from paper_1707_08500_gb300 import psatd as P
    cuts = (n, n, n)
    wl = I.custom("overlap", (sum(n),) * 3, cuts, ng, 8, fields="wavepacket", precision=precision)
    glob = {k: v.cuda() for k, v in I.global_fields(wl).items()}

    def run(sync):
        sol = P.Solver(wl, gauss=True)
        st = torch.cuda.current_stream().cuda_stream
        src = [glob[k].to(sol.dtype) for k in ("Jx", "Jy", "Jz", "rho")]
        src = [[t * (k + 1) for t in src] for k in range(4)]
        out = [[torch.zeros_like(src[0][0]) for _ in I.EB_NAMES] for _ in range(4)]
        sums = [torch.zeros_like(sol.gauss_out) for _ in range(4)]
        P.psatd_scatter_global(sol.plan, [glob[k].to(sol.dtype) for k in I.EB_NAMES], [sol.arenas[k] for k in I.EB_NAMES], st)
        torch.cuda.synchronize()
        for k in range(4):
            P.psatd_scatter_global(sol.plan, src[k], [sol.arenas[v] for v in ("Jx", "Jy", "Jz", "rho")], st)
            if sync:
                torch.cuda.synchronize()
            P.psatd_push(sol.plan, sol.fields, sums[k].data_ptr(), st)
            if sync:
                torch.cuda.synchronize()
            P.psatd_gather_global(sol.plan, [sol.arenas[v] for v in I.EB_NAMES], out[k], st)
            if sync:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        assert P.psatd_check(sol.plan) == 0
        return [t for o in out for t in o] + sums

    for a, b in zip(run(False), run(True)):
        assert torch.equal(a, b)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [(128, 128, 64), (96, 96, 96)])
def test_queued_yee_steps_are_not_slower_than_single_ones(n):
    """128 and 108 blocks, fewer than SMs: a step whose blocks start early must
    not find them crowded on some SMs (two to an SM take twice as long)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_08500_gb300 import build, fdtd
    build.build()
    s = fdtd.YeeSolver(n, 0.5, precision="f64", device="cuda")
    a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))

    def microseconds(steps):
        a.record()
        for _ in range(steps):
            s.step()
        b.record()
        torch.cuda.synchronize()
        return a.elapsed_time(b) * 1e3 / steps

    microseconds(5)
    single = sorted(microseconds(1) for _ in range(21))[10]
    queued = sorted(microseconds(20) for _ in range(9))[4]
    assert queued < 1.2 * single, (queued, single)


@pytest.mark.gpu
def test_captured_with_other_streams_and_copies():
    """A step captured into a graph between work of other kinds -- copies and
    memsets on its stream, sources spread on a second stream that joins, a step
    of another plan that joins -- replays bit for bit as the calls alone."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_08500_gb300 import build
    build.build()
    from paper_1707_08500_gb300 import psatd as P
    wl = I.custom("capture", (64,) * 3, ((32, 32),) * 3, 8, 8, fields="wavepacket", precision="f32")
    glob = {k: v.cuda().float() for k, v in I.global_fields(wl).items()}
    src = ("Jx", "Jy", "Jz", "rho")

    def fresh():
        sols = [P.Solver(wl, gauss=True) for _ in range(2)]
        for s in sols:
            s.load_global(glob)
        return sols, [torch.zeros_like(glob["Ex"]) for _ in I.EB_NAMES], [glob[k].clone() for k in src]

    def enqueue(sols, out, up, main, side):
        a, b = sols
        up[0].copy_(glob["Jx"])                                        # copies on the main stream
        a.gauss_out.zero_()
        side.wait_stream(main)
        with torch.cuda.stream(side):
            up[1].copy_(glob["Jy"])
            P.psatd_scatter_global(a.plan, up, [a.arenas[k] for k in src], side.cuda_stream)
            b.push(side.cuda_stream)
        main.wait_stream(side)                                         # joins, then the step
        a.push(main.cuda_stream)
        P.psatd_gather_global(a.plan, [a.arenas[k] for k in I.EB_NAMES], out, main.cuda_stream)
        b.push(main.cuda_stream)

    want, out_w, up_w = fresh()
    got, out_g, up_g = fresh()
    main, side = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(main):
        for _ in range(2):
            enqueue(want, out_w, up_w, main, side)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=main):
        enqueue(got, out_g, up_g, torch.cuda.current_stream(), side)
    for _ in range(2):
        g.replay()
    torch.cuda.synchronize()
    for x, y in zip(out_g, out_w):
        assert torch.equal(x, y)
    for s, t in zip(got, want):
        assert P.psatd_check(s.plan) == 0
        assert torch.equal(s.gauss_out, t.gauss_out)
        for k in I.EB_NAMES:
            assert torch.equal(s.arenas[k], t.arenas[k])
