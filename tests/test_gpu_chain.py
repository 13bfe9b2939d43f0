"""Stages launched as a chain (a stage's CTAs may become resident while the stage
before it drains): results of transforms enqueued back to back, on one stream, on two
and replayed from a captured graph are bit for bit those of transforms run one at a
time.  And the stages with a CTA per tile, against the FP64 oracle (the bar of the other
parity tests, relative L2 <= 1e-12)."""
import numpy as np
import pytest

import oracle
from paper_1501_07350_gb300 import openfft as of
from paper_1501_07350_gb300 import synth

pytestmark = pytest.mark.gpu

# kernels of every family: warp, asynchronous output (256, 512), any length, generic (2048)
SHAPES = [(32, 32, 32), (64, 48, 100), (256, 32, 512), (36, 2048, 5)]


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    from paper_1501_07350_gb300 import _build
    _build.build()
    of.load()
    assert _t.cuda.is_available()
    return _t


@pytest.mark.parametrize("dtype", [of.C2C_F64, of.C2C_F32])
@pytest.mark.parametrize("shape", SHAPES)
def test_chained_transforms_match_single_ones(torch, shape, dtype):
    tdt = torch.complex128 if dtype == of.C2C_F64 else torch.complex64
    n = int(np.prod(shape))
    gen = torch.Generator(device="cuda").manual_seed(n)
    streams = [torch.cuda.Stream() for _ in range(2)]
    plans = [of.Plan(*shape, 2, dtype, stream=s) for s in streams]
    xs = [torch.randn(n, generator=gen, device="cuda", dtype=tdt) for _ in streams]
    bufs = [[torch.empty_like(x) for _ in range(3)] for x in xs]
    torch.cuda.synchronize()

    def steps(i):
        x, (y, z, w) = xs[i], bufs[i]
        return [(x, y, of.FORWARD), (y, z, of.BACKWARD), (z, w, of.FORWARD)]

    want = []
    for i, p in enumerate(plans):
        for a, b, d in steps(i):
            p.exec(a, b, d)
            torch.cuda.synchronize()
        want.append([b.clone() for b in bufs[i]])

    def check():
        torch.cuda.synchronize()
        for i in range(2):
            for b, r in zip(bufs[i], want[i]):
                assert torch.equal(torch.view_as_real(b), torch.view_as_real(r))
                b.fill_(float("nan"))
        torch.cuda.synchronize()

    for _ in range(3):
        for i, p in enumerate(plans):
            for a, b, d in steps(i):
                p.exec(a, b, d)
    check()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=streams[0]):
        for a, b, d in steps(0):
            plans[0].exec(a, b, d)
    for i in range(2):
        for b, r in zip(bufs[i], want[i]):
            b.copy_(r)
    bufs[0][2].fill_(float("nan"))
    torch.cuda.synchronize()
    graph.replay()
    graph.replay()
    check()
    for p in plans:
        p.close()


# 256- and 512-point double-float stages: one to two tiles (3, 5 lines), a ragged last tile
# (126 lines), more tiles than an SM holds CTAs for; transposed and, as the last stage,
# contiguous output (a CTA per line), entry and exit formats in each position.
@pytest.mark.parametrize("n", [256, 512])
@pytest.mark.parametrize("other", [(1, 3), (5, 1), (9, 14), (75, 98)])
def test_a_cta_per_tile(torch, n, other):
    a, b = other
    for shape in ((n, a, b), (a, n, b), (a, b, n)):
        x = synth.complex_field(shape, seed=n)
        xd = torch.from_numpy(np.ascontiguousarray(x.reshape(-1))).to(device="cuda", dtype=torch.complex128)
        plan = of.Plan(*shape, 1, of.C2C_F64)
        try:
            for direction, odir in ((of.FORWARD, oracle.FORWARD), (of.BACKWARD, oracle.BACKWARD)):
                yd = torch.full_like(xd, float("nan"))
                plan.exec(xd, yd, direction)
                torch.cuda.synchronize()
                err = oracle.rel_l2(yd.cpu().numpy(), oracle.fft3d(x, *shape, 1, odir))
                assert err < 1e-12, (shape, direction, err)
        finally:
            plan.close()


# Chains whose stale data is wrong data: two inputs in turn, every buffer filled with NaN
# before its first run, results copied in stream order; then replays of a captured chain
# whose input changes between them, beside work on a second stream.  Real plans run each
# of their last stages: the warp kernels (512 points in float load without staging), the
# generic stage (under 2^15 points) and the any-length kernel.
@pytest.mark.parametrize("shape,dtype", [(s, d) for s in SHAPES for d in (of.C2C_F64, of.C2C_F32)] +
                         [(s, d) for s in ((8, 4, 512), (16, 64, 128), (9, 10, 15), (40, 36, 30), (24, 20, 256))
                          for d in (of.R2C_F64, of.R2C_F32)])
def test_chains_on_changing_inputs(torch, shape, dtype):
    real = dtype in (of.R2C_F64, of.R2C_F32)
    wide = dtype in (of.C2C_F64, of.R2C_F64)
    ct = torch.complex128 if wide else torch.complex64
    n, half = int(np.prod(shape)), shape[0] * shape[1] * (shape[2] // 2 + 1)
    xt = (torch.float64 if wide else torch.float32) if real else ct
    gen = torch.Generator(device="cuda").manual_seed(n)
    xs = [torch.randn(n, generator=gen, device="cuda", dtype=xt) for _ in range(2)]
    streams = [torch.cuda.Stream() for _ in range(2)]
    plans = [of.Plan(*shape, 2, dtype, stream=s) for s in streams]

    def buffers():
        sizes = [(half, ct), (n, xt), (half, ct)] if real else [(n, ct)] * 3
        return [torch.full((m,), float("nan"), device="cuda", dtype=t) for m, t in sizes]

    def steps(plan, x, b):
        if real:
            return [lambda: of.openfft_exec_r2c(plan.handle, x, b[0]), lambda: of.openfft_exec_c2r(plan.handle, b[0], b[1]),
                    lambda: of.openfft_exec_r2c(plan.handle, b[1], b[2])]
        return [lambda: plan.exec(x, b[0], of.FORWARD), lambda: plan.exec(b[0], b[1], of.BACKWARD),
                lambda: plan.exec(b[1], b[2], of.FORWARD)]

    def equal(got, want):
        parts = lambda t: torch.view_as_real(t) if t.is_complex() else t
        return all(torch.equal(parts(g), parts(w)) for g, w in zip(got, want))

    want = []
    for x in xs:
        b = buffers()
        torch.cuda.synchronize()
        for step in steps(plans[0], x, b):
            step()
            torch.cuda.synchronize()
        want.append(b)
    bufs = [buffers() for _ in plans]
    torch.cuda.synchronize()
    got = [[], []]
    for k in range(6):
        for i, p in enumerate(plans):
            for step in steps(p, xs[(k + i) % 2], bufs[i]):
                step()
            with torch.cuda.stream(streams[i]):
                got[i].append([b.clone() for b in bufs[i]])
    torch.cuda.synchronize()
    for i in range(2):
        for k in range(6):
            assert equal(got[i][k], want[(k + i) % 2]), (i, k)
    x, b = xs[0].clone(), buffers()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=streams[0]):
        for step in steps(plans[0], x, b):
            step()
    got, beside = [], []
    for k in range(4):
        with torch.cuda.stream(streams[0]):
            x.copy_(xs[k % 2])
            graph.replay()
            got.append([t.clone() for t in b])
        for step in steps(plans[1], xs[1 - k % 2], bufs[1]):
            step()
        with torch.cuda.stream(streams[1]):
            beside.append([t.clone() for t in bufs[1]])
    torch.cuda.synchronize()
    for k in range(4):
        assert equal(got[k], want[k % 2]) and equal(beside[k], want[1 - k % 2]), k
    for p in plans:
        p.close()


# The allocation-free call writes its twiddle tables ahead of its stages on every call, at
# one place for all lengths: calls of different lengths back to back, on lengths whose
# kernels read the tables where they are (warp kernels) and whose kernels copy them.
@pytest.mark.parametrize("dtype", [of.C2C_F64, of.C2C_F32])
def test_noalloc_calls_of_different_lengths_back_to_back(torch, dtype):
    tdt = torch.complex128 if dtype == of.C2C_F64 else torch.complex64
    shapes = [(64, 64, 64), (128, 64, 32), (32, 256, 64), (64, 48, 100), (128, 32, 128), (36, 40, 30)]
    gen = torch.Generator(device="cuda").manual_seed(3)
    xs = [torch.randn(int(np.prod(s)), generator=gen, device="cuda", dtype=tdt) for s in shapes]
    stream = torch.cuda.current_stream()

    def run(shape, x, direction):
        y = torch.full_like(x, float("nan"))
        of.openfft_exec_c2c_noalloc(*shape, 1, dtype, x, y, direction, stream)
        return y

    calls = [(s, x, d) for s, x in zip(shapes, xs) for d in (of.FORWARD, of.BACKWARD)]
    want = []
    for c in calls:
        torch.cuda.synchronize()
        want.append(run(*c))
    torch.cuda.synchronize()
    got = [run(*c) for _ in range(3) for c in calls]
    torch.cuda.synchronize()
    for k, g in enumerate(got):
        assert torch.equal(torch.view_as_real(g), torch.view_as_real(want[k % len(calls)])), calls[k % len(calls)][0]
