"""Batched persistent form (openfft_plan_many / openfft_exec_many) against the oracle.

Every transform of a batch is compared with the FP64 oracle on its own input:
complex64 plans within 1e-5 relative L2, complex128 (double-float) within
1e-12.  A host-side test hook makes one dependency wait of the persistent
kernel run out; the kernel must report OPENFFT_ERR_TIMEOUT through the status
word and leave the context usable (no trap, no hang).
"""
import numpy as np
import pytest

import oracle
from paper_1501_07350_gb300 import openfft as of
from paper_1501_07350_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    from paper_1501_07350_gb300 import _build
    _build.build()
    of.load()
    assert _t.cuda.is_available()
    return _t


def _inputs(torch, shapes, seed0, dtype):
    tdt = torch.complex64 if dtype == of.C2C_F32 else torch.complex128
    xs = [synth.complex_field(s, seed=seed0 + i) for i, s in enumerate(shapes)]
    xd = [torch.from_numpy(x.reshape(-1)).to("cuda", tdt) for x in xs]
    return xs, xd


def _check_batch(torch, plan, shapes, Ps, xs, xd, dtype, tol):
    yd = [torch.full_like(x, float("nan")) for x in xd]
    of.openfft_set_stream(plan, torch.cuda.current_stream())
    of.openfft_exec_many(plan, xd, yd, of.FORWARD)
    of.openfft_sync(plan)
    for (Na, Nb, Nc), P, x, y in zip(shapes, Ps, xs, yd):
        xin = x.astype(np.complex64).astype(np.complex128) if dtype == of.C2C_F32 else x
        ref = oracle.fft3d(xin, Na, Nb, Nc, P, oracle.FORWARD)
        assert oracle.rel_l2(y.cpu().numpy().astype(np.complex128), ref) < tol, (Na, Nb, Nc)
    zd = [torch.full_like(x, float("nan")) for x in xd]
    of.openfft_exec_many(plan, yd, zd, of.BACKWARD)
    of.openfft_sync(plan)
    for x, z in zip(xd, zd):
        assert float(torch.linalg.vector_norm(z - x) / torch.linalg.vector_norm(x)) < tol


def test_batch_uneven_complex64(torch):
    shapes = synth.batch_shapes(synth.config_seed(4), 12)
    Ps = [8] * len(shapes)
    plan = of.openfft_plan_many(shapes, Ps, of.C2C_F32)
    try:
        xs, xd = _inputs(torch, shapes, synth.config_seed(4) + 1, of.C2C_F32)
        _check_batch(torch, plan, shapes, Ps, xs, xd, of.C2C_F32, 1e-5)
        # second replay with a new pointer set
        xs2, xd2 = _inputs(torch, shapes, 777, of.C2C_F32)
        _check_batch(torch, plan, shapes, Ps, xs2, xd2, of.C2C_F32, 1e-5)
    finally:
        of.openfft_destroy(plan)


def test_batch_complex128_and_generic_lengths(torch):
    # 36, 25, 49 and 14 have no specialised tile body: the generic body runs them
    shapes = [(48, 48, 48), (9, 25, 14), (7, 49, 6), (100, 108, 120), (36, 40, 30), (1, 8, 1)]
    Ps = [8, 7, 42, 8, 64, 1]
    plan = of.openfft_plan_many(shapes, Ps, of.C2C_F64)
    try:
        xs, xd = _inputs(torch, shapes, 4242, of.C2C_F64)
        _check_batch(torch, plan, shapes, Ps, xs, xd, of.C2C_F64, 1e-12)
    finally:
        of.openfft_destroy(plan)
    plan = of.openfft_plan_many(shapes, Ps, of.C2C_F32)
    try:
        xs, xd = _inputs(torch, shapes, 4343, of.C2C_F32)
        _check_batch(torch, plan, shapes, Ps, xs, xd, of.C2C_F32, 1e-5)
    finally:
        of.openfft_destroy(plan)


def test_batch_wait_timeout_is_reported(torch):
    shapes = [(48, 48, 48), (64, 64, 64)]
    Ps = [8, 8]
    plan = of.openfft_plan_many(shapes, Ps, of.C2C_F32)
    try:
        xs, xd = _inputs(torch, shapes, 5, of.C2C_F32)
        yd = [torch.empty_like(x) for x in xd]
        of.openfft_set_stream(plan, torch.cuda.current_stream())
        of.openfft_batch_debug(plan, 1, 2_000_000)       # ~1 ms of clock cycles
        of.openfft_batch_debug(plan, 2, 1)               # a first-stage tile that never comes
        of.openfft_exec_many(plan, xd, yd, of.FORWARD)
        with pytest.raises(of.OpenFFTError) as ei:
            of.openfft_sync(plan)
        assert ei.value.status == of.ERR_TIMEOUT
        # the context is intact: undo the hook and run again
        of.openfft_batch_debug(plan, 2, 0)
        of.openfft_batch_debug(plan, 1, 2_000_000_000)
        _check_batch(torch, plan, shapes, Ps, xs, xd, of.C2C_F32, 1e-5)
    finally:
        of.openfft_destroy(plan)


def test_batch_argument_errors(torch):
    with pytest.raises(of.OpenFFTError) as ei:
        of.openfft_plan_many([(8, 8, 8), (11, 8, 8)], [2, 2], of.C2C_F32)
    assert ei.value.status == of.ERR_UNSUPPORTED_RADIX
    with pytest.raises(of.OpenFFTError) as ei:
        of.openfft_plan_many([(8, 8, 8)], [65], of.C2C_F32)
    assert ei.value.status == of.ERR_P_TOO_LARGE
    plan = of.openfft_plan_many([(8, 8, 8)], [2], of.C2C_F32)
    try:
        x = torch.zeros(512, dtype=torch.complex64, device="cuda")
        with pytest.raises(of.OpenFFTError) as ei:
            of.openfft_exec_many(plan, [x], [x], of.FORWARD)
        assert ei.value.status == of.ERR_ALIAS
        with pytest.raises(of.OpenFFTError):
            of.openfft_exec_c2c(plan, x, torch.zeros_like(x), of.FORWARD)
    finally:
        of.openfft_destroy(plan)


@pytest.mark.parametrize("dtype,tol", [(of.C2C_F32, 1e-5), (of.C2C_F64, 1e-12)])
@pytest.mark.parametrize("shapes", [[(2048, 2, 3), (5, 4, 3)],           # the longest axis: the narrowest tiles
                                    [(448, 6, 10), (12, 500, 9)],        # tiles of 4 lines in double-float
                                    [(16, 16, 16)] * 40])                # more items than CTAs take at once, one tile each
def test_batch_tile_widths(torch, shapes, dtype, tol):
    Ps = [1] * len(shapes)
    plan = of.openfft_plan_many(shapes, Ps, dtype)
    try:
        xs, xd = _inputs(torch, shapes, 99, dtype)
        _check_batch(torch, plan, shapes, Ps, xs, xd, dtype, tol)
    finally:
        of.openfft_destroy(plan)


@pytest.mark.parametrize("dtype,tol", [(of.C2C_F32, 1e-5), (of.C2C_F64, 1e-12)])
def test_plans_of_several_sizes_at_once(torch, dtype, tol):
    """Plans that share a kernel and differ in shared memory, each first run in a
    direction after a smaller or a larger one has been made."""
    Ps = [1]
    batches = [[(100, 108, 120)], [(16, 20, 24)], [(60, 50, 40)], [(2048, 3, 4)], [(1536, 2, 3)]]
    plans = [of.openfft_plan_many(shapes, Ps, dtype) for shapes in batches]
    try:
        for plan, shapes in zip(plans, batches):
            xs, xd = _inputs(torch, shapes, 31, dtype)
            _check_batch(torch, plan, shapes, Ps, xs, xd, dtype, tol)
    finally:
        for plan in plans:
            of.openfft_destroy(plan)


# The kernel of plans with a long axis: tiles of 8, 4, 2 and 1 lines, one, two and four
# groups of threads, fewer tiles than groups, ragged last tiles, fewer lines than a tile.
@pytest.mark.parametrize("dtype,tol", [(of.C2C_F32, 1e-5), (of.C2C_F64, 1e-12)])
@pytest.mark.parametrize("shapes", [[(2048, 9, 5), (30, 36, 40)], [(600, 7, 9), (300, 5, 4), (48, 10, 9), (2, 3, 1)],
                                    [(1, 1792, 6), (375, 3, 30), (360, 7, 2)], [(1024, 10, 3), (21, 500, 1), (1, 1, 700)],
                                    [(96, 1250, 2), (7, 9, 10)] + [(16, 18, 20)] * 30])
def test_long_axes_beside_short_ones(torch, shapes, dtype, tol):
    Ps = [1] * len(shapes)
    plan = of.openfft_plan_many(shapes, Ps, dtype)
    try:
        xs, xd = _inputs(torch, shapes, 51, dtype)
        _check_batch(torch, plan, shapes, Ps, xs, xd, dtype, tol)
    finally:
        of.openfft_destroy(plan)


@pytest.mark.parametrize("dtype", [of.C2C_F32, of.C2C_F64])
def test_a_long_axis_does_not_slow_the_others(torch, dtype):
    """One 2048x48x48 beside 63 48^3 takes no longer than the two as batches of their own
    (and a third of that)."""
    tdt = torch.complex64 if dtype == of.C2C_F32 else torch.complex128

    def best(shapes):
        plan = of.openfft_plan_many(shapes, [1] * len(shapes), dtype)
        try:
            of.openfft_set_stream(plan, torch.cuda.current_stream())
            xs = [torch.randn(int(np.prod(s)), device="cuda", dtype=tdt) for s in shapes]
            ys = [torch.empty_like(x) for x in xs]
            times = []
            for _ in range(12):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                of.openfft_exec_many(plan, xs, ys, of.FORWARD)
                b.record()
                of.openfft_sync(plan)
                torch.cuda.synchronize()
                times.append(a.elapsed_time(b))
            return min(times)
        finally:
            of.openfft_destroy(plan)

    long, short = [(2048, 48, 48)], [(48, 48, 48)] * 63
    assert best(long + short) < 4 / 3 * (best(long) + best(short))


@pytest.mark.parametrize("shape,count,dtype", [((1, 1, 1), 5687, of.C2C_F32), ((3, 3, 3), 5666, of.C2C_F32),
                                               ((1, 1, 1), 5686, of.C2C_F64), ((2048, 1, 1), 3868, of.C2C_F32),
                                               ((2048, 1, 1), 2047, of.C2C_F64)])
def test_the_largest_counts(torch, shape, count, dtype):
    """As many transforms as the queue tables leave room for beside the narrowest tiles."""
    tdt = torch.complex64 if dtype == of.C2C_F32 else torch.complex128
    n = int(np.prod(shape))
    plan = of.openfft_plan_many([shape] * count, [1] * count, dtype)
    try:
        of.openfft_set_stream(plan, torch.cuda.current_stream())
        x = torch.randn((count, n), device="cuda", dtype=tdt)
        y = torch.full_like(x, float("nan"))
        of.openfft_exec_many(plan, list(x), list(y), of.FORWARD)
        of.openfft_sync(plan)
        want = torch.fft.fftn(x.to(torch.complex128).reshape((count,) + shape), dim=(1, 2, 3)).permute(0, 3, 2, 1).reshape(count, n)
        assert float(torch.linalg.vector_norm(y - want) / torch.linalg.vector_norm(want)) < (1e-5 if dtype == of.C2C_F32 else 1e-12)
    finally:
        of.openfft_destroy(plan)
    with pytest.raises(of.OpenFFTError) as ei:
        of.openfft_plan_many([shape] * 6000, [1] * 6000, dtype)
    assert ei.value.status == of.ERR_UNSUPPORTED
