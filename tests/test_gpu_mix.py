"""The stage kernel of the lengths without one of their own (csrc/fft_mix.cuh), on
the GPU against the FP64 oracle: every radix it is compiled for in first, middle and
last passes, lines shorter and longer than a CTA's threads cover in one round,
ragged tiles (90 lines in tiles of 4 or 8), each axis position, both directions.

Bars as for every other parity test: relative L2 <= 1e-12 for complex128 plans,
<= 1e-5 for complex64 against the oracle on the same input upcast."""
import numpy as np
import pytest

import oracle
from paper_1501_07350_gb300 import openfft as of
from paper_1501_07350_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = {of.C2C_F64: 1e-12, of.C2C_F32: 1e-5}


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    from paper_1501_07350_gb300 import _build
    _build.build()
    of.load()
    assert _t.cuda.is_available()
    return _t


def _exec(torch, plan, x, direction, dtype):
    tdt = torch.complex128 if dtype == of.C2C_F64 else torch.complex64
    xd = torch.from_numpy(np.ascontiguousarray(x.reshape(-1))).to(device="cuda", dtype=tdt)
    yd = torch.full_like(xd, float("nan"))
    of.openfft_set_stream(plan, torch.cuda.current_stream())
    of.openfft_exec_c2c(plan, xd, yd, direction)
    of.openfft_sync(plan)
    return yd.cpu().numpy().astype(np.complex128)


# one pass (2..10, 12, 15), two (16 9, 15 15, 10 10), three (8 6 6, 7 7 7), many (243 = 3^5),
# odd lengths, and the longest that fit a tile
LENGTHS = [2, 3, 5, 6, 7, 9, 10, 12, 15, 18, 20, 28, 45, 49, 63, 72, 75, 80, 90, 105, 120, 126, 144, 160, 189, 210, 225,
           240, 243, 288, 320, 343, 384, 420, 448, 500, 625, 750, 1000, 1250, 1792, 2000]


@pytest.mark.parametrize("dtype", [of.C2C_F64, of.C2C_F32])
@pytest.mark.parametrize("n", LENGTHS)
def test_every_radix_and_position(torch, n, dtype):
    for shape in ((n, 9, 10), (10, n, 9), (9, 10, n)):
        x = synth.complex_field(shape, seed=n)
        xin = x if dtype == of.C2C_F64 else x.astype(np.complex64).astype(np.complex128)
        plan = of.openfft_plan(*shape, 1, dtype)
        try:
            for direction, odir in ((of.FORWARD, oracle.FORWARD), (of.BACKWARD, oracle.BACKWARD)):
                ref = oracle.fft3d(xin, *shape, 1, odir)
                err = oracle.rel_l2(_exec(torch, plan, x, direction, dtype), ref)
                assert err < TOL[dtype], (shape, direction, err)
        finally:
            of.openfft_destroy(plan)


@pytest.mark.parametrize("shape", [(36, 10, 48), (9, 25, 14), (256, 6, 80)])
def test_complex64_arrays_at_8_byte_addresses(torch, shape):
    """complex64 arrays that start 8 bytes off a 16-byte boundary (a view into a larger
    tensor): the copies of a line then take 8 bytes at a time."""
    n = int(np.prod(shape))
    x = synth.complex_field(shape, seed=n).astype(np.complex64)
    plan = of.openfft_plan(*shape, 1, of.C2C_F32)
    try:
        of.openfft_set_stream(plan, torch.cuda.current_stream())
        for off_in, off_out in ((1, 0), (0, 1), (1, 1)):
            xd = torch.empty(n + 1, dtype=torch.complex64, device="cuda")[off_in:off_in + n]
            xd.copy_(torch.from_numpy(x.reshape(-1)))
            yd = torch.full((n + 1,), float("nan"), dtype=torch.complex64, device="cuda")[off_out:off_out + n]
            for direction, odir in ((of.FORWARD, oracle.FORWARD), (of.BACKWARD, oracle.BACKWARD)):
                ref = oracle.fft3d(x.astype(np.complex128), *shape, 1, odir)
                of.openfft_exec_c2c(plan, xd, yd, direction)
                of.openfft_sync(plan)
                assert oracle.rel_l2(yd.cpu().numpy().astype(np.complex128), ref) < TOL[of.C2C_F32]
    finally:
        of.openfft_destroy(plan)


# The factor 1 / N is applied in two parts: a sum that overflows in the last butterfly of a
# backward transform (the first value of a constant array, 4e38 before the factor) stays
# infinite.  Powers of two (no second part) and other lengths (of either sign).
@pytest.mark.parametrize("shape", [(64, 48, 100), (36, 10, 48), (256, 32, 32), (30, 28, 36), (9, 25, 14)])
def test_overflow_stays_infinite(torch, shape):
    n = int(np.prod(shape))
    plan = of.openfft_plan(*shape, 1, of.C2C_F32)
    try:
        y = _exec(torch, plan, np.full(n, 4e38 / n, dtype=np.complex64), of.BACKWARD, of.C2C_F32)
        assert y[0].real == np.inf, y[0]
    finally:
        of.openfft_destroy(plan)


# Double-float grids: as many CTAs as tiles (more than the SMs hold), and fewer (each CTA
# takes several), in the same transform: 29160 to 45000 lines in tiles of 4.
def test_grids_of_several_waves(torch):
    shape = (250, 180, 162)
    x = synth.complex_field(shape, seed=7)
    plan = of.openfft_plan(*shape, 1, of.C2C_F64)
    try:
        for direction, odir in ((of.FORWARD, oracle.FORWARD), (of.BACKWARD, oracle.BACKWARD)):
            err = oracle.rel_l2(_exec(torch, plan, x, direction, of.C2C_F64), oracle.fft3d(x, *shape, 1, odir))
            assert err < TOL[of.C2C_F64], (direction, err)
    finally:
        of.openfft_destroy(plan)
