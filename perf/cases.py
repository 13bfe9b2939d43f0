"""The transforms that performance is measured on: sizes, inputs, one pass, and
the exact results, through the package's public entry points.

A case names a kind of call and its sizes:
  c2c    openfft_exec_c2c on a plan (complex128 or complex64, one direction)
  r2c    openfft_exec_r2c (real abc array -> half spectrum in cba order)
  c2r    openfft_exec_c2r (half spectrum -> real abc array)
  batch  openfft_exec_many (several transforms of uneven sizes in one call)
  nd     openfft_nd_exec (4-D and 5-D transforms)
`bits` is the width of one real number (64: complex128 / double, 32: complex64
/ float).  Plans use the default tuning, as a caller gets them.
"""
import math

import torch

from paper_1501_07350_gb300 import openfft as of


def listed():
    return [
        # the smallest configuration: a call is three short launches, so its
        # time is launch latency and the host path (small grids in a loop of
        # time steps)
        {"name": "c128_32cubed_fwd", "kind": "c2c", "dims": "32x32x32", "P": 4, "bits": 64, "dir": "fwd"},
        # a small ragged single-precision grid, inverse: lengths of three
        # different kernels, P that divides nothing
        {"name": "c64_64x48x100_bwd", "kind": "c2c", "dims": "64x48x100", "P": 33, "bits": 32, "dir": "bwd"},
        # the ordinary double-precision grid, both directions: a spectral
        # solver's forward transform and the inverse that follows it
        {"name": "c128_256cubed_fwd", "kind": "c2c", "dims": "256x256x256", "P": 64, "bits": 64, "dir": "fwd"},
        {"name": "c128_256cubed_bwd", "kind": "c2c", "dims": "256x256x256", "P": 16, "bits": 64, "dir": "bwd"},
        # the same grid in single precision
        {"name": "c64_256cubed_fwd", "kind": "c2c", "dims": "256x256x256", "P": 64, "bits": 32, "dir": "fwd"},
        # the largest configuration: 2.1 GB each way
        {"name": "c128_512cubed_fwd", "kind": "c2c", "dims": "512x512x512", "P": 256, "bits": 64, "dir": "fwd"},
        # the mixed-radix configuration
        {"name": "c128_120x144x160_fwd", "kind": "c2c", "dims": "120x144x160", "P": 32, "bits": 64, "dir": "fwd"},
        # its doubled grid, lengths with no kernel of their own, inverse
        {"name": "c128_240x288x320_bwd", "kind": "c2c", "dims": "240x288x320", "P": 64, "bits": 64, "dir": "bwd"},
        # the batched configuration: 64 uneven transforms in one call
        {"name": "batch64_c64_fwd", "kind": "batch", "dims": "48x48x48,64x64x64,96x96x96,100x108x120", "count": 64,
         "P": 8, "bits": 32, "dir": "fwd"},
        # real data, double precision: the forward transform of a real field
        {"name": "r2c_f64_256cubed", "kind": "r2c", "dims": "256x256x256", "P": 64, "bits": 64, "dir": "fwd"},
        # real data, single precision, the inverse, on a grid of odd lengths
        {"name": "c2r_f32_180x200x225", "kind": "c2r", "dims": "180x200x225", "P": 32, "bits": 32, "dir": "bwd"},
        # a 4-D transform, inverse
        {"name": "nd_c64_64x36x40x48_bwd", "kind": "nd", "dims": "64x36x40x48", "P": 16, "bits": 32, "dir": "bwd"},
    ]


def _lengths(lo, hi):
    """Every axis length in [lo, hi] the library transforms (factors 2, 3, 5, 7)."""
    out = []
    for n in range(lo, hi + 1):
        m = n
        for f in (2, 3, 5, 7):
            while m % f == 0:
                m //= f
        if m == 1:
            out.append(n)
    return out


def _draw_dims(rng, ndim, lo_points, hi_points):
    """ndim axis lengths of 8..512 whose product is log-uniform in the range;
    half of the axes are powers of two, as in practice."""
    powers = [8, 16, 32, 64, 128, 256, 512]
    smooth = _lengths(8, 512)
    target = math.exp(rng.uniform(math.log(lo_points), math.log(hi_points)))
    for _ in range(200):
        dims = []
        left = target
        for i in range(ndim):
            want = left ** (1.0 / (ndim - i)) * math.exp(rng.uniform(-0.5, 0.5))
            pool = powers if rng.random() < 0.5 else smooth
            dims.append(min(pool, key=lambda n: abs(math.log(n / want)) + 0.15 * rng.random()))
            left = max(1.0, left / dims[-1])
        if lo_points / 2 <= math.prod(dims) <= hi_points:
            return dims
    return [32] * ndim


def draw(rng):
    kind = rng.choices(["c2c", "r2c", "c2r", "batch", "nd"], [10, 2, 2, 1, 1])[0]
    bits = rng.choice([64, 32])
    direction = rng.choice(["fwd", "bwd"])
    if kind == "batch":
        count = rng.randint(4, 48)
        shapes = [_draw_dims(rng, 3, 24 ** 3, 128 ** 3) for _ in range(rng.randint(2, 4))]
        return {"kind": kind, "dims": ",".join("x".join(map(str, s)) for s in shapes), "count": count, "P": 8,
                "bits": bits, "dir": direction}
    if kind == "nd":
        dims = _draw_dims(rng, rng.choice([4, 4, 5]), 2 ** 15, 2 ** 25)
    else:
        dims = _draw_dims(rng, 3, 2 ** 14, 2 ** 27)
    if kind == "r2c":
        direction = "fwd"
    elif kind == "c2r":
        direction = "bwd"
    # P up to the limit of every ordering of these sizes, 1024 at most
    half = [n // 2 + 1 for n in dims] if kind in ("r2c", "c2r") else list(dims)
    limit = min(half) ** 2
    P = int(round(math.exp(rng.uniform(0.0, math.log(min(1024, limit))))))
    return {"kind": kind, "dims": "x".join(map(str, dims)), "P": max(1, P), "bits": bits, "dir": direction}


# ------------------------------------------------------------------ inputs --

def _dims(text):
    return tuple(int(v) for v in text.split("x"))


def _shapes(case):
    """The shape of every transform of a batched case, cycling through the list."""
    menu = [_dims(t) for t in case["dims"].split(",")]
    return [menu[i % len(menu)] for i in range(case["count"])]


def _real_type(case):
    return torch.float64 if case["bits"] == 64 else torch.float32


def _complex_type(case):
    return torch.complex128 if case["bits"] == 64 else torch.complex64


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _decay(shape):
    """Amplitude of a smooth field's spectrum at every frequency of `shape`."""
    r2 = torch.zeros((), device="cuda", dtype=torch.float64)
    for i, n in enumerate(shape):
        k = torch.fft.fftfreq(n, device="cuda", dtype=torch.float64)
        r2 = r2 + (k * k).reshape([n if j == i else 1 for j in range(len(shape))])
    return 1.0 / (1.0 + 64.0 * r2)


def _field(shape, case, gen):
    """Input of one complex transform: a standard normal field forward, a
    decaying spectrum (stored with its axes reversed) backward."""
    n = math.prod(shape)
    x = torch.view_as_complex(torch.randn((n, 2), generator=gen, device="cuda", dtype=_real_type(case)))
    if case["dir"] == "bwd":
        rev = tuple(reversed(shape))
        x = x.reshape(rev).mul_((math.sqrt(n) * _decay(rev)).to(_real_type(case))).reshape(-1)
    return x


def _inputs(case, seed):
    gen = _generator(seed)
    kind = case["kind"]
    if kind == "batch":
        return [_field(s, case, gen) for s in _shapes(case)]
    shape = _dims(case["dims"])
    if kind in ("c2c", "nd"):
        return [_field(shape, case, gen)]
    x = torch.randn(shape, generator=gen, device="cuda", dtype=_real_type(case))
    if kind == "r2c":
        return [x.reshape(-1)]
    # the half spectrum of a real field, cba order
    half = torch.fft.rfftn(x.to(torch.float64)).permute(2, 1, 0).contiguous()
    return [half.to(_complex_type(case)).reshape(-1)]


# -------------------------------------------------------------- the passes --

class _State:
    """What a program keeps between calls: inputs, outputs and the plan, which
    is destroyed with the state."""

    def __init__(self, call, inputs, outputs, release):
        self.call, self.inputs, self.outputs, self._release = call, inputs, outputs, release

    def __del__(self):
        try:
            torch.cuda.synchronize()
            self._release()
        except Exception:
            pass


def prepare(case, seed):
    kind, bits = case["kind"], case["bits"]
    direction = of.FORWARD if case["dir"] == "fwd" else of.BACKWARD
    xs = _inputs(case, seed)
    if kind == "batch":
        shapes = _shapes(case)
        plan = of.openfft_plan_many(shapes, [case["P"]] * len(shapes), of.C2C_F64 if bits == 64 else of.C2C_F32)
        of.openfft_set_stream(plan, torch.cuda.current_stream())
        ys = [torch.empty_like(x) for x in xs]
        return _State(lambda: of.openfft_exec_many(plan, xs, ys, direction), xs, ys,
                      lambda: of.openfft_destroy(plan))
    x = xs[0]
    shape = _dims(case["dims"])
    if kind == "nd":
        y = torch.empty_like(x)
        plan = of.openfft_nd_plan(shape, case["P"], of.C2C_F64 if bits == 64 else of.C2C_F32)
        of.openfft_nd_set_stream(plan, torch.cuda.current_stream())
        return _State(lambda: of.openfft_nd_exec(plan, x, y, direction), xs, [y], lambda: of.openfft_nd_destroy(plan))
    Na, Nb, Nc = shape
    if kind == "c2c":
        y = torch.empty_like(x)
        plan = of.Plan(Na, Nb, Nc, case["P"], of.C2C_F64 if bits == 64 else of.C2C_F32)
        return _State(lambda: plan.exec(x, y, direction), xs, [y], plan.close)
    plan = of.Plan(Na, Nb, Nc, case["P"], of.R2C_F64 if bits == 64 else of.R2C_F32)
    if kind == "r2c":
        y = torch.empty((Nc // 2 + 1) * Nb * Na, device="cuda", dtype=_complex_type(case))
        return _State(lambda: of.openfft_exec_r2c(plan.handle, x, y), xs, [y], plan.close)
    y = torch.empty(Na * Nb * Nc, device="cuda", dtype=_real_type(case))
    return _State(lambda: of.openfft_exec_c2r(plan.handle, x, y), xs, [y], plan.close)


def run(state):
    state.call()
    return state.outputs


# ------------------------------------------------------ the least of a pass --

def work(case):
    """Each input read once, each output written once; 5 N log2 N operations
    per complex transform, half of that per real one."""
    shapes = _shapes(case) if case["kind"] == "batch" else [_dims(case["dims"])]
    real = case["kind"] in ("r2c", "c2r")
    E = case["bits"] // 4
    nbytes = flops = 0
    for s in shapes:
        n = math.prod(s)
        nbytes += n * E // 2 + n // s[-1] * (s[-1] // 2 + 1) * E if real else 2 * n * E
        flops += (2.5 if real else 5.0) * n * math.log2(n)
    return {"bytes": nbytes, "flops": flops}


# -------------------------------------------------------------------- exact --

def exact(case, seed):
    """The transforms of the same inputs by torch.fft in 64 bits."""
    out = []
    kind = case["kind"]
    shapes = _shapes(case) if kind == "batch" else [_dims(case["dims"])]
    for x, shape in zip(_inputs(case, seed), shapes):
        rev = tuple(reversed(range(len(shape))))
        if kind == "r2c":
            y = torch.fft.rfftn(x.reshape(shape).to(torch.float64)).permute(rev)
        elif kind == "c2r":
            Na, Nb, Nc = shape
            h = x.reshape(Nc // 2 + 1, Nb, Na).to(torch.complex128).permute(rev)
            h = torch.fft.ifft(torch.fft.ifft(h, dim=0), dim=1)
            y = torch.fft.irfft(h, n=Nc, dim=2)
        elif case["dir"] == "fwd":
            y = torch.fft.fftn(x.reshape(shape).to(torch.complex128)).permute(rev)
        else:
            y = torch.fft.ifftn(x.reshape(tuple(reversed(shape))).to(torch.complex128).permute(rev).contiguous())
        out.append(y.contiguous().reshape(-1))
    return out
