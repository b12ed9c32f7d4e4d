"""Performance cases: the transforms a user of libfftu runs, through the Python binding of the C ABI.

A case is a plain dict:
  kind       "transform"  one fftu_exec, or a forward and an inverse one
             "convolve"   fftu_exec_pointwise: forward, product in the frequency domain, inverse
             "batch"      fftu_batch_exec: many transforms of different shapes in one launch
  shape      "512x512x512"; of a batch "32x64x32 64x64x64 ..."
  grid       the cyclic grid p, "8x8x8", or "default" for the planner's
  dtype      "c64" or "c128"
  direction  "forward", "inverse", or "both" (forward, then the inverse of its result)
  inplace    in == out (with "both": the array is transformed there and back)
  precision  "native", "bf16" or "fp16" (radix-16 stages as split tensor-core contractions, complex64)
  layout     "natural" or "cyclic" (processor-major storage)
  inputs     "uniform" (real and imaginary parts in [-1, 1)) or "loguniform" (magnitudes 1e-3 to 1e3)
"""
import math

import torch

import paper_2203_11795_gb300 as fftu

_TORCH = {"c64": torch.complex64, "c128": torch.complex128}
_BYTES = {"c64": 8, "c128": 16}
_PRECISION = {"native": fftu.FFTU_PREC_NATIVE, "bf16": fftu.FFTU_PREC_SPLIT_BF16, "fp16": fftu.FFTU_PREC_SPLIT_FP16}
_LAYOUT = {"natural": fftu.FFTU_LAYOUT_NATURAL, "cyclic": fftu.FFTU_LAYOUT_CYCLIC}


def _case(name=None, kind="transform", shape="", grid="default", dtype="c64", direction="forward", inplace=False,
          precision="native", layout="natural", inputs="uniform"):
    c = {"kind": kind, "shape": shape, "grid": grid, "dtype": dtype, "direction": direction, "inplace": inplace,
         "precision": precision, "layout": layout, "inputs": inputs}
    return c if name is None else {"name": name, **c}


def _text(shape):
    return "x".join(str(v) for v in shape)


def _shape(text):
    return tuple(int(v) for v in text.split("x"))


def _shapes(case):
    return [_shape(t) for t in case["shape"].split()]


def _uneven(rng, count):
    """Shapes of an uneven batch: 3D, each side 32, 64 or 128."""
    return " ".join(_text(rng.choice((32, 64, 128)) for _ in range(3)) for _ in range(count))


def listed():
    import random
    return [
        # the smallest request of a serving mix: launches and latency count
        _case("cube32_c64", shape="32x32x32"),
        # double precision on a small cube, the smallest workload that the library is checked on at p = 2 x 2 x 2
        _case("cube64_c128_p2", shape="64x64x64", grid="2x2x2", dtype="c128"),
        # one 2D image of a serving mix, back from the frequency domain
        _case("plane1024_c64_inverse", shape="1024x1024", direction="inverse"),
        # an ordinary cube whose array is transformed in place, there and back (no second array)
        _case("cube128_c64_inplace", shape="128x128x128", direction="both", inplace=True),
        # one split-step propagation or convolution step: forward, product, inverse
        _case("convolve256_c64", kind="convolve", shape="256x256x256"),
        # 64 uneven transforms of ragged shapes in one persistent launch
        _case("batch64_uneven_c64", kind="batch", shape=_uneven(random.Random(2024), 64)),
        # five dimensions, short sub-FFTs on every axis
        _case("tensor32x5_c64", shape="32x32x32x32x32"),
        # four dimensions in double precision
        _case("tensor64x4_c128", shape="64x64x64x64", dtype="c128"),
        # the headline workload: 1 GiB array, forward and inverse
        _case("cube512_c64_p8", shape="512x512x512", grid="8x8x8", direction="both"),
        # the same array with its radix-16 stages on the tensor cores, inputs over six decades
        _case("cube512_bf16_loguniform", shape="512x512x512", grid="8x8x8", precision="bf16", inputs="loguniform"),
        # two dimensions with long lines
        _case("plane16384_c64", shape="16384x16384"),
        # the largest array: 8 GiB
        _case("cube1024_c64_p8", shape="1024x1024x1024", grid="8x8x8"),
    ]


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choices(("transform", "convolve", "batch"), weights=(70, 15, 15))[0]
    dtype = "c128" if rng.random() < 0.25 else "c64"
    if kind == "batch":
        return _case(kind="batch", shape=_uneven(rng, rng.choice((4, 8, 16, 24, 40, 64))), dtype=dtype,
                     direction=rng.choice(("forward", "inverse")))
    split = kind == "transform" and dtype == "c64" and rng.random() < 0.1
    # log2 of the number of elements, spread evenly: 2^12 (32 KB) to 2^27 (1 GiB) in complex64, 2^25 in complex128
    lg = rng.randint(12, 25 if dtype == "c128" else 27)
    d = rng.choices((1, 2, 3, 4, 5), weights=(1, 5, 10, 3, 3))[0]
    top = 11 if dtype == "c128" else 12  # sides up to 2048 / 4096
    while d * top < lg:
        d += 1
    # sides: an even share of the bits, then some bits moved from one axis to another (ragged shapes)
    bits = [lg // d + (1 if l < lg % d else 0) for l in range(d)]
    rng.shuffle(bits)
    for _ in range(rng.choice((0, 0, 1, 2, 3))):
        a, b = rng.randrange(d), rng.randrange(d)
        if a != b and bits[a] > 2 and bits[b] < top:
            bits[a] -= 1
            bits[b] += 1
    grid = "default"
    if rng.random() < 0.35:  # a grid of the user's own: p_l^2 | n_l, p_l up to 16
        grid = _text(2 ** rng.randint(min(1, b // 2), min(4, b // 2)) for b in bits)
    inplace = kind == "transform" and rng.random() < 0.15
    return _case(kind=kind, shape=_text(2 ** b for b in bits), grid=grid, dtype=dtype,
                 direction="both" if inplace else "forward" if kind == "convolve" else
                 rng.choice(("forward", "inverse", "both")), inplace=inplace,
                 precision=rng.choice(("bf16", "fp16")) if split else "native",
                 layout="cyclic" if kind == "transform" and rng.random() < 0.08 else "natural",
                 inputs="loguniform" if split and rng.random() < 0.5 else "uniform")


def _array(gen, shape, dtype, inputs):
    real = torch.float64 if dtype == "c128" else torch.float32
    if inputs == "loguniform":
        size = torch.rand(shape, generator=gen, device="cuda", dtype=real).mul_(6).sub_(3)
        return torch.polar(size.mul_(math.log(10)).exp_(),
                           torch.rand(shape, generator=gen, device="cuda", dtype=real).mul_(2 * math.pi))
    return torch.view_as_complex(torch.rand((*shape, 2), generator=gen, device="cuda", dtype=real).mul_(2).sub_(1))


def _inputs(case, seed):
    """The case's arrays: one per shape; of a convolution the array and its multiplier."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    arrays = [_array(gen, s, case["dtype"], case["inputs"]) for s in _shapes(case)]
    if case["kind"] == "convolve":
        arrays.append(_array(gen, arrays[0].shape, case["dtype"], case["inputs"]))
    return arrays


class _State:
    """Inputs, outputs and the plans that a program keeps."""

    def __init__(self, case, seed):
        self.case, self.xs, self.plans, self.batch = case, _inputs(case, seed), [], None
        grid = None if case["grid"] == "default" else _shape(case["grid"])
        shapes = _shapes(case)
        dirs = (False, True) if case["kind"] == "convolve" or case["direction"] == "both" else \
            (case["direction"] == "inverse",)
        for s in shapes:
            for inverse in dirs:
                self.plans.append(fftu.Plan(s, grid, dtype=_TORCH[case["dtype"]], inverse=inverse,
                                            precision=_PRECISION[case["precision"]], layout=_LAYOUT[case["layout"]]))
        if case["kind"] == "convolve":
            self.ys = [torch.empty_like(self.xs[0]) for _ in range(2)]
        elif case["kind"] == "batch":
            self.ys = [torch.empty_like(x) for x in self.xs]
            self.batch = fftu.fftu_batch_create([p.handle for p in self.plans])
            self.ins, self.outs = [x.data_ptr() for x in self.xs], [y.data_ptr() for y in self.ys]
        else:
            self.ys = [] if case["inplace"] else [torch.empty_like(self.xs[0]) for _ in dirs]

    def __del__(self):
        if getattr(self, "batch", None):
            fftu.fftu_batch_destroy(self.batch)  # before the plans whose tables it reads


def prepare(case, seed):
    return _State(case, seed)


def run(s):
    case = s.case
    if case["kind"] == "convolve":
        x, mul = s.xs
        out, spectrum = s.ys
        fftu.fftu_exec_pointwise(s.plans[0].handle, s.plans[1].handle, x.data_ptr(), mul.data_ptr(),
                                 spectrum.data_ptr(), out.data_ptr(), torch.cuda.current_stream().cuda_stream)
        return [out, spectrum]
    if case["kind"] == "batch":
        fftu.fftu_batch_exec(s.batch, s.ins, s.outs, torch.cuda.current_stream().cuda_stream)
        return s.ys
    x = s.xs[0]
    if case["inplace"]:
        for p in s.plans:
            p.exec(x, x)
        return [x]
    for p, y in zip(s.plans, s.ys):
        x = p.exec(x, y)
    return s.ys


def work(case):
    size = _BYTES[case["dtype"]]
    sizes = [math.prod(s) for s in _shapes(case)]
    n, fft = sum(sizes), sum(5 * v * math.log2(v) for v in sizes)
    if case["kind"] == "convolve":  # reads the array and the multiplier, writes the spectrum and the result
        return {"bytes": 4 * n * size, "flops": 2 * fft + 6 * n}
    k = 2 if case["direction"] == "both" else 1
    return {"bytes": k * 2 * n * size, "flops": k * fft}


def _to_cyclic(case, a, back=False):
    """Natural order to processor-major storage (or back), as a reshape and a transpose."""
    n = a.shape
    grid = _shape(case["grid"]) if case["grid"] != "default" else \
        tuple(2 ** min(3, (v.bit_length() - 1) // 2) for v in n)
    d = len(n)
    if back:  # (s_1 .. s_d, r_1 .. r_d) -> (r_1, s_1, r_2, s_2, ...)
        a = a.reshape(*grid, *(v // p for v, p in zip(n, grid)))
        return a.permute([k for l in range(d) for k in (d + l, l)]).reshape(n)
    a = a.reshape([k for v, p in zip(n, grid) for k in (v // p, p)])
    return a.permute([2 * l + 1 for l in range(d)] + [2 * l for l in range(d)]).reshape(n)


def exact(case, seed):
    xs = [x.to(torch.complex128) for x in _inputs(case, seed)]
    if case["kind"] == "convolve":
        spectrum = torch.fft.fftn(xs[0]) * xs[1]
        return [torch.fft.ifftn(spectrum), spectrum]
    if case["kind"] == "transform" and case["layout"] == "cyclic":
        xs = [_to_cyclic(case, x, back=True) for x in xs]
    if case["direction"] == "both":
        ys = xs if case["inplace"] else [torch.fft.fftn(xs[0]), xs[0]]
    else:
        f = torch.fft.fftn if case["direction"] == "forward" else torch.fft.ifftn
        ys = [f(x) for x in xs]
    return [_to_cyclic(case, y) for y in ys] if case["kind"] == "transform" and case["layout"] == "cyclic" else ys
