"""The work that programs have this library do, as cases to be timed.

A case is a dict of plain values.  ``kind`` names the entry point:

  dft      Plan(n, batch, r, precision).exec: 1-D transforms of n = r^k or
           n = q r^k points, forward or inverse
  noalloc  exec_noalloc: the same without a plan, for small working sets
  dft2     Plan2.exec: 2-D transforms of n1 x n2 arrays
  conv2    Plan2.conv: circular 2-D convolutions with one given spectrum
  stencil  StencilPlan.apply: k sweeps of a 3 x 3 linear stencil

Sizes and distributions are those of the repository's own workloads
(``inputs.WORKLOADS``, the benchmark's ``--grid`` run and its precision and
mixed-radix rows) and of its tests.
"""
import math

import torch

import paper_1908_06649_gb300 as pkg

# (direction name -> exponent sign of the entry points)
_DIR = {"forward": pkg.FORWARD, "inverse": pkg.INVERSE}

# the heat update of the stencil tests; a program's own weights differ a
# little from it
_HEAT = ((0.0, 0.1, 0.0), (0.15, 0.5, 0.15), (0.0, 0.1, 0.0))


def _dft(n, batch, r=16, precision=3, direction="forward", values="normal", kind="dft"):
    return {"kind": kind, "n": n, "batch": batch, "r": r, "precision": precision,
            "direction": direction, "values": values}


def listed():
    cases = {
        # a short batch of short transforms, one launch: the call itself
        "n4096_b64": _dft(4096, 64, values="uniform"),
        # very many short transforms (spectra of short signal windows: three
        # tones and noise each)
        "n256_b1048576_tones": _dft(256, 1 << 20, values="tones"),
        # the headline workload: a large batch of two-pass transforms
        "n65536_b1024": _dft(65536, 1024),
        # the radix sweep: the same length on the smallest tensor unit ...
        "n32768_r8_b4096": _dft(32768, 4096, r=8),
        # ... and, in the other direction, on the largest
        "n32768_r32_b4096_inverse": _dft(32768, 4096, r=32, direction="inverse"),
        # a few very long transforms, three passes
        "n16777216_b4": _dft(1 << 24, 4, values="uniform"),
        # a length that is no power of the radix: q r^k, q a power of two,
        # and a batch that no block size divides
        "n131072_mixed_b500": _dft(2 * 16 ** 4, 500),
        # an odd factor (3 r^2), inverse, an ordinary batch of prime size
        "n768_odd_b10007_inverse": _dft(768, 10007, direction="inverse"),
        # the low-precision mode on an ordinary batch
        "n65536_bf16_b300": _dft(65536, 300, precision=4),
        # a filter applied to many images
        "conv2_256x256_b500": {"kind": "conv2", "n1": 256, "n2": 256, "batch": 500, "r": 16,
                               "precision": 3},
        # the stencil workload of the benchmark
        "stencil_4096_k16": {"kind": "stencil", "side": 4096, "steps": 16, "r": 16,
                             "precision": 3},
        # large images, transformed a few at a time
        "dft2_4096x4096_b4": {"kind": "dft2", "n1": 4096, "n2": 4096, "batch": 4, "r": 16,
                              "precision": 3, "direction": "forward"},
    }
    return [dict(c, name=name) for name, c in cases.items()]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _batch_for(rng, n, most_points, least_points=1 << 13):
    """A batch with about a log-uniform number of points in all, any number."""
    points = _log_uniform(rng, max(n, least_points), max(n, most_points))
    return max(1, points // n)


def draw(rng):
    kind = rng.choice(("dft", "dft", "dft", "dft", "mixed", "mixed", "noalloc", "dft2", "dft2",
                       "conv2", "stencil", "stencil"))
    r = rng.choice((8, 16, 16, 32))
    log2r = {8: 3, 16: 4, 32: 5}[r]
    direction = rng.choice(("forward", "inverse"))
    values = rng.choice(("uniform", "normal"))
    if kind == "dft":
        n = r ** rng.randint(1, 24 // log2r)
        return _dft(n, _batch_for(rng, n, 1 << 26), r, rng.choice((3, 3, 3, 1, 4, 5)), direction,
                    rng.choice((values, "tones")) if 64 <= n <= 65536 else values)
    if kind == "mixed":
        if rng.random() < 0.5:
            q = 2 ** rng.randint(1, log2r - 1)
            k = rng.randint(2, 3 if r == 32 else 4)
        else:
            q = rng.choice((3, 5, 6, 7, 9, 10, 12, 15))
            k = rng.randint(1, 3 if r == 8 else 2)
        n = q * r ** k
        return _dft(n, _batch_for(rng, n, 1 << 26), r, rng.choice((3, 3, 1)), direction, values)
    if kind == "noalloc":
        n = r ** rng.randint(1, {8: 4, 16: 4, 32: 3}[r])
        return _dft(n, _batch_for(rng, n, 1 << 22), r, rng.choice((3, 1)), direction, values,
                    kind="noalloc")
    if kind in ("dft2", "conv2"):
        most = 24 // log2r  # n1 n2 <= 2^24
        k1 = rng.randint(1, min(most - 1, 16 // log2r))
        k2 = rng.randint(1, min(most - k1, 16 // log2r))
        n1, n2 = r ** k1, r ** k2
        c = {"kind": kind, "n1": n1, "n2": n2, "batch": _batch_for(rng, n1 * n2, 1 << 25),
             "r": r, "precision": rng.choice((3, 3, 1, 5, 4) if kind == "dft2" else (3, 3, 1, 5))}
        return dict(c, direction=direction) if kind == "dft2" else c
    # one warpgroup pass per axis holds 3 k points up to 512, 256 and 1024
    steps = _log_uniform(rng, 1, {8: 160, 16: 80, 32: 200}[r])
    return {"kind": "stencil", "side": _log_uniform(rng, 100, 4000), "steps": steps, "r": r,
            "precision": rng.choice((3, 3, 1))}


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _signal(values, batch, n, g):
    """batch x n complex64 values: uniform in [-1, 1]^2, N(0, 1) in both parts,
    or three tones of random integer frequencies plus N(0, 0.01^2)."""
    if values == "uniform":
        x = torch.rand(batch, n, 2, generator=g, device="cuda").mul_(2).sub_(1)
        return torch.view_as_complex(x)
    x = torch.view_as_complex(torch.randn(batch, n, 2, generator=g, device="cuda"))
    if values == "tones":
        x *= 0.01
        j = torch.arange(n, device="cuda")
        roots = torch.exp(2j * math.pi * torch.arange(n, device="cuda", dtype=torch.float64) / n)
        roots = roots.to(torch.complex64)
        step = max(1, (1 << 24) // n)
        for b in range(0, batch, step):
            rows = min(step, batch - b)
            f = torch.randint(0, n, (rows, 3), generator=g, device="cuda")
            for t in range(3):
                x[b:b + rows] += roots[(f[:, t:t + 1] * j) % n]
    return x


def _inputs(case, seed):
    """The tensors of a case, and the stencil's weights."""
    g = _generator(seed)
    kind = case["kind"]
    if kind in ("dft", "noalloc"):
        return {"x": _signal(case["values"], case["batch"], case["n"], g)}
    if kind == "stencil":
        A = torch.randn(case["side"], case["side"], generator=g, device="cuda")
        w = torch.tensor(_HEAT, dtype=torch.float64)
        w += 0.02 * torch.rand(3, 3, generator=torch.Generator().manual_seed(seed),
                               dtype=torch.float64)
        w = (w / w.sum()).to(torch.float32)
        return {"A": A, "w": w.tolist()}
    n1, n2, batch = case["n1"], case["n2"], case["batch"]
    t = {"x": _signal("normal", batch, n1 * n2, g).reshape(batch, n1, n2)}
    if kind == "conv2":
        # the spectrum of a smooth real filter: a unit-sum Gaussian
        i = torch.minimum(torch.arange(n1), n1 - torch.arange(n1)).to(torch.float64)
        j = torch.minimum(torch.arange(n2), n2 - torch.arange(n2)).to(torch.float64)
        s = 1.0 + (seed % 7) / 4
        h = torch.exp(-(i[:, None] ** 2 + j[None, :] ** 2) / (2 * s * s))
        t["spectrum"] = torch.fft.fft2(h / h.sum()).to(torch.complex64).cuda()
    return t


def prepare(case, seed):
    state = dict(_inputs(case, seed), case=case)
    kind, r, prec = case["kind"], case["r"], case["precision"]
    if kind == "dft":
        state["plan"] = pkg.Plan(case["n"], case["batch"], r, prec)
    elif kind in ("dft2", "conv2"):
        state["plan"] = pkg.Plan2(case["n1"], case["n2"], case["batch"], r, prec)
    elif kind == "stencil":
        state["plan"] = pkg.StencilPlan(case["side"], case["steps"], r, prec)
    state["out"] = torch.empty_like(state["A"] if kind == "stencil" else state["x"])
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "dft":
        return state["plan"].exec(state["x"], state["out"], _DIR[case["direction"]])
    if kind == "noalloc":
        return pkg.exec_noalloc(state["x"], state["out"], case["n"], case["batch"], case["r"],
                                case["precision"], _DIR[case["direction"]])
    if kind == "dft2":
        return state["plan"].exec(state["x"], state["out"], _DIR[case["direction"]])
    if kind == "conv2":
        return state["plan"].conv(state["x"], state["spectrum"], state["out"])
    return state["plan"].apply(state["A"], state["out"], w3x3=state["w"])


def work(case):
    """Every input read once, every output written once; the operations of a
    fast transform (5 N log2 N, half of it for real data)."""
    kind = case["kind"]
    if kind in ("dft", "noalloc"):
        pts = case["n"] * case["batch"]
        return {"bytes": 16 * pts, "flops": 5 * pts * math.log2(case["n"])}
    if kind == "stencil":
        # forward and inverse real transforms and one product per point
        pts = case["side"] ** 2
        return {"bytes": 8 * pts, "flops": 5 * pts * math.log2(pts) + 3 * pts}
    one = case["n1"] * case["n2"]
    pts = one * case["batch"]
    flops = 5 * pts * math.log2(one)
    if kind == "conv2":
        return {"bytes": 16 * pts + 8 * one, "flops": 2 * flops + 6 * pts}
    return {"bytes": 16 * pts, "flops": flops}


def exact(case, seed):
    """What run returns, by 64-bit library transforms of the same inputs."""
    t = _inputs(case, seed)
    kind = case["kind"]
    if kind == "stencil":
        # on a periodic grid at least 2 k larger than A nothing wraps into
        # it: k sweeps multiply the spectrum by P(e^{i u}, e^{i v})^k
        side, k = case["side"], case["steps"]
        m = side + 2 * k
        u = 2 * math.pi * torch.arange(m, device="cuda", dtype=torch.float64) / m
        v = u[:m // 2 + 1]
        p = torch.zeros(m, m // 2 + 1, device="cuda", dtype=torch.complex128)
        for a in (-1, 0, 1):
            for b in (-1, 0, 1):
                p += t["w"][a + 1][b + 1] * torch.exp(1j * (a * u[:, None] + b * v[None, :]))
        grid = torch.zeros(m, m, device="cuda", dtype=torch.float64)
        grid[:side, :side] = t["A"]
        return torch.fft.irfft2(torch.fft.rfft2(grid) * p ** k, s=(m, m))[:side, :side].contiguous()
    x = t["x"].to(torch.complex128)
    if kind == "conv2":
        return torch.fft.ifft2(torch.fft.fft2(x) * t["spectrum"].to(torch.complex128))
    forward = case["direction"] == "forward"
    if kind == "dft2":
        return torch.fft.fft2(x) if forward else torch.fft.ifft2(x)
    return torch.fft.fft(x) if forward else torch.fft.ifft(x)
