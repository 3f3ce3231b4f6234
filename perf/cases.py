"""Timed cases: the work that programs have this solver do, through its public
entry points, over the range of meshes and precisions it accepts.

A case is one of

* ``solve``    Plan.solve on device tensors: one potential from one source,
               the call inside a time-step loop (the plan is kept, the source
               is new every step);
* ``batch``    submit_batch: independent grids of different shapes in one call;
* ``host``     Plan.solve_host: source and potential in pinned host memory,
               copies inside the call;
* ``noalloc``  ipf_solve_noalloc: no plan, no allocation, the Green's spectrum
               rebuilt inside the call.

Sources are the seeded bodies of the package's test problems (uniform spheres
of random place, size and density and one Gaussian, on a zero background).
"""
import math

import numpy as np
import torch

from paper_1106_0557_gb300 import Plan, native, sources, submit_batch

FOUR_PI = 4.0 * math.pi
_REAL = {"f32": torch.float32, "f64": torch.float64, "df64": torch.float64}
_BYTES = {"f32": 4, "f64": 8, "df64": 8}

# volume limits of drawn meshes (cells), so that no drawn case costs more than
# the largest listed one
_VOLUME = {"f32": 2.0e8, "df64": 4.0e7, "f64": 8.0e6}
_AXIS = {"f32": 1152, "df64": 640, "f64": 400}


def _solve(name, n, dtype="f32", h=None, kind="solve"):
    h = h or (1.0 / n[0],) * 3
    return {"name": name, "kind": kind, "dtype": dtype, "nx": n[0], "ny": n[1], "nz": n[2], "hx": h[0], "hy": h[1],
            "hz": h[2]}


def listed():
    return [
        # the smallest mesh of the tests and of the serving mix: latency, five launches
        _solve("f32_32", (32, 32, 32)),
        # a ragged mesh with anisotropic cells
        _solve("f32_100x70x30", (100, 70, 30), h=(1.0, 0.5, 0.25)),
        # an ordinary cube, the largest shape of the ragged batch
        _solve("f32_128", (128, 128, 128)),
        # a cube of the serving mix (N is any whole number from 32 to 384 there)
        _solve("f32_309", (309, 309, 309)),
        # the benchmark's workload
        _solve("f32_256", (256, 256, 256)),
        # the binary-spheroid box, 2:1:1
        _solve("f32_768x384x384", (768, 384, 384)),
        # the paper's largest mesh
        _solve("f32_1152", (1152, 1152, 1152)),
        # FP64-class solves of the serving mix
        _solve("df64_196", (196, 196, 196), "df64"),
        # the same path in native FP64, on a ragged anisotropic mesh
        _solve("f64_96x80x64", (96, 80, 64), "f64", h=(1.0, 1.0, 2.0)),
        # 64 independent ragged grids in one call
        {"name": "f32_batch64", "kind": "batch", "count": 64, "first": 0},
        # the benchmark's workload from pinned host memory
        _solve("f32_host_256", (256, 256, 256), kind="host"),
        # the allocation-free call
        _solve("f32_noalloc_64", (64, 64, 64), kind="noalloc"),
    ]


def _axis(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["solve", "batch", "host", "noalloc"], [12, 2, 1, 1])[0]
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(2, 64), "first": rng.randint(1, 1000)}
    if kind == "noalloc":
        dtype, lo, hi, vol = rng.choice(["f32", "f64"]), 8, 90, 1.0e5
    else:
        dtype = rng.choices(["f32", "df64", "f64"], [6, 3, 1])[0]
        lo, hi, vol = 16, _AXIS[dtype], _VOLUME[dtype]
        if kind == "host":
            hi, vol = min(hi, 400), min(vol, 3.0e7)
    while True:
        if rng.random() < 0.5:
            n = (_axis(rng, lo, hi),) * 3
        else:
            n = tuple(_axis(rng, lo, hi) for _ in range(3))
        if n[0] * n[1] * n[2] <= vol:
            break
    h = (1.0 / n[0],) * 3 if rng.random() < 0.5 else tuple(rng.choice([0.25, 0.5, 1.0, 1.5]) for _ in range(3))
    c = _solve("", n, dtype, h, kind)
    del c["name"]
    return c


def _mesh(case):
    return (case["nx"], case["ny"], case["nz"]), (case["hx"], case["hy"], case["hz"])


def _grids(case, seed):
    """(N, h, bodies) of a batch: shapes from the case, bodies from the seed."""
    out = []
    for i in range(case["count"]):
        g = sources.rng(case["first"] + i)
        N = tuple(int(v) for v in g.choice(sources.BATCH_SIZES, 3))
        h = (1.0 / 128,) * 3
        out.append((N, h, sources.multi_sphere_bodies(sources.rng([seed, i]), tuple(n * v for n, v in zip(N, h)))))
    return out


def _source(case, seed):
    N, h = _mesh(case)
    bodies = sources.multi_sphere_bodies(sources.rng(seed), tuple(n * v for n, v in zip(N, h)))
    return sources.rasterize_torch(bodies, N, h, dtype=_REAL[case["dtype"]])


def prepare(case, seed):
    if case["kind"] == "batch":
        plans, src, out = [], [], []
        for N, h, bodies in _grids(case, seed):
            plans.append(Plan(N, h, "f32"))
            src.append(sources.rasterize_torch(bodies, N, h, dtype=torch.float32))
            out.append(torch.empty_like(src[-1]))
        return {"kind": "batch", "plans": plans, "src": src, "out": out}
    N, h = _mesh(case)
    src = _source(case, seed)
    if case["kind"] == "noalloc":
        return {"kind": "noalloc", "n": N, "h": h, "dtype": case["dtype"], "src": src, "out": torch.empty_like(src)}
    state = {"kind": case["kind"], "plan": Plan(N, h, case["dtype"])}
    if case["kind"] == "host":
        src = src.cpu().pin_memory()
        out = torch.empty(src.shape, dtype=src.dtype, pin_memory=True)
        state.update(pinned=(src, out), src=src.numpy(), out=out.numpy())
    else:
        state.update(src=src, out=torch.empty_like(src))
    return state


def run(state):
    kind = state["kind"]
    if kind == "solve":
        return state["plan"].solve(state["src"], out=state["out"])
    if kind == "batch":
        return submit_batch(state["plans"], state["src"], state["out"])
    if kind == "host":
        return state["plan"].solve_host(state["src"], out=state["out"])
    native.ipf_solve_noalloc(state["n"], state["h"], state["dtype"], state["src"].data_ptr(), state["out"].data_ptr(),
                             torch.cuda.current_stream().cuda_stream)
    return state["out"]


def _work(N, real, spectrum=True):
    """Source and potential once each, and the kept transform of the Green's
    function (its even octant on the doubled mesh); the flops of the padded
    transforms with the zero lines left out, 5 n log2 n per complex line."""
    nx, ny, nz = N
    cells = nx * ny * nz
    octant = (nx + 1) * (ny + 1) * (nz + 1)
    line = lambda n: 5.0 * 2 * n * math.log2(2 * n)  # noqa: E731
    flops = 2 * (ny * nz * line(nx) / 2 + nx * nz * line(ny) + 2 * nx * ny * line(nz)) + 2.0 * 4 * nx * ny * nz
    if not spectrum:  # built inside the call: a cosine transform per axis
        flops += octant * 2.5 * (math.log2(2 * nx) + math.log2(2 * ny) + math.log2(2 * nz))
    return {"bytes": float(real * (2 * cells + (octant if spectrum else 0))), "flops": flops}


def work(case):
    if case["kind"] == "batch":
        parts = [_work(N, 4) for N, _, _ in _grids(case, 0)]
        return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}
    return _work(_mesh(case)[0], _BYTES[case["dtype"]], case["kind"] != "noalloc")


def tolerance(case):
    # four to five times the distance from the 64-bit transforms of `exact`
    # that was measured over these ranges: FP32 0.9e-7 to 1.3e-7, FP64 3e-16
    # (larger meshes up to 5e-16, of which the FFTs of `exact` hold a part),
    # float pairs (48 bits) 5.7e-15; "max": against the result's root mean
    # square, or the value itself where that is larger
    dtype = case.get("dtype", "f32")
    if dtype == "f32":
        return {"rel": 5e-7, "max": 3e-6}
    if dtype == "f64":
        return {"rel": 2e-15, "max": 1.5e-14}
    return {"rel": 3e-14, "max": 2e-13}


def _convolve(src, N, h):
    """The discrete aperiodic convolution in FP64: transforms of the zero-padded
    source and of the doubled-mesh Green's table, their product, back, cropped."""
    nx, ny, nz = N
    dev = src.device

    def offsets(n, w):
        i = torch.arange(2 * n, device=dev, dtype=torch.float64)
        return torch.minimum(i, 2 * n - i) * w

    x, y, z = offsets(nx, h[0]).view(1, 1, -1), offsets(ny, h[1]).view(1, -1, 1), offsets(nz, h[2]).view(-1, 1, 1)
    num = -h[0] * h[1] * h[2] / FOUR_PI
    G = x * x + y * y + z * z
    G[0, 0, 0] = min(h) ** 2
    G.sqrt_().reciprocal_().mul_(num)
    s = (2 * nz, 2 * ny, 2 * nx)
    Gt = torch.fft.rfftn(G)
    del G
    St = torch.fft.rfftn(src.to(torch.float64), s=s)
    St.mul_(Gt)
    del Gt
    return torch.fft.irfftn(St, s=s)[:nz, :ny, :nx].contiguous()


def exact(case, seed):
    if case["kind"] == "batch":
        return [_convolve(sources.rasterize_torch(b, N, h, dtype=torch.float32), N, h)
                for N, h, b in _grids(case, seed)]
    N, h = _mesh(case)
    if N[0] * N[1] * N[2] > 2.5e8:  # the doubled mesh in FP64 complex values would not fit
        return None
    phi = _convolve(_source(case, seed), N, h)
    return phi.cpu().numpy() if case["kind"] == "host" else phi
