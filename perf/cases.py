"""Performance cases of the V_loc library: the calls that plane-wave codes make of it.

A case is one call (or one forward and backward) through the public Python
API on inputs that are resident on the GPU: a grid (n1, n2, n3), the cut-off
sphere of radius ``r`` in integer Miller units, a block of bands and an
operation.  ``listed`` are the reference sizes, ``draw`` gives more of the
same ranges, ``prepare`` / ``run`` make and time one, ``work`` counts what a
pass cannot do without and ``exact`` is the same result in plain FP64
``torch.fft``.

Operations: ``apply`` (A c), ``apply_h`` (diag + A), ``gamma_h`` (diag + A on
real bands, half sphere), ``grad`` (A c, then dL/dc and dL/dV for a given
upstream gradient), ``density``, ``halves`` (G -> r and r -> G) and ``batch``
(several grids in one call).
"""
import math

import numpy as np
import torch

# Uneven batch: cubes n^3 with r = n / 4, bands 64, 128, ... 512 (the largest grids hold the most bands).
BATCH = (48, 60, 72, 96, 100, 120, 128, 144)
CELL_PER_POINT = 0.35  # grid spacing in bohr: the kinetic term is |2 pi G / L|^2 / 2 with L = n * spacing


def _case(op, grid, r, bands, dtype="c64", name=None, **extra):
    n1, n2, n3 = grid
    case = {"op": op, "n1": n1, "n2": n2, "n3": n3, "r": r, "bands": bands, "dtype": dtype,
            "order": "canonical", "double_float": False}
    case.update(extra)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # One band on the smallest grid, FP64: a single trial vector, where latency and launches count.
        _case("apply", (24, 24, 24), 6.0, 1, "c128", name="one_band_24_fp64"),
        # A small block in a band-by-band or block-Davidson step: H applied to a few bands.
        _case("apply_h", (48, 48, 48), 12.0, 8, name="few_bands_48"),
        # Both half transforms with full real-space grids (exchange, projections): c -> psi(r), u(r) -> c.
        _case("halves", (64, 64, 64), 16.0, 256, name="halves_64"),
        # The reference-precision apply of a block of bands.
        _case("apply", (64, 64, 64), 16.0, 256, "c128", name="block_64_fp64"),
        # The headline block: 1024 bands at 96^3, FP32.
        _case("apply", (96, 96, 96), 24.0, 1024, name="block_96"),
        # The same block on an orthorhombic cell (radices 2, 3 and 5).
        _case("apply", (96, 96, 120), 24.0, 1024, name="block_96x96x120"),
        # FP64 data through the double-float kernels.
        _case("apply", (96, 96, 96), 24.0, 256, "c128", name="double_float_96", double_float=True),
        # Gamma-point sampling at the 500-atom size (80^3, 1001 real bands): the eigensolver's matrix-vector product.
        _case("gamma_h", (80, 80, 80), 20.3, 1001, name="gamma_80"),
        # A cell with three different axes, a cut-off between grid steps and the caller's own plane-wave order.
        _case("apply_h", (72, 90, 108), 17.3, 200, name="ragged_72x90x108", order="shuffled"),
        # Differentiable apply: forward, then the gradients of the coefficients and of the potential.
        _case("grad", (96, 96, 96), 24.0, 512, name="grad_96"),
        # Charge density of a block with occupations.
        _case("density", (100, 100, 100), 24.6, 640, name="density_100"),
        # Eight cells of different size in one graph-captured call (k-points or fragments of uneven size).
        _case("batch", (0, 0, 0), 0.0, 64, name="batch_48_to_144"),
    ]


def _smooth(lo, hi):
    out = []
    for n in range(lo, hi + 1):
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1:
            out.append(n)
    return out


def draw(rng):
    op, dtype, df = rng.choice(
        [("apply", "c64", False)] * 3 + [("apply_h", "c64", False)] * 2 + [("apply", "c128", False)] * 2
        + [("apply", "c128", True), ("gamma_h", "c64", False), ("gamma_h", "c64", False), ("grad", "c64", False),
           ("density", "c64", False), ("halves", "c64", False), ("batch", "c64", False)])
    if op == "batch":  # the same eight cells with other band counts
        return _case("batch", (0, 0, 0), 0.0, rng.randint(4, 63))
    # a cut-off, then a grid that holds its product sphere: every axis the next few 2/3/5-smooth lengths above 4 r
    r = round(math.exp(rng.uniform(math.log(6.0), math.log(32.0))), 2)
    lengths = _smooth(math.ceil(4 * r), math.ceil(5 * r) + 2)
    if rng.random() < 0.4:  # a cubic cell
        grid = (rng.choice(lengths),) * 3
    else:
        grid = tuple(rng.choice(lengths) for _ in range(3))
    case = _case(op, grid, r, 1, dtype, double_float=df,
                 order="shuffled" if op != "gamma_h" and rng.random() < 0.3 else "canonical")
    flops = 7e9 if dtype == "c128" else 1e11  # the listed blocks' work
    cap = min(1024, flops / work(case)["flops"], 4e9 / (8.0 * grid[0] * grid[1] * grid[2]) if op == "halves" else 1024)
    case["bands"] = max(1, round(math.exp(rng.uniform(0.0, math.log(max(1.0, cap))))))
    return case


# ------------------------------------------------------------------ inputs
def _parts(case):
    """The single-grid cases a case consists of (a batch has eight)."""
    if case["op"] != "batch":
        return [case]
    return [_case("apply", (n, n, n), n / 4, case["bands"] * (i + 1)) for i, n in enumerate(BATCH)]


def _sphere(case, seed):
    """Miller indices h^2 + k^2 + l^2 <= r^2, int32 [npw, 3], stick by stick (or shuffled); the half sphere for Gamma."""
    ns, r = (case["n1"], case["n2"], case["n3"]), case["r"]
    axes = [np.arange(max(-int(r), -(n // 2)), min(int(r), (n + 1) // 2 - 1) + 1) for n in ns]
    h, k, l = np.meshgrid(*axes, indexing="ij")
    keep = h * h + k * k + l * l <= r * r
    if case["op"] == "gamma_h":
        keep &= (h > 0) | ((h == 0) & (k > 0)) | ((h == 0) & (k == 0) & (l >= 0))
    g = np.stack([h[keep], k[keep], l[keep]], axis=1).astype(np.int32)
    if case["order"] == "shuffled":
        return np.ascontiguousarray(g[np.random.default_rng(seed).permutation(len(g))])
    return np.ascontiguousarray(g[np.lexsort((g[:, 2], g[:, 1] % ns[1], g[:, 0] % ns[0]))])


def _potential(ns, gen, dtype):
    """Smooth real V(r): the modes |q|_inf <= 4 with amplitudes falling as exp(-|q|^2 / 8) around a constant."""
    q = torch.arange(-4, 5, device="cuda", dtype=torch.float64)
    amp = 0.25 * torch.exp(-(q[:, None, None] ** 2 + q[None, :, None] ** 2 + q[None, None, :] ** 2) / 8.0)
    v = amp * torch.randn((9, 9, 9), generator=gen, device="cuda", dtype=torch.complex128)
    v[4, 4, 4] = 1.0
    for n in ns:  # transform the leading mode axis and move it to the back, three times
        e = torch.exp(2j * math.pi * q[:, None] * torch.arange(n, device="cuda", dtype=torch.float64)[None, :] / n)
        v = torch.tensordot(v, e, dims=([0], [0]))
    return v.real.to(dtype).contiguous()


def _inputs(case, seed):
    """G-list and device tensors of a single-grid case, from the seed alone."""
    ns = (case["n1"], case["n2"], case["n3"])
    cdt, rdt = (torch.complex64, torch.float32) if case["dtype"] == "c64" else (torch.complex128, torch.float64)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    g = _sphere(case, seed)
    g2 = torch.from_numpy((g.astype(np.float64) ** 2).sum(axis=1)).to("cuda")

    def block():
        c = torch.randn((case["bands"], len(g)), generator=gen, device="cuda", dtype=cdt)
        c *= (math.sqrt(2.0) / (1.0 + g2)).to(rdt)
        return c

    d = {"g": g, "c": block(), "V": _potential(ns, gen, rdt)}
    op = case["op"]
    if op == "gamma_h":  # a real band has a real c(0)
        zero = np.flatnonzero(~g.any(axis=1))
        d["c"][:, zero] = d["c"][:, zero].real.to(cdt)
    if op in ("apply_h", "gamma_h"):
        k = 2.0 * math.pi * g / (CELL_PER_POINT * np.asarray(ns, dtype=np.float64))
        d["diag"] = torch.from_numpy(0.5 * (k ** 2).sum(axis=1)).to("cuda", rdt)
    if op == "grad":
        d["g_out"] = block()
    if op == "density":
        d["occ"] = 2.0 * torch.rand(case["bands"], generator=gen, device="cuda", dtype=rdt)
    if op == "halves":
        d["u"] = torch.randn((case["bands"], *ns), generator=gen, device="cuda", dtype=cdt)
    return d


def prepare(case, seed):
    """The inputs on the GPU, the plan and the output buffers that a program keeps."""
    from paper_1601_07378_gb300 import vloc
    states = []
    for i, part in enumerate(_parts(case)):
        d = _inputs(part, seed + 1000003 * i)
        d["plan"] = vloc.VlocPlan((part["n1"], part["n2"], part["n3"]), d["g"], d["c"].dtype,
                                  gamma=part["op"] == "gamma_h", double_float=part["double_float"],
                                  graph=case["op"] == "batch")
        if part["op"] in ("apply", "apply_h", "gamma_h"):
            d["out"] = torch.empty_like(d["c"])
        elif part["op"] == "halves":
            d["psi"], d["out"] = torch.empty_like(d["u"]), torch.empty_like(d["c"])
        elif part["op"] == "density":
            d["rho"] = torch.empty_like(d["V"])
        elif part["op"] == "grad":
            d["c"].requires_grad_(True)
            d["V"].requires_grad_(True)
        states.append(d)
    return {"op": case["op"], "parts": states}


def run(state):
    from paper_1601_07378_gb300 import vloc
    op, d = state["op"], state["parts"][0]
    plan = d["plan"]
    if op == "apply":
        return plan.apply(d["c"], d["V"], d["out"])
    if op in ("apply_h", "gamma_h"):
        return plan.apply_h(d["c"], d["V"], d["diag"], d["out"])
    if op == "density":
        return plan.density(d["c"], d["occ"], d["rho"])
    if op == "halves":
        return plan.to_real(d["c"], d["psi"]), plan.to_recip(d["u"], d["out"])
    if op == "grad":
        out = vloc.vloc_apply(d["c"], d["V"], plan)
        gc, gv = torch.autograd.grad(out, (d["c"], d["V"]), d["g_out"])
        return out.detach(), gc, gv
    parts = state["parts"]
    return vloc.apply_batched([p["plan"] for p in parts], [p["c"] for p in parts], [p["V"] for p in parts],
                              [p["out"] for p in parts])


# -------------------------------------------------------------------- work
def work(case):
    """Bytes (each input read once, each output written once) and the 5 n log2 n flops of the pruned 1-D
    transforms: the occupied sticks along z, the planes that meet them along y, every line along x."""
    total = {"bytes": 0.0, "flops": 0.0}
    for p in _parts(case):
        n1, n2, n3, r, nb, op = p["n1"], p["n2"], p["n3"], p["r"], p["bands"], p["op"]
        cplx, real = (8, 4) if p["dtype"] == "c64" else (16, 8)
        grid = n1 * n2 * n3
        m = [min(int(r), (n - 1) // 2) for n in (n1, n2, n3)]
        h, k = np.meshgrid(np.arange(-m[0], m[0] + 1), np.arange(-m[1], m[1] + 1), indexing="ij")
        left = r * r - h * h - k * k
        sticks, planes = int((left >= 0).sum()), 2 * m[0] + 1
        npw = int((2 * np.minimum(np.floor(np.sqrt(np.maximum(left, 0.0))), m[2]) + 1)[left >= 0].sum())
        lines = [(sticks, n3), (planes * n3, n2), (n2 * n3, n1)]
        half = sum(5.0 * count * n * math.log2(n) for count, n in lines)  # one direction of one band
        if op == "gamma_h":  # two real bands per complex transform
            half, npw = half / 2, (npw + 1) // 2
        block = nb * npw * cplx
        if op == "density":
            b, f = block + nb * real + grid * real, nb * (half + 4.0 * grid)
        elif op == "halves":
            b, f = 2 * block + 2 * nb * grid * cplx, nb * 2 * half
        elif op == "grad":  # c, g in; out, dL/dc out; V in, dL/dV out
            b, f = 4 * block + 2 * grid * real, nb * (4 * half + 8.0 * grid)
        else:
            b, f = 2 * block + grid * real, nb * (2 * half + 2.0 * grid)
            if op in ("apply_h", "gamma_h"):
                b, f = b + npw * real, f + 4.0 * nb * npw
        total["bytes"] += b
        total["flops"] += f
    return total


# ------------------------------------------------------------------- exact
def _exact_part(case, seed):
    d = _inputs(case, seed)
    ns, op, nb = (case["n1"], case["n2"], case["n3"]), case["op"], case["bands"]
    grid = ns[0] * ns[1] * ns[2]
    g = torch.from_numpy(d["g"].astype(np.int64)).to("cuda")
    n = torch.tensor(ns, device="cuda")

    def flat(x):
        m = torch.remainder(x, n)
        return (m[:, 0] * ns[1] + m[:, 1]) * ns[2] + m[:, 2]

    at, minus = flat(g), flat(-g)
    V = d["V"].to(torch.float64)
    step = max(1, int(4e8 // (16 * grid)))  # about 0.4 GB of grids at a time

    def to_real(c):
        x = torch.zeros((len(c), grid), dtype=torch.complex128, device="cuda")
        c = c.to(torch.complex128)
        if op == "gamma_h":
            x[:, minus] = c.conj()
        x[:, at] = c
        return torch.fft.ifftn(x.view(-1, *ns), dim=(1, 2, 3), norm="forward")

    def to_recip(u):
        return torch.fft.fftn(u, dim=(1, 2, 3), norm="forward").reshape(len(u), grid)[:, at]

    blocks = range(0, nb, step)
    if op == "density":
        rho = torch.zeros(ns, dtype=torch.float64, device="cuda")
        for i in blocks:
            w = d["occ"][i:i + step].to(torch.float64)
            rho += (w[:, None, None, None] * to_real(d["c"][i:i + step]).abs() ** 2).sum(0)
        return rho
    if op == "halves":
        return (torch.cat([to_real(d["c"][i:i + step]) for i in blocks]),
                torch.cat([to_recip(d["u"][i:i + step].to(torch.complex128)) for i in blocks]))

    def action(x):
        y = torch.cat([to_recip(V * to_real(x[i:i + step])) for i in blocks])
        return y + d["diag"].to(torch.float64) * x if "diag" in d else y

    out = action(d["c"])
    if op != "grad":
        return out
    gv = torch.zeros(ns, dtype=torch.float64, device="cuda")
    for i in blocks:
        gv += (to_real(d["g_out"][i:i + step]).conj() * to_real(d["c"][i:i + step])).real.sum(0)
    return out, action(d["g_out"]), gv / grid


def exact(case, seed):
    """What ``run`` returns for these inputs, in FP64 with torch.fft."""
    parts = [_exact_part(p, seed + 1000003 * i) for i, p in enumerate(_parts(case))]
    return parts if case["op"] == "batch" else parts[0]
