"""Performance cases: whole advances through the public API, over the sizes,
tiles, modes and storage types that the library's workloads use.

One pass is what a simulation does with a handle it keeps: set the state from
device memory, advance, read the state back to device memory (``get_state``
waits for the result, as it always does).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1602_07558_gb300.swept2d import Swept2D, SweptBatch, heat_advance_static

GAMMA, CFL, KAPPA, R, COURANT = 1.4, 0.3, 0.5, 0.2, 0.3
EULER = (GAMMA, CFL, KAPPA)
PARAMS = {"heat": (R,), "heat_kahan": (R,), "wave": (COURANT,), "euler_rk2": EULER,
          "euler_kahan": EULER}
NV = {"heat": 1, "heat_kahan": 2, "wave": 2, "euler_rk2": 8, "euler_kahan": 12}
TORCH = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}


def _grid(name, op, dtype, nx, ny, tile, steps, mode, graph=False, threads=0, field="smooth"):
    return {"name": name, "kind": "grid", "op": op, "dtype": dtype, "nx": nx, "ny": ny,
            "tile": tile, "steps": steps, "mode": mode, "graph": graph, "threads": threads,
            "field": field}


def _batch(name, op, dtype, grids, steps, mode, sizes_seed=3, lo=32, hi=512):
    return {"name": name, "kind": "batch", "op": op, "dtype": dtype, "grids": grids,
            "steps": steps, "mode": mode, "graph": True, "sizes_seed": sizes_seed, "lo": lo,
            "hi": hi}


def listed():
    return [
        # a latency-bound small simulation, replayed as a graph (16 tiles)
        _grid("heat_64_f64", "heat", "f64", 64, 64, 16, 512, "swept", graph=True,
              field="uniform"),
        # the headline grid; 500 steps leave a tail of 20 that does not fill a half cycle
        _grid("heat_4096_f64", "heat", "f64", 4096, 4096, 64, 500, "swept", threads=512),
        # a grid whose sides no tile divides: one launch per step
        _grid("heat_naive_1009x757", "heat", "f64", 1009, 757, 0, 300, "naive"),
        # reduced-precision long diffusion runs, one persistent launch
        _grid("heat_2048_f32", "heat_kahan", "f32", 2048, 2048, 64, 2000, "persistent"),
        _grid("heat_2048_bf16", "heat_kahan", "bf16", 2048, 2048, 64, 2000, "persistent"),
        # leapfrog wave from a localised source
        _grid("wave_1024_f64", "wave", "f64", 1024, 1024, 32, 1000, "swept", field="source"),
        # two-stage gas dynamics in the three storage types
        _grid("euler_2048_f64", "euler_rk2", "f64", 2048, 2048, 32, 50, "swept",
              field="pulse"),
        _grid("euler_2048_f32", "euler_kahan", "f32", 2048, 2048, 32, 200, "swept",
              field="pulse"),
        _grid("euler_2048_bf16", "euler_kahan", "bf16", 2048, 2048, 32, 200, "swept",
              field="pulse"),
        # many independent grids of uneven sides in {32, 48, ..., 512}
        _batch("batch_heat_f32", "heat_kahan", "f32", 1024, 300, "persistent_one"),
        _batch("batch_euler_f32", "euler_kahan", "f32", 256, 50, "swept"),
        # a caller that may not allocate device memory
        {"name": "heat_static_768", "kind": "static", "nx": 768, "ny": 768, "tile": 16,
         "steps": 403},
    ]


# Gcell-steps a drawn case may take, so that none costs more than the largest
# listed one (roughly the listed rates)
_BUDGET = {("heat", "f64"): 6.0, ("heat_kahan", "f32"): 8.0, ("heat_kahan", "bf16"): 8.0,
           ("wave", "f64"): 2.0, ("euler_rk2", "f64"): 0.15, ("euler_kahan", "f32"): 0.6,
           ("euler_kahan", "bf16"): 0.6}


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["grid"] * 7 + ["batch"] * 2 + ["static"])
    if kind == "static":
        tile = rng.choice([8, 16, 32])
        return {"kind": "static", "nx": tile * _log_int(rng, 2, 768 // tile),
                "ny": tile * _log_int(rng, 2, 768 // tile), "tile": tile,
                "steps": _log_int(rng, 10, 500)}
    op, dtype = rng.choice(sorted(_BUDGET))
    budget = _BUDGET[op, dtype] * 1e9
    if kind == "batch":
        if op == "wave":
            op, dtype = "heat", "f64"
        grids = _log_int(rng, 8, 512)
        cap = int(budget / (grids * 272.0 * 272.0))
        mode = rng.choice(["swept", "naive", "persistent", "persistent_one"])
        c = _batch("", op, dtype, grids, _log_int(rng, 8, max(16, min(400, cap))), mode,
                   sizes_seed=rng.randrange(10_000))
        del c["name"]
        return c
    euler = op.startswith("euler")
    mode = rng.choice(["swept", "swept", "persistent", "naive"])
    if mode == "naive" and rng.random() < 0.5:
        tile, nx, ny = 0, _log_int(rng, 33, 2500), _log_int(rng, 33, 2500)
    else:
        tile = rng.choice([8, 10, 16, 16, 24, 32, 32] + ([] if euler else [40, 48, 64, 64]))
        top = 2048 if euler or op == "wave" else 4096
        nx = tile * _log_int(rng, 1, top // tile)
        ny = tile * _log_int(rng, 1, top // tile)
    steps = _log_int(rng, 5, max(10, min(2000, int(budget / (nx * ny)))))
    # (the smooth modes have no mean and die out within the run on smaller grids)
    heat = rng.choice(["smooth", "uniform"]) if min(nx, ny) >= 128 else "uniform"
    field = {"wave": "source"}.get(op, "pulse" if euler else heat)
    c = _grid("", op, dtype, nx, ny, tile, steps, mode, graph=rng.random() < 0.5,
              threads=rng.choice([0, 0, 128, 256]) if tile else 0, field=field)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs

def _modes(rng, nx, ny, nmodes, kmax=8):
    """Sum of plane waves, integer wave vectors in [-kmax, kmax]^2 without 0,
    amplitudes N(0,1)/|k|^2: a random smooth periodic field."""
    k = rng.integers(-kmax, kmax + 1, size=(4 * nmodes, 2))
    k = k[(k != 0).any(axis=1)][:nmodes]
    amp = rng.standard_normal(len(k)) / (k * k).sum(axis=1)
    ph = rng.uniform(0.0, 2.0 * np.pi, len(k))
    dev = dict(dtype=torch.float64, device="cuda")
    kx, ky = torch.tensor(k[:, 0], **dev), torch.tensor(k[:, 1], **dev)
    a, p = torch.tensor(amp, **dev), torch.tensor(ph, **dev)
    x = (2.0 * np.pi / nx) * torch.arange(nx, **dev)[None] * kx[:, None] + p[:, None]
    y = (2.0 * np.pi / ny) * torch.arange(ny, **dev)[:, None] * ky[None]
    return (torch.cos(y) * a) @ torch.cos(x) - (torch.sin(y) * a) @ torch.sin(x)


def _field(field, op, nx, ny, seed):
    """Initial state in binary64, (nvars, ny, nx), before rounding to storage."""
    rng = np.random.default_rng(seed)
    if field == "pulse":                 # gas at rest with a smooth density and pressure pulse
        phi = _modes(rng, nx, ny, 16)
        phi = phi / phi.abs().max()
        zero = torch.zeros_like(phi)
        U = torch.stack([1.0 + 0.1 * phi, zero, zero, (1.0 + 0.1 * phi) / (GAMMA - 1.0)])
        return torch.cat([U, U] + ([torch.zeros_like(U)] if op == "euler_kahan" else []))
    if field == "source":                # a Gaussian bump at rest, off the centre by the seed
        sx, sy = rng.uniform(0.4, 0.6, 2) * (nx, ny)
        dev = dict(dtype=torch.float64, device="cuda")
        x, y = torch.arange(nx, **dev)[None] - sx, torch.arange(ny, **dev)[:, None] - sy
        u = torch.exp(-(x * x + y * y) / 16.0)
        return torch.stack([u, u])
    if field == "smooth":
        u = _modes(rng, nx, ny, 32)
    else:
        g = torch.Generator(device="cuda").manual_seed(seed)
        u = torch.rand((ny, nx), generator=g, dtype=torch.float64, device="cuda")
    return torch.stack([u, torch.zeros_like(u)]) if op == "heat_kahan" else u[None]


def _sizes(case):
    rng = np.random.default_rng(case["sizes_seed"])
    vals = np.arange(case["lo"], case["hi"] + 1, 16)
    nx = [int(v) for v in rng.choice(vals, size=case["grids"])]
    ny = [int(v) for v in rng.choice(vals, size=case["grids"])]
    return nx, ny, [32 if a % 32 == 0 and b % 32 == 0 else 16 for a, b in zip(nx, ny)]


def _initial(case, seed):
    """The initial state as the call gets it (rounded to the storage type)."""
    if case["kind"] == "static":
        return _field("smooth", "heat", case["nx"], case["ny"], seed)
    if case["kind"] == "batch":
        nx, ny, _ = _sizes(case)
        field = "pulse" if case["op"].startswith("euler") else "uniform"
        parts = [_field(field, case["op"], a, b, 100_000 * seed + i).reshape(-1)
                 for i, (a, b) in enumerate(zip(nx, ny))]
        return torch.cat(parts).to(TORCH[case["dtype"]])
    u = _field(case["field"], case["op"], case["nx"], case["ny"], seed)
    return u.to(TORCH[case["dtype"]]).contiguous()


def prepare(case, seed):
    u0 = _initial(case, seed)
    state = {"case": case, "in": u0, "out": torch.empty_like(u0)}
    if case["kind"] != "static":
        stream = torch.cuda.Stream()
        kw = dict(op=case["op"], params=PARAMS[case["op"]], stream=stream, dtype=case["dtype"])
        if case["kind"] == "batch":
            nx, ny, tiles = _sizes(case)
            h = SweptBatch(nx, ny, tiles, **kw)
        else:
            h = Swept2D(case["nx"], case["ny"], tile=case["tile"], **kw)
            if case["threads"]:
                h.set_tuning(case["threads"], h.query("stage") != 0.0)
        state.update(stream=stream, handle=h)
    torch.cuda.synchronize()
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "static":
        heat_advance_static(state["in"], state["out"], case["nx"], case["ny"], case["tile"], R,
                            case["steps"], stream=torch.cuda.current_stream())
        return state["out"]
    h = state["handle"]
    state["stream"].wait_stream(torch.cuda.current_stream())
    h.set_state(state["in"])
    h.advance(case["steps"], mode=case["mode"], graph=case["graph"])
    return h.get_state(state["out"])


# --------------------------------------------------------- work, tolerances

# floating-point operations of one cell and time step (a fused multiply-add is
# two): pair sums and primitives formed once per point, two stages for Euler
_FLOPS = {"heat": 6, "heat_kahan": 10, "wave": 8, "euler_rk2": 2 * 86, "euler_kahan": 2 * 86 + 3}


def _cells(case):
    if case["kind"] == "batch":
        nx, ny, _ = _sizes(case)
        return sum(a * b for a, b in zip(nx, ny))
    return case["nx"] * case["ny"]


def work(case):
    op, dtype = case.get("op", "heat"), case.get("dtype", "f64")
    cells = _cells(case)
    size = {"f64": 8, "f32": 4, "bf16": 2}[dtype]
    return {"bytes": 2 * cells * NV[op] * size, "flops": cells * case["steps"] * _FLOPS[op]}


def tolerance(case):
    """About four times the distance to ``exact`` measured over the listed and
    drawn cases: heat and Euler below 2e-16 in binary64, the undamped wave
    1.3e-14, the compensated forms 1.2e-7 (binary32) and 3.5e-3 (bfloat16)."""
    op, dtype = case.get("op", "heat"), case.get("dtype", "f64")
    if dtype == "f64":
        return {"rel": 6e-14 if op == "wave" else 1e-15}
    return {"rel": 5e-7 if dtype == "f32" else 1.4e-2}


# ------------------------------------------------- the same in plain binary64

class _Roll:
    """Neighbours of every point of one periodic grid."""

    def __init__(self, nx, ny):
        self.spacing = (1.0 / nx, 1.0 / ny)

    def __call__(self, u):               # east, west, south, north
        return (torch.roll(u, -1, -1), torch.roll(u, 1, -1), torch.roll(u, -1, -2),
                torch.roll(u, 1, -2))

    def per_grid_max(self, s):
        return s.max()


class _Gather:
    """The same for many grids held one after the other."""

    def __init__(self, nx, ny):
        idx, dx, dy, gid, off = [], [], [], [], 0
        for i, (a, b) in enumerate(zip(nx, ny)):
            g = off + torch.arange(a * b, device="cuda").reshape(b, a)
            idx.append(torch.stack([torch.roll(g, s, d).reshape(-1)
                                    for s, d in ((-1, 1), (1, 1), (-1, 0), (1, 0))]))
            n = a * b
            dx.append(torch.full((n,), 1.0 / a, dtype=torch.float64, device="cuda"))
            dy.append(torch.full((n,), 1.0 / b, dtype=torch.float64, device="cuda"))
            gid.append(torch.full((n,), i, dtype=torch.int64, device="cuda"))
            off += n
        self.idx, self.gid, self.count = torch.cat(idx, 1), torch.cat(gid), len(nx)
        self.spacing = (torch.cat(dx), torch.cat(dy))

    def __call__(self, u):
        return tuple(u[..., i] for i in self.idx)

    def per_grid_max(self, s):
        out = torch.zeros(self.count, dtype=s.dtype, device=s.device)
        return out.scatter_reduce_(0, self.gid, s, "amax")[self.gid]


def _euler_exact(U, nb, steps):
    dx, dy = nb.spacing
    r, m, q, E = U
    p = (GAMMA - 1.0) * (E - 0.5 * (m * m + q * q) / r)
    c = torch.sqrt(GAMMA * p / r)
    a = nb.per_grid_max(torch.maximum(m.abs() / r + c, q.abs() / r + c))
    h = torch.minimum(dx, dy) if torch.is_tensor(dx) else min(dx, dy)
    dt = CFL * h / a

    def rate(W):
        r, m, q, E = W
        u, v = m / r, q / r
        p = (GAMMA - 1.0) * (E - 0.5 * (m * u + q * v))
        F = torch.stack([m, m * u + p, q * u, (E + p) * u])
        G = torch.stack([q, m * v, q * v + p, (E + p) * v])
        We, Ww, Ws, Wn = nb(W)
        Fe, Fw, _, _ = nb(F)
        _, _, Gs, Gn = nb(G)
        return ((KAPPA * a / dx) * (We + Ww - 2.0 * W) + (KAPPA * a / dy) * (Ws + Wn - 2.0 * W)
                - (0.5 / dx * (Fe - Fw) + 0.5 / dy * (Gs - Gn)))

    for _ in range(steps):
        mid = U + 0.5 * dt * rate(U)
        U = U + dt * rate(mid)
    return U, mid


def _advance_exact(op, planes, nb, steps):
    """planes (nvars, ...) in binary64 -> the planes after `steps` steps; the
    compensation planes of the compensated forms are 0 in exact arithmetic."""
    if op in ("euler_rk2", "euler_kahan"):
        U, mid = _euler_exact(planes[:4], nb, steps)
        return torch.cat([U, mid] + ([torch.zeros_like(U)] if op == "euler_kahan" else []))
    u, old = planes[0], planes[1] if len(planes) > 1 else None
    for _ in range(steps):
        e, w, s, n = nb(u)
        d = (e + s) + (w + n) - 4.0 * u
        if op == "wave":
            u, old = 2.0 * u - old + COURANT * COURANT * d, u
        else:
            u = u + R * d
    if op == "wave":
        return torch.stack([u, old])
    return torch.stack([u, torch.zeros_like(u)]) if op == "heat_kahan" else u[None]


def exact(case, seed):
    u0 = _initial(case, seed).to(torch.float64)
    if case["kind"] != "batch":
        return _advance_exact(case.get("op", "heat"), u0, _Roll(case["nx"], case["ny"]),
                              case["steps"])
    nx, ny, _ = _sizes(case)
    nv, off, parts = NV[case["op"]], 0, []
    for a, b in zip(nx, ny):             # per grid (nvars, ny nx), pooled side by side
        parts.append(u0[off:off + nv * a * b].reshape(nv, a * b))
        off += nv * a * b
    got = _advance_exact(case["op"], torch.cat(parts, 1), _Gather(nx, ny), case["steps"])
    off, out = 0, []
    for a, b in zip(nx, ny):
        out.append(got[:, off:off + a * b].reshape(-1))
        off += a * b
    return torch.cat(out)
