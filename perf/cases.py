"""Performance cases of the Jacobi3D library: what its users have it do, through the public entry points.

Five kinds of work, each a dict of plain values:

* ``step``: install a state (one grid or a batch), advance it ``iters`` iterations, optionally evaluate the FP64
  residual, copy the iterate out: the loop of a program that time-steps or smooths its own fields.
* ``solve``: install a state and iterate to a tolerance with a check every ``check_every`` iterations.
* ``serve``: a burst of solve requests to the continuous-batching server, the results awaited on the host.
* ``check``: the allocation-free residual of a padded array that the caller owns.
* ``channel``: one message between two blocks: the receive posted, then the send.
"""
import math
import time

import numpy as np
import torch

import paper_2102_12416_gb300 as jg

TORCH = {"f64": torch.float64, "f32": torch.float32}
ELEM = {"f64": 8, "f32": 4}
ALIGN = 64  # values: the grids of a batch start on 256-byte (f32) or 512-byte (f64) boundaries of the output


def _step(name, size, split, dtype, iters, *, mode="count", path="graph", bc="uniform", interior="zero", residual=True,
          io="device"):
    return {"name": name, "kind": "step", "grids": 1, "nx": size[0], "ny": size[1], "nz": size[2], "mode": mode,
            "bx": split[0], "by": split[1], "bz": split[2], "dtype": dtype, "iters": iters, "path": path, "bc": bc,
            "interior": interior, "residual": residual, "io": io}


def _batch(name, grids, block, dtype, iters, *, lo=16, hi=192, path="graph", sides=2):
    return {"name": name, "kind": "step", "grids": grids, "lo": lo, "hi": hi, "sides": sides, "mode": "shape", "bx": block,
            "by": block, "bz": block, "dtype": dtype, "iters": iters, "path": path, "bc": "uniform", "interior": "zero",
            "residual": True, "io": "device"}


def listed():
    return [
        # the smallest problem of the benchmark set, bound by latency: 64^3 FP64 in 2x2x2 blocks, 100 iterations
        _step("step_64c_f64", (64, 64, 64), (2, 2, 2), "f64", 100, bc="linear", interior="uniform"),
        # a few iterations at a time from a coupled program: small grid, short call, one launch per iteration
        _step("step_128c_f32_short", (128, 128, 128), (32, 32, 32), "f32", 10, mode="shape", path="fused", bc="linear_noise",
              interior="uniform", residual=False),
        # odd extents, blocks with padded rows, all iterations in one persistent launch
        _step("step_ragged_f32_persist", (301, 203, 157), (5, 3, 4), "f32", 50, path="persistent", interior="uniform"),
        # the headline grid: 512^3 FP64 in 8x8x8 blocks of 64^3 (100 of its 1000 iterations)
        _step("step_512c_f64", (512, 512, 512), (8, 8, 8), "f64", 100),
        # the single-precision grid bound by memory: 768^3 FP32 in 12^3 blocks of 64^3 (100 of its 200 iterations)
        _step("step_768c_f32", (768, 768, 768), (12, 12, 12), "f32", 100, bc="linear_noise"),
        # batches of independent grids of all sizes, stepped together, in both precisions
        _batch("batch256_f32", 256, 32, "f32", 100),
        _batch("batch256_f64", 256, 32, "f64", 50),
        # a state loaded from pinned host memory, its residual looked at, and stored to the host again
        _step("load_check_store_f64", (384, 384, 384), (6, 6, 6), "f64", 0, interior="uniform", io="host"),
        # one solve to a tolerance, with a residual check every 100 iterations
        {"name": "solve_96c_f32", "kind": "solve", "nx": 96, "ny": 96, "nz": 96, "mode": "shape", "bx": 32, "by": 32,
         "bz": 32, "dtype": "f32", "path": "graph", "bc": "linear_noise", "interior": "zero", "tol": 1e-4, "check_every": 100,
         "max_iters": 20000},
        # a burst of requests of the serving stream (lognormal sides) at the server
        {"name": "serve_32_f32", "kind": "serve", "requests": 32, "lo": 32, "hi": 256, "dtype": "f32", "tol": 1e-5,
         "check_every": 100, "max_iters": 20000, "slots": 64},
        # the residual of a caller's own array, with nothing allocated
        {"name": "check_256c_f64", "kind": "check", "nx": 256, "ny": 256, "nz": 256, "dtype": "f64"},
        # one face-sized message between two blocks
        {"name": "channel_32k", "kind": "channel", "bytes": 32768, "posted": True},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 7 + ["batch"] * 4 + ["solve"] * 3 + ["serve"] * 2 + ["check"] * 2 + ["channel"] * 2)
    dtype = rng.choice(["f64", "f32"])
    bc, interior = rng.choice(["linear", "linear_noise", "uniform"]), rng.choice(["zero", "uniform", "bc"])
    if bc == "linear":
        interior = "uniform"  # else nothing in the state depends on the seed
    if kind == "step":
        nx, ny, nz = (_log(rng, 32, 640) for _ in range(3))
        block = [max(16, min(n, _log(rng, 24, 96))) for n in (nx, ny, nz)]
        iters = _log(rng, 1, 200)
        iters = max(1, min(iters, int((1.2e10 if dtype == "f64" else 4e10) / (nx * ny * nz))))
        case = _step("", (nx, ny, nz), block, dtype, iters, mode="shape", path=rng.choice(["graph", "graph", "fused", "persistent"]),
                     bc=bc, interior=interior, residual=rng.random() < 0.5, io="host" if rng.random() < 0.2 else "device")
        if rng.random() < 0.5:
            case |= {"mode": "count", **{b: max(1, n // w) for b, n, w in zip(("bx", "by", "bz"), (nx, ny, nz), block)}}
    elif kind == "batch":
        lo, hi, grids = _log(rng, 12, 48), _log(rng, 64, 192), _log(rng, 8, 256)
        iters = _log(rng, 10, 100)
        iters = max(5, min(iters, int((1.0e10 if dtype == "f64" else 2.8e10) / (grids * ((lo + hi) / 2.0) ** 3 * 1.3))))
        case = _batch("", grids, rng.choice([24, 32, 48, 64]), dtype, iters, lo=lo, hi=hi, path=rng.choice(["graph", "graph", "persistent"]),
                      sides=rng.randrange(1 << 20))
    elif kind == "solve":
        nx, ny, nz = (_log(rng, 24, 128) for _ in range(3))
        b = rng.choice([24, 32, 64])
        case = {"kind": "solve", "nx": nx, "ny": ny, "nz": nz, "mode": "shape", "bx": b, "by": b, "bz": b, "dtype": dtype,
                "path": rng.choice(["graph", "graph", "persistent"]), "bc": bc, "interior": "zero" if interior == "bc" else interior,
                "tol": 10.0 ** -rng.randint(3, 4), "check_every": rng.choice([50, 100]), "max_iters": 20000}
    elif kind == "serve":
        case = {"kind": "serve", "requests": rng.randint(4, 10 if dtype == "f64" else 32), "lo": rng.choice([24, 32]), "hi": rng.choice([96, 128, 160]),
                "dtype": dtype, "tol": 1e-4, "check_every": 100, "max_iters": 20000, "slots": 64}
    elif kind == "check":
        nx, ny, nz = (_log(rng, 32, 512) for _ in range(3))
        case = {"kind": "check", "nx": nx, "ny": ny, "nz": nz, "dtype": dtype}
    else:
        case = {"kind": "channel", "bytes": _log(rng, 8, 4 << 20), "posted": rng.random() < 0.5}
    case.pop("name", None)
    return case


def _sizes(case):
    """(nx, ny, nz) of every grid: the case's own, or a batch's sides drawn uniformly from [lo, hi] in steps of 16 or, for
    ranges that are no multiples of 16, of 1."""
    if case.get("grids", 1) == 1:
        return [(case["nx"], case["ny"], case["nz"])]
    r = np.random.RandomState(case["sides"])
    step = 16 if case["lo"] % 16 == 0 and case["hi"] % 16 == 0 else 1
    return [tuple(int(case["lo"] + step * v) for v in row) for row in r.randint(0, (case["hi"] - case["lo"]) // step + 1, (case["grids"], 3))]


def _requests(case, seed):
    """Request sides: lognormal around 64, clipped to [lo, hi]. The sizes belong to the case, the data to the seed."""
    z = np.random.RandomState(6).standard_normal((case["requests"], 3))
    sides = np.clip(np.rint(np.exp(math.log(64.0) + 0.5 * z)), case["lo"], case["hi"]).astype(int)
    return [(tuple(int(v) for v in s), dict(bc="linear_noise", bc_seed=1000 * seed + r, noise_amp=1e-3, interior="zero"))
            for r, s in enumerate(sides)]


def _field(size, case, gen):
    """A padded (nz+2, ny+2, nx+2) state on the GPU: Dirichlet boundary and interior as the case says."""
    nx, ny, nz = size
    dev, shape = "cuda", (nz + 2, ny + 2, nx + 2)
    bc, interior, dtype = case.get("bc", "uniform"), case.get("interior", "uniform"), TORCH[case["dtype"]]

    def function():
        if bc == "uniform":
            return torch.rand(shape, generator=gen, device=dev, dtype=dtype)
        x, y, z = (torch.arange(n + 2, device=dev, dtype=dtype) / (n + 1) for n in (nx, ny, nz))
        g = x[None, None, :] + 2 * y[None, :, None] + 3 * z[:, None, None]
        return g + 1e-3 * torch.rand(shape, generator=gen, device=dev, dtype=dtype) if bc == "linear_noise" else g.contiguous()

    u = function()
    if interior == "zero":
        u[1:-1, 1:-1, 1:-1] = 0
    elif interior == "uniform":
        u[1:-1, 1:-1, 1:-1] = torch.rand((nz, ny, nx), generator=gen, device=dev, dtype=dtype)
    return u


def _fields(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return [_field(s, case, gen) for s in _sizes(case)]


def _offsets(sizes):
    offs, n = [], 0
    for s in sizes:
        offs.append(n)
        n += -(-s[0] * s[1] * s[2] // ALIGN) * ALIGN
    return offs, n


class _Server:
    def __init__(self, case):
        self.s = jg.serve_create(32 << 30, case["slots"], case["dtype"], check_every=case["check_every"], round_checks=2)

    def __del__(self):
        jg.serve_destroy(self.s)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "channel":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        h = jg.Jacobi3D((16, 16, 16), ("count", (2, 1, 1)), "f32")
        src = torch.randint(0, 256, (case["bytes"],), generator=gen, device="cuda", dtype=torch.uint8)
        return {"kind": kind, "h": h, "ch": jg.channel_open(h.h, 1, 0, 1, case["bytes"]), "src": src, "dst": torch.empty_like(src),
                "bytes": case["bytes"], "posted": case["posted"]}
    if kind == "serve":
        reqs = [(s, init, np.empty(s[::-1], np.float64 if case["dtype"] == "f64" else np.float32)) for s, init in _requests(case, seed)]
        return {"kind": kind, "server": _Server(case), "reqs": reqs, "tol": case["tol"], "max_iters": case["max_iters"]}
    fields = _fields(case, seed)
    if kind == "check":
        return {"kind": kind, "u": fields[0], "grid": _sizes(case)[0], "dtype": case["dtype"],
                "out": torch.zeros(3, device="cuda", dtype=torch.float64)}
    sizes = _sizes(case)
    stream = torch.cuda.current_stream()
    h = jg.Jacobi3D(sizes, [(case["mode"], (case["bx"], case["by"], case["bz"]))] * len(sizes), case["dtype"], path=case["path"],
                    stream=stream)
    offs, n = _offsets(sizes)
    host = case.get("io") == "host"
    if host:
        fields = [u.cpu().pin_memory() for u in fields]
        out = torch.zeros(n, dtype=TORCH[case["dtype"]]).pin_memory()
    else:
        out = torch.zeros(n, device="cuda", dtype=TORCH[case["dtype"]])
    ptrs = [out.data_ptr() + o * ELEM[case["dtype"]] for o in offs]
    return {"kind": kind, "h": h, "fields": fields, "out": out, "ptrs": ptrs, "stream": stream, "host": host, "case": case}


def run(state):
    kind = state["kind"]
    if kind == "channel":
        ch, src, dst, n = state["ch"], state["src"].data_ptr(), state["dst"].data_ptr(), state["bytes"]
        stream = torch.cuda.current_stream()
        if state["posted"]:  # expected message: the receive is there before its send
            jg.channel_recv(ch, 1, dst, n, stream)
            jg.channel_send(ch, 0, src, n, stream)
        else:
            jg.channel_send(ch, 0, src, n, stream)
            jg.channel_recv(ch, 1, dst, n, stream)
        return state["dst"]
    if kind == "serve":
        s = state["server"].s
        tickets = [jg.serve_submit(s, g, ("shape", (32, 32, 32)), init, state["tol"], state["max_iters"], out)
                   for g, init, out in state["reqs"]]
        done = []
        for t in tickets:
            while (res := jg.serve_poll(s, t)) is None:
                time.sleep(2e-4)
            done.append(res)
        return {"u": [out for _, _, out in state["reqs"]], "iters": np.array([r.iters for r in done]),
                "rel": np.array([r.rel for r in done])}
    if kind == "check":
        jg.jacobi_residual_noalloc(state["u"].data_ptr(), state["grid"], state["dtype"], state["out"].data_ptr(),
                                   torch.cuda.current_stream())
        return state["out"]
    h, case, stream = state["h"], state["case"], state["stream"]
    device = not state["host"]
    for g, u in enumerate(state["fields"]):
        jg.jacobi_set_state(h.h, g, u.data_ptr(), device, stream)
    got = {}
    if kind == "solve":
        iters, rel, status = h.solve(case["tol"], case["max_iters"], case["check_every"])
        got = {"iters": np.array(iters), "rel": np.array(rel), "status": np.array(status)}
    else:
        h.step(case["iters"])
        if case["residual"]:
            rel, res = h.residual()
            got = {"rel": np.array(rel), "abs": np.array(res)}
    for g, p in enumerate(state["ptrs"]):
        jg.jacobi_copy_out(h.h, g, p, device, stream=stream)
    return {"u": state["out"], **got}


def _solve_iters(size, tol):
    """About how many sweeps the slowest mode of a grid needs to fall to tol."""
    rate = sum(math.cos(math.pi / (n + 1)) for n in size) / 3.0
    return math.log(1.0 / tol) / -math.log(rate)


def work(case):
    kind = case["kind"]
    if kind == "channel":
        return {"bytes": 2 * case["bytes"], "flops": 0}
    e = ELEM[case["dtype"]]
    if kind == "serve":
        sizes = [s for s, _ in _requests(case, 0)]
    else:
        sizes = _sizes(case)
    points = [s[0] * s[1] * s[2] for s in sizes]
    padded = [(s[0] + 2) * (s[1] + 2) * (s[2] + 2) for s in sizes]
    if kind == "check":
        return {"bytes": padded[0] * e, "flops": 9 * points[0]}
    if kind == "step":
        return {"bytes": (sum(padded) + sum(points)) * e, "flops": (6 * case["iters"] + (9 if case["residual"] else 0)) * sum(points)}
    # a solve: its sweeps (estimated) with a residual every check_every of them; the server makes the state itself
    flops = sum(p * _solve_iters(s, case["tol"]) * (6 + 9 / case["check_every"]) for p, s in zip(points, sizes))
    return {"bytes": (sum(points) + (sum(padded) if kind == "solve" else 0)) * e, "flops": flops}


def _sweep(u, v):
    """One 64-bit sweep of the padded array u into the interior of v."""
    w = v[1:-1, 1:-1, 1:-1]
    torch.add(u[1:-1, 1:-1, :-2], u[1:-1, 1:-1, 2:], out=w)
    w += u[1:-1, :-2, 1:-1]
    w += u[1:-1, 2:, 1:-1]
    w += u[:-2, 1:-1, 1:-1]
    w += u[2:, 1:-1, 1:-1]
    w /= 6.0


def _norms(u):
    """(|b - A u|, |b|) of a padded array in 64 bits."""
    c = u[1:-1, 1:-1, 1:-1]
    r = u[1:-1, 1:-1, :-2] + u[1:-1, 1:-1, 2:] + u[1:-1, :-2, 1:-1] + u[1:-1, 2:, 1:-1] + u[:-2, 1:-1, 1:-1] + u[2:, 1:-1, 1:-1] - 6.0 * c
    b = torch.zeros_like(c)
    b[:, :, 0] += u[1:-1, 1:-1, 0]
    b[:, :, -1] += u[1:-1, 1:-1, -1]
    b[:, 0, :] += u[1:-1, 0, 1:-1]
    b[:, -1, :] += u[1:-1, -1, 1:-1]
    b[0] += u[0, 1:-1, 1:-1]
    b[-1] += u[-1, 1:-1, 1:-1]
    return float(r.norm()), float(b.norm())


def exact(case, seed):
    kind = case["kind"]
    if kind in ("serve", "channel"):
        return None
    fields = [u.double() for u in _fields(case, seed)]
    if kind == "check":
        r, b = _norms(fields[0])
        return torch.tensor([r, b, r / b if b > 0 else r], dtype=torch.float64)
    sizes = _sizes(case)
    offs, n = _offsets(sizes)
    out = torch.zeros(n, dtype=torch.float64, device="cuda")
    rel, res = [], []
    for u, s, o in zip(fields, sizes, offs):
        v = u.clone()
        for k in range(case["max_iters"] if kind == "solve" else case["iters"]):
            if kind == "solve" and k % case["check_every"] == 0:
                r, b = _norms(u)
                if r <= case["tol"] * b:
                    break
            _sweep(u, v)
            u, v = v, u
        if kind == "solve" or case["residual"]:
            r, b = _norms(u)
            rel.append(r / b if b > 0 else r)
            res.append(r)
        out[o:o + s[0] * s[1] * s[2]] = u[1:-1, 1:-1, 1:-1].reshape(-1)
        del v
    if kind == "solve":
        return {"u": out, "iters": None, "rel": np.array(rel), "status": None}
    if case["residual"]:
        return {"u": out, "rel": np.array(rel), "abs": np.array(res)}
    return {"u": out}
