"""What a user of the library has it do, as measurable cases.

One pass of most cases is one step of the method: ``pi_bin`` and
``pi_interact`` on device-resident positions (the two calls a simulation
makes per time step).  The others are a batch of uneven systems in one
``pi_batch_bin`` / ``pi_batch_interact``, and a set of jobs from and to
pinned host memory through the request loop.  Contexts and output arrays are
made once and kept, as a simulation or a server keeps them; the options stay
at their defaults except those a case names.

``listed`` covers the smallest systems of the batched and served mixes (1 k
particles) to 16.8 M, 1 to 32 particles per cell, uniform and clustered
layouts, plain and compensated sums, the Gaussian and Lennard-Jones kernels,
sorted and input-order outputs, cubic and other boxes.  ``draw`` gives more
cases of the same ranges.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2406_16091_gb300 import binding as B
from paper_2406_16091_gb300 import serving
from paper_2406_16091_gb300 import workloads as W

KERNELS = {"gaussian": B.PI_KERNEL_GAUSSIAN, "lj": B.PI_KERNEL_LJ, "lowflop": B.PI_KERNEL_LOWFLOP,
           "highflop": B.PI_KERNEL_HIGHFLOP}
# useful FLOP of one within-cutoff ordered pair: 3 (displacement), 5 (r^2), 1 (S), 6 (V) and the kernel value
FLOP_PER_PAIR = {"gaussian": 17, "lj": 24, "lowflop": 15, "highflop": 174}
CLUSTERS, SIGMA, BACKGROUND = 64, 0.03, 0.10  # the clustered layout of the precision study


def _step(name, n, ppc, **kw):
    case = {"name": name, "kind": "step", "n": n, "ppc": float(ppc), "layout": "uniform", "box": "unit",
            "kernel": "gaussian", "precision": "fp32", "order": "sorted", "h_div": 2.0}
    case.update(kw)
    return case


def listed():
    return [
        # the smallest system of the batched and served mixes: latency and launches
        _step("tiny_1531", 1531, 6),
        # the paper's plain method at its small size: 16^3 cells, 8 per cell
        _step("small_32768", 32768, 8),
        # an ordinary simulation: odd count, a box that is no cube, input-order outputs
        _step("slab_262147", 262147, 4, box="slab", order="original"),
        # the scale sweep: the benchmark's occupancy, the sparsest and the densest
        _step("scale_8", 2097152, 8),
        _step("scale_1", 2097152, 1, order="original"),
        _step("scale_32", 2097152, 32),
        # the precision study: clusters with a heavy-tailed occupancy, plain sums
        _step("clustered_4m", 4194304, 2, layout="clustered"),
        # the precision study's compensated sums on a smaller clustered system
        _step("kahan_clustered_1m", 1048573, 2, layout="clustered", precision="kahan"),
        # the potential the paper names, input-order outputs
        _step("lj_500009", 500009, 8, kernel="lj", order="original"),
        # many uneven systems in one set of launches (the batched workload, a quarter of its systems)
        {"name": "batch_64", "kind": "batch", "systems": 64, "n_lo": 1024, "n_hi": 262144, "shape_seed": 1004},
        # a queue of requests from pinned host memory, half clustered, through the native request loop
        {"name": "serve_12", "kind": "serve", "jobs": 12, "n_lo": 1024, "n_hi": 262144, "shape_seed": 1005},
        # the largest: past the L2
        _step("large_16m", 16777217, 8),
    ]


def draw(rng):
    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    kind = rng.choice(["step"] * 6 + ["batch", "serve"])
    if kind != "step":
        lo = int(log(1024, 8192))
        count = {"systems": rng.randint(3, 64)} if kind == "batch" else {"jobs": rng.randint(3, 12)}
        return {"kind": kind, **count, "n_lo": lo, "n_hi": int(log(2 * lo, 262144)),
                "shape_seed": rng.randrange(1 << 20)}
    layout = rng.choice(["uniform", "uniform", "clustered"])
    precision = rng.choice(["fp32", "fp32", "fp32", "kahan"])
    kernel = rng.choice(["gaussian"] * 4 + ["lj", "lowflop", "highflop"])
    ppc = log(1, 32) if layout == "uniform" else log(1, 16)
    # pairs grow as n * ppc: no drawn case costs more than the largest listed one
    room = 33.5e6 if layout == "uniform" else 6e6
    if precision == "kahan":
        room /= 3
    if kernel in ("lj", "highflop"):
        room /= 2 if kernel == "lj" else 6
    n = int(log(1000, min(8e6, room / ppc)))
    return _step("", n | rng.randint(0, 1), ppc, layout=layout, precision=precision, kernel=kernel,
                 order=rng.choice(["sorted", "original"]),
                 box=rng.choice(["unit", "slab"]) if layout == "uniform" else "unit",
                 h_div=rng.choice([2.0, 2.0, 2.0, 6.0]) if kernel == "gaussian" else 2.0)


# ---- sizes and inputs -------------------------------------------------------------------

def _system(n, ppc, layout="uniform", box="unit", h_div=2.0):
    """One system's box, cutoff and kernel length: cells of a mean occupancy of about ppc."""
    if box == "slab":
        # four times as wide as high, not at the origin
        lo, ext = (-2.0, 0.5, 10.0), (4.0, 3.0, 1.0)
        cells = max(1, round((n / ppc / 12.0) ** (1.0 / 3.0)))
    else:
        lo, ext = (0.0, 0.0, 0.0), (1.0, 1.0, 1.0)
        cells = max(3, round((n / ppc) ** (1.0 / 3.0)))
    hi = tuple(a + e for a, e in zip(lo, ext))
    rc = W.rc_for_cells(cells)
    return {"n": n, "lo": lo, "hi": hi, "rc": rc, "h": float(np.float32(rc) / np.float32(h_div)), "layout": layout}


def _systems(case):
    if case["kind"] == "step":
        return [_system(case["n"], case["ppc"], case["layout"], case["box"], case["h_div"])]
    rng = np.random.Generator(np.random.PCG64(case["shape_seed"]))
    out = []
    for k in range(case["systems"] if case["kind"] == "batch" else case["jobs"]):
        n = int(math.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]))))
        if case["kind"] == "batch":
            out.append(_system(n, rng.uniform(2.0, 16.0)))
        else:
            out.append(_system(n, float(rng.choice([2.0, 4.0, 8.0, 16.0])), "clustered" if k % 2 else "uniform"))
    return out


def _positions(sys, gen):
    """Device positions (x, y, z) of one system."""
    n, dev = sys["n"], gen.device
    if sys["layout"] == "uniform":
        cols = []
        for a, b in zip(sys["lo"], sys["hi"]):
            v = torch.rand(n, generator=gen, device=dev) * (b - a) + a
            cols.append(torch.clamp(v, a, float(np.nextafter(np.float32(b), np.float32(a)))))
        return cols
    n_cl = n - int(round(n * BACKGROUND))
    centres = torch.rand((CLUSTERS, 3), generator=gen, device=dev)
    parts, have = [torch.rand((n - n_cl, 3), generator=gen, device=dev)], 0
    while have < n_cl:
        which = torch.randint(CLUSTERS, (2 * (n_cl - have) + 64,), generator=gen, device=dev)
        p = centres[which] + SIGMA * torch.randn((len(which), 3), generator=gen, device=dev)
        p = p[((p >= 0) & (p < 1)).all(1)][: n_cl - have]
        parts.append(p)
        have += len(p)
    p = torch.cat(parts)[torch.randperm(n, generator=gen, device=dev)]
    p = torch.clamp(p, 0.0, float(np.nextafter(np.float32(1), np.float32(0))))
    return [p[:, d].contiguous() for d in range(3)]


def _inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return [(s, _positions(s, gen)) for s in _systems(case)]


class _Context:
    """A library handle that goes with the state that holds it."""

    def __init__(self, handle, destroy):
        self.handle, self._destroy = handle, destroy

    def __del__(self):
        self._destroy(self.handle)


# ---- what is measured ------------------------------------------------------------------

def prepare(case, seed):
    ins = _inputs(case, seed)
    state = {"case": case}
    if case["kind"] == "serve":
        # the server with its slots, and the jobs with their pinned blocks
        state["jobs"] = [serving.make_job(k, *(c.cpu().numpy() for c in pos), s["lo"], s["hi"], s["rc"], s["h"])
                         for k, (s, pos) in enumerate(ins)]
        caps = [c for c in (16384, 65536, 262144) if c < 4 * case["n_hi"]]
        state["server"] = serving.Server([(c, 4) for c in caps])
        state["guard"] = _Context(state["server"], serving.Server.close)
        return state
    pos = [torch.cat([p[d] for _, p in ins]) for d in range(3)]
    n = len(pos[0])
    if case["kind"] == "batch":
        ctx = B.pi_batch_create([(s["lo"], s["hi"]) for s, _ in ins], [s["rc"] for s, _ in ins],
                                [s["n"] for s, _ in ins])
        state["counts"], state["h"] = [s["n"] for s, _ in ins], [s["h"] for s, _ in ins]
    else:
        s = ins[0][0]
        ctx = B.pi_create(s["lo"], s["hi"], s["rc"], n)
        B.pi_set_option(ctx, B.PI_OPT_KERNEL, KERNELS[case["kernel"]])
        B.pi_set_option(ctx, B.PI_OPT_PRECISION,
                        B.PI_PREC_KAHAN if case["precision"] == "kahan" else B.PI_PREC_FP32)
        state["h"] = s["h"]
    out = {k: torch.empty(n, device="cuda") for k in ("S", "Vx", "Vy", "Vz")}
    out["nbr"] = torch.empty(n, dtype=torch.int32, device="cuda")
    if case.get("order") != "original":
        # sorted outputs: slot k belongs to input particle perm[k]
        out["perm"] = torch.empty(n, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    state.update(ctx=ctx, guard=_Context(ctx, B.pi_destroy), pos=pos, n=n, out=out)
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "serve":
        state["server"].run(state["jobs"])
        return [[j.S, j.Vx, j.Vy, j.Vz, j.nbr] for j in state["jobs"]]
    stream, out = torch.cuda.current_stream(), state["out"]
    args = (out["S"], out["Vx"], out["Vy"], out["Vz"], out["nbr"])
    if case["kind"] == "batch":
        B.pi_batch_bin(state["ctx"], *state["pos"], state["counts"], stream)
        B.pi_batch_interact(state["ctx"], state["h"], *args, B.PI_ORDER_SORTED, stream)
    else:
        order = B.PI_ORDER_ORIGINAL if case["order"] == "original" else B.PI_ORDER_SORTED
        B.pi_bin(state["ctx"], *state["pos"], state["n"], stream)
        B.pi_interact(state["ctx"], state["h"], *args, order, stream)
    if "perm" in out:
        B.pi_copy_binned(state["ctx"], perm=out["perm"], stream=stream)
    return out


def work(case):
    """Each position read once, each output written once; the FLOP of the expected within-cutoff pairs."""
    total_bytes = total_flops = 0.0
    for s in _systems(case):
        n, rc = s["n"], s["rc"]
        ext = [b - a for a, b in zip(s["lo"], s["hi"])]
        ball = 4.0 / 3.0 * math.pi * rc ** 3
        if s["layout"] == "uniform":
            # pair counts of a ball cut by the box's faces, to first order
            cut = math.prod(max(0.4, 1.0 - 3.0 / 8.0 * min(1.0, rc / e)) for e in ext)
            nbr = (n - 1) / math.prod(ext) * ball * cut
        else:
            # the mean density that a particle of a cluster sees (its own cluster, smeared over the cutoff), and the rest
            own = (1 - BACKGROUND) * n / CLUSTERS / (4 * math.pi * (SIGMA ** 2 + rc ** 2 / 10)) ** 1.5
            nbr = ball * ((1 - BACKGROUND) * own + n)
        total_bytes += n * (12 + 20 + (4 if case.get("order") != "original" and case["kind"] != "serve" else 0))
        total_flops += n * nbr * FLOP_PER_PAIR[case.get("kernel", "gaussian")]
    return {"bytes": int(total_bytes), "flops": int(total_flops)}


def tolerance(case):
    # about four times the distance from `exact` measured over these ranges: FP32 sums of up to some 30 (uniform, 8
    # per cell) to several hundred (dense clusters) terms, compensated sums, and terms whose own FP32 error counts
    # (Lennard-Jones).  The neighbour counts and the permutation are whole numbers, and exact.
    if case["kind"] == "serve" or case.get("layout") == "clustered" and case["precision"] == "fp32":
        return {"rel": 4e-6, "max": 8e-5}
    if case.get("precision") == "kahan" and case["kernel"] in ("gaussian", "lowflop"):
        return {"rel": 6e-7, "max": 4e-6}
    return {"rel": 2e-6, "max": 3e-5}


# ---- 64-bit reference ---------------------------------------------------------------------

def _exact_cells(pos, s):
    """The FP32 cell of each particle by its definition: clamp(floor((p - lo) * inv_w), 0, n - 1), x fastest."""
    dims = [max(1, int((b - a) / s["rc"])) for a, b in zip(s["lo"], s["hi"])]
    cell, mul = 0, 1
    for p, a, b, m in zip(pos, s["lo"], s["hi"], dims):
        inv = torch.tensor(m / (b - a), dtype=torch.float64).to(torch.float32).to(p.device)
        c = torch.floor((p - torch.tensor(a, dtype=torch.float32, device=p.device)) * inv).to(torch.int64)
        cell = cell + torch.clamp(c, 0, m - 1) * mul
        mul *= m
    return cell, dims


def _exact_system(pos, s, kernel):
    """Sums in 64 bits over the pairs that the FP32 cutoff test r2 < fl32(rc * rc) accepts, r2 = fma(dz, dz, fma(dy,
    dy, dx * dx)); cells of the grid only to find candidates.  In sorted order, with the stable permutation."""
    cell, (nx, ny, nz) = _exact_cells(pos, s)
    perm = torch.sort(cell, stable=True).indices
    cell = cell[perm]
    p = [c[perm] for c in pos]
    p64 = [c.double() for c in p]
    n, dev = len(cell), cell.device
    start = torch.searchsorted(cell, torch.arange(nx * ny * nz + 1, device=dev))
    cx, cy, cz = cell % nx, cell // nx % ny, cell // (nx * ny)
    rc2 = torch.tensor(np.float32(s["rc"]) * np.float32(s["rc"]), device=dev)
    h2 = float(np.float32(s["h"])) ** 2
    out = {k: torch.zeros(n, dtype=torch.float64, device=dev) for k in ("S", "Vx", "Vy", "Vz")}
    nbr = torch.zeros(n, dtype=torch.int32, device=dev)
    one = torch.ones(1, dtype=torch.int32, device=dev)
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            ok = (cy + dy >= 0) & (cy + dy < ny) & (cz + dz >= 0) & (cz + dz < nz)
            row = nx * ((cy + dy).clamp(0, ny - 1) + ny * (cz + dz).clamp(0, nz - 1))
            first = start[row + (cx - 1).clamp(min=0)]
            count = torch.where(ok, start[row + (cx + 1).clamp(max=nx - 1) + 1] - first, 0)
            ends = torch.cumsum(count, 0)
            a, done = 0, 0
            while a < n:
                # as many targets as 2^26 candidates cover
                b = max(a + 1, int(torch.searchsorted(ends, done + (1 << 26), right=True)))
                m = count[a:b]
                i = torch.repeat_interleave(torch.arange(a, b, device=dev), m)
                j = torch.arange(len(i), device=dev) - (ends[a:b] - m - done)[i - a] + first[i]
                done, a = int(ends[b - 1]), b
                d32 = [c[j] - c[i] for c in p]
                r2 = (d32[0] * d32[0]).double()
                for d in d32[1:]:
                    r2 = (d.double() * d.double() + r2).float().double()
                keep = torch.nonzero((r2.float() < rc2) & (i != j)).squeeze(1)
                i, j = i[keep], j[keep]
                d = [c[j] - c[i] for c in p64]
                r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
                if kernel == "gaussian":
                    K = torch.exp(-r2 / h2)
                elif kernel == "lowflop":
                    K = torch.ones_like(r2)
                else:
                    q = (h2 / (r2 + h2 / 100)) ** 3
                    K = 4 * (q * q - q)
                out["S"].index_add_(0, i, K)
                for k, c in zip(("Vx", "Vy", "Vz"), d):
                    out[k].index_add_(0, i, c * K)
                nbr.index_add_(0, i, one.expand(len(i)))
    out["nbr"] = nbr
    return out, perm


def exact(case, seed):
    res = []
    for s, pos in _inputs(case, seed):
        out, perm = _exact_system(pos, s, case.get("kernel", "gaussian"))
        if case["kind"] == "serve" or case.get("order") == "original":
            out = {k: torch.empty_like(v).index_copy_(0, perm, v) for k, v in out.items()}
        else:
            # the sorted slots of the systems follow each other, and so do their input particles
            out["perm"] = (perm + sum(len(r["S"]) for r in res)).to(torch.int32)
        res.append(out)
    if case["kind"] == "serve":
        return [[r[k].cpu() for k in ("S", "Vx", "Vy", "Vz", "nbr")] for r in res]
    return {k: torch.cat([r[k] for r in res]) for k in res[0]}
