"""What is timed when this framework is measured: simulations as its users run them.

A pass enqueues sweeps of lattices that a program already holds and reads back what
such a program keeps: the (M, E) of every sweep and the configuration (or, of a scan,
the moments).  The chain goes on from pass to pass.  Sizes and temperatures are those
of the package's workloads (single lattices from L = 64 to 65,536, the 64-temperature
scan, uneven batches, serving requests, cubes) and the row widths of its tests.
"""
import math
import random

import numpy as np
import torch

from paper_1903_11714_gb300 import ising, serve, workloads


def listed():
    return [
        # the smallest call: one sweep at a time with a look at (M, E) and the lattice, as a
        # program does that watches or steers a small system
        {"name": "watch_64", "kind": "packed", "L": 64, "beta": workloads.BETA_TC, "hot": True, "sweeps": 1},
        # a small lattice for a long time at the critical point
        {"name": "small_128", "kind": "packed", "L": 128, "beta": workloads.BETA_TC, "hot": True, "sweeps": 1000},
        # rows of an odd number of words, in the disordered phase
        {"name": "ragged_320", "kind": "packed", "L": 320, "beta": 0.40, "hot": True, "sweeps": 300},
        # an ordinary single lattice, as one point of a scan
        {"name": "medium_1024", "kind": "packed", "L": 1024, "beta": 0.45, "hot": False, "sweeps": 400},
        # the headline lattice: 4.3e9 spins at the critical point
        {"name": "large_65536", "kind": "packed", "L": 65536, "beta": workloads.BETA_TC, "hot": True, "sweeps": 50},
        # the temperature scan, 64 replicas, with the moments of each temperature's new samples
        {"name": "scan_64x1024", "kind": "scan", "count": 64, "L": 1024, "beta0": 0.35, "beta1": 0.55, "sweeps": 200},
        # a batch of lattices of uneven size and temperature, made from arrays
        {"name": "uneven_32", "kind": "uneven", "count": 32, "smallest": 64, "largest": 2048, "pick": 4,
         "sweeps": 300},
        # a serving loop: requests of uneven size and length, batched as they come
        {"name": "serve_24", "kind": "serve", "count": 24, "largest": 2048, "most_sweeps": 1000, "pick": 5},
        # the plain byte-per-spin kernel
        {"name": "bytes_4096", "kind": "int8", "L": 4096, "beta": workloads.BETA_TC, "hot": True, "sweeps": 100},
        # a small cube, as in the 3D Binder scan
        {"name": "cube_128", "kind": "cubic", "L": 128, "beta": workloads.BETA_C3, "hot": False, "sweeps": 200},
        # a large cube at the critical point
        {"name": "cube_1024", "kind": "cubic", "L": 1024, "beta": workloads.BETA_C3, "hot": True, "sweeps": 20},
        # lattices in the caller's own device memory, swept without any allocation
        {"name": "own_memory_4", "kind": "noalloc", "L0": 256, "L1": 1024, "count": 4, "beta0": 0.38, "beta1": 0.50,
         "sweeps": 100},
    ]


def _log(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def _side(rng, a, b, unit=64):
    return unit * max(1, round(_log(rng, a, b) / unit))


def _sweeps(rng, sites, most_sweeps, most_flips):
    return max(1, min(round(_log(rng, 1, most_sweeps)), int(most_flips // sites)))


def draw(rng):
    kind = rng.choice(["packed"] * 5 + ["scan", "uneven", "serve", "int8", "int8", "cubic", "cubic", "noalloc"])
    beta = rng.uniform(0.30, 0.60)
    hot = rng.random() < 0.6
    if kind == "packed":
        L = _side(rng, 64, 32768)
        return {"kind": kind, "L": L, "beta": beta, "hot": hot, "sweeps": _sweeps(rng, L * L, 2000, 2e10)}
    if kind == "scan":
        L, count = _side(rng, 64, 1280), rng.randint(8, 96)
        return {"kind": kind, "count": count, "L": L, "beta0": 0.35, "beta1": rng.uniform(0.45, 0.60),
                "sweeps": max(10, _sweeps(rng, count * L * L, 1000, 1.3e10))}
    if kind == "uneven":
        top = 64 << rng.randint(2, 6)
        count = rng.randint(6, 64) if top <= 1024 else rng.randint(4, 16)
        return {"kind": kind, "count": count, "smallest": 64, "largest": top, "pick": rng.randint(0, 10 ** 6),
                "sweeps": max(2, _sweeps(rng, count * top * top // 5, 500, 1e10))}
    if kind == "serve":
        return {"kind": kind, "count": rng.randint(6, 32), "largest": _side(rng, 512, 2560),
                "most_sweeps": round(_log(rng, 200, 1000)), "pick": rng.randint(0, 10 ** 6)}
    if kind == "int8":  # whole 64-byte segments, or sides that are only a multiple of 8
        L = _side(rng, 64, 8192) if rng.random() < 0.6 else _side(rng, 32, 4096, unit=8)
        return {"kind": kind, "L": L, "beta": beta, "hot": hot, "sweeps": _sweeps(rng, L * L, 500, 3e9)}
    if kind == "cubic":
        L = _side(rng, 64, 1024)
        return {"kind": kind, "L": L, "beta": workloads.BETA_C3 * rng.uniform(0.9, 1.1), "hot": hot,
                "sweeps": _sweeps(rng, L ** 3, 500, 2e10)}
    return {"kind": kind, "L0": _side(rng, 64, 512), "L1": _side(rng, 512, 4096), "count": rng.randint(1, 8),
            "beta0": 0.38, "beta1": rng.uniform(0.40, 0.60), "sweeps": round(_log(rng, 1, 200))}


def _spread(a, b, count):
    return [a + (b - a) * k / max(1, count - 1) for k in range(count)]


def _lattices(case, seed):
    """(L, beta, seed, start) of every lattice of a case of several."""
    n, key = case["count"], 1_000_003 * (seed + 1)
    if case["kind"] == "scan":
        return [(case["L"], b, key + k, ising.COLD) for k, b in enumerate(_spread(case["beta0"], case["beta1"], n))]
    if case["kind"] == "noalloc":
        sides = [64 * max(1, round(s / 64)) for s in _spread(case["L0"], case["L1"], n)]
        return [(L, b, key + k, ising.HOT) for k, (L, b) in enumerate(zip(sides, _spread(case["beta0"], case["beta1"], n)))]
    # powers of two as in the uneven batch, one in four of them half as large again
    rng, steps = random.Random(case["pick"]), int(math.log2(case["largest"] // case["smallest"]))
    out = []
    for k in range(n):
        L = case["smallest"] << rng.randint(0, steps)
        if rng.random() < 0.25 and 3 * L // 2 <= case["largest"] and L >= 128:
            L = 3 * L // 2
        out.append((L, rng.uniform(0.30, 0.60), key + k, rng.choice([ising.HOT, ising.COLD])))
    return out


def _requests(case, seed):
    rng, out = random.Random(case["pick"]), []
    for k in range(case["count"]):
        out.append(workloads.Request(rid=k, arrival=float(k // 3), L=_side(rng, 256, case["largest"]),
                                     beta=rng.uniform(0.35, 0.55), seed=1_000_003 * (seed + 1) + k,
                                     sweeps=round(_log(rng, 100, case["most_sweeps"]))))
    return out


def _pinned(shape, dtype):
    return torch.empty(shape, dtype=dtype, pin_memory=True).numpy()


def prepare(case, seed):
    kind, key = case["kind"], 1_000_003 * (seed + 1)
    state = {"case": case, "done": 0}
    if kind in ("packed", "cubic", "int8"):
        L, start = case["L"], ising.HOT if case["hot"] else ising.COLD
        if kind == "cubic":
            state["lattice"] = ising.Lattice3D(L, case["beta"], key, start)
        else:
            state["lattice"] = ising.Lattice(L, case["beta"], key, start, ising.PACKED if kind == "packed" else ising.INT8)
        if kind == "int8":
            state["spins"] = _pinned((L, L), torch.int8)
        else:
            words = (L if kind == "packed" else L * L) * (L // 64)
            state["planes"] = [_pinned((words,), torch.int32).view(np.uint32) for _ in range(2)]
    elif kind in ("scan", "uneven"):
        Ls, betas, seeds, starts = zip(*_lattices(case, seed))
        state["batch"] = ising.Batch.from_arrays(Ls, betas, seeds, starts)
    elif kind == "serve":
        state["requests"] = _requests(case, seed)
        state["server"] = serve.Server(hbm_budget_bytes=1 << 28, slots=64, max_L=case["largest"])
    else:
        lattices = _lattices(case, seed)
        gen = torch.Generator(device="cuda").manual_seed(seed)
        state["planes"] = [[torch.randint(-2 ** 31, 2 ** 31, (L * L // 64,), dtype=torch.int32, device="cuda", generator=gen)
                            for _ in range(2)] for L, _, _, _ in lattices]
        state["me"] = [torch.zeros(2 * case["sweeps"], dtype=torch.int64, device="cuda") for _ in lattices]
        state["lattices"] = lattices
    return state


def run(state):
    case = state["case"]
    n, first = case.get("sweeps", 0), state["done"]
    state["done"] = first + n
    if "server" in state:
        results, _ = state["server"].serve(state["requests"], realtime=False, keep_history=True)
        results.sort(key=lambda r: r.rid)
        return {"M": np.array([r.M for r in results]), "E": np.array([r.E for r in results]),
                "history": np.concatenate([np.stack(r.history) for r in results], axis=1)}
    if "batch" in state:
        b = state["batch"]
        b.run(n)
        M, E = (np.stack(v) for v in zip(*(b.history(k, first, n) for k in range(case["count"]))))
        if case["kind"] == "uneven":
            return {"M": M, "E": E, "spins": np.concatenate([b.get_lattice(k).ravel() for k in range(case["count"])])}
        moments = [b.moments(k, first) for k in range(case["count"])]
        return {"M": M, "E": E, "moments": np.array([[m[q] for q in _MOMENTS] for m in moments])}
    if "me" in state:
        Ls, betas, seeds, _ = zip(*state["lattices"])
        ising.ising_sweep_packed_noalloc([p[0].data_ptr() for p in state["planes"]], [p[1].data_ptr() for p in state["planes"]],
                                         Ls, betas, seeds, first, n, [m.data_ptr() for m in state["me"]],
                                         torch.cuda.current_stream(), wait=False)
        return {"planes": [p for pair in state["planes"] for p in pair], "me": state["me"]}
    lat = state["lattice"]
    lat.sweep(n)
    M, E = lat.history(first, n)
    if case["kind"] == "int8":
        # the C entry point itself, into page-locked memory that the program keeps
        rc = ising.lib().ising_get_lattice(lat.h, ising._ptr(state["spins"], ising.ctypes.c_int8))
        if rc != ising.ISING_OK:
            raise ising.IsingError(rc, ising.last_error())
        return {"M": M, "E": E, "spins": state["spins"]}
    black, white = lat.get_planes(*state["planes"])
    return {"M": M, "E": E, "black": black.view(np.int32), "white": white.view(np.int32)}


_MOMENTS = ("abs_m", "m2", "m4", "e", "e2", "binder")


def _sites(case):
    """(sites, sweeps) of every lattice that a pass sweeps."""
    if case["kind"] == "serve":
        return [(r.L ** 2, r.sweeps) for r in _requests(case, 0)]
    if case["kind"] in ("packed", "int8", "cubic"):
        return [(case["L"] ** (3 if case["kind"] == "cubic" else 2), case["sweeps"])]
    return [(L * L, case["sweeps"]) for L, _, _, _ in _lattices(case, 0)]


def work(case):
    """Bytes: each lattice read and written once and its (M, E) written.  Operations, per
    32 sites and update: two Philox4x32-10 calls (the bit planes that decide nearly every
    site) of 20 32-bit products (two halves each) and 20 three-input exclusive-ors, a
    comparison of each of their eight planes (two logic operations) and the neighbour
    count (15, of six neighbours 25)."""
    per_word = 2 * (40 + 20 + 8) + (25 if case["kind"] == "cubic" else 15)
    bits = 8 if case["kind"] == "int8" else 1
    sites = _sites(case)
    return {"bytes": sum(2 * s * bits / 8 + 16 * n for s, n in sites), "flops": sum(s * n for s, n in sites) * per_word / 32}


# ---- the scan in plain torch, 64-bit integers throughout

def _philox(k0, k1, c0, c1, c2):
    """Philox4x32-10 of the counter words (c0, c1, c2, 0) under keys (k0, k1)."""
    low = 0xFFFFFFFF
    x = [c0, c1, c2, torch.zeros_like(c1)]
    for r in range(10):
        a, b = x[0] * 0xD2511F53, x[2] * 0xCD9E8D57  # modulo 2^64: both halves are right
        r0, r1 = (k0 + r * 0x9E3779B9) & low, (k1 + r * 0xBB67AE85) & low
        x = [((b >> 32) & low) ^ x[1] ^ r0, b & low, ((a >> 32) & low) ^ x[3] ^ r1, a & low]
    return x


def _uniforms(k0, k1, sweep, colour, L):
    """The 32-bit uniforms [R, L, L/2] of one colour's sites, less 2^31 (as int32)."""
    words = L * L // 64
    q = torch.arange(8 * words, device=k0.device)[None, :].expand(k0.shape[0], -1)
    out = _philox(k0, k1, torch.full_like(q, sweep), q, torch.full_like(q, colour))
    planes = torch.stack(out, dim=-1).view(-1, words, 32)  # plane 31 - k of word g at [g, k]
    planes = torch.where(planes >= 2 ** 31, planes - 2 ** 32, planes).to(torch.int32)
    bit = torch.arange(32, dtype=torch.int32, device=k0.device)
    u = torch.zeros(planes.shape, dtype=torch.int32, device=k0.device)
    for k in range(32):
        u = (u << 1) | ((planes[:, :, k, None] >> bit) & 1)
    return (u ^ -2 ** 31).view(-1, L, L // 2)


def exact(case, seed):
    if case["kind"] != "scan" or sum(s * n for s, n in _sites(case)) > 1.5e10:
        return None  # every output is a whole number, or it would take too long
    L, n, lattices = case["L"], case["sweeps"], _lattices(case, seed)
    N = L * L
    key = torch.tensor([k for _, _, k, _ in lattices], device="cuda")[:, None]
    k0, k1 = key & 0xFFFFFFFF, (key >> 32) & 0xFFFFFFFF
    # U < T_h = ceil(exp(-2 beta h) 2^32), as int32 values less 2^31 (T_h < 2^32: beta > 0)
    T = [torch.tensor([math.ceil(math.exp(-2 * b * h) * 2 ** 32) - 2 ** 31 for _, b, _, _ in lattices], dtype=torch.int32,
                      device="cuda")[:, None, None] for h in (2, 4)]
    spins = torch.ones((len(lattices), L, L), dtype=torch.int8, device="cuda")
    M, E = [], []

    def pick(a, c):  # the colour's sites, [R, L, L/2]: column 2m + ((i + c) & 1) of row i
        v = a.view(-1, L // 2, 2, L // 2, 2)
        return torch.stack([v[:, :, 0, :, c], v[:, :, 1, :, 1 - c]], dim=2).reshape(-1, L, L // 2)

    for s in range(n):
        for c in (0, 1):
            h = spins * (spins.roll(1, 1) + spins.roll(-1, 1) + spins.roll(1, 2) + spins.roll(-1, 2))
            h, u = pick(h, c), _uniforms(k0, k1, s, c, L)
            flip = (h <= 0) | ((h == 2) & (u < T[0])) | ((h == 4) & (u < T[1]))
            turn = (1 - 2 * flip.to(torch.int8)).view(-1, L // 2, 2, L // 2)
            v = spins.view(-1, L // 2, 2, L // 2, 2)
            v[:, :, 0, :, c] *= turn[:, :, 0]
            v[:, :, 1, :, 1 - c] *= turn[:, :, 1]
        M.append(spins.sum((1, 2), dtype=torch.int64))
        E.append(-(spins * (spins.roll(-1, 1) + spins.roll(-1, 2))).sum((1, 2), dtype=torch.int64))
    M, E = (torch.stack(v, dim=1).cpu().numpy() for v in (M, E))
    rows = []
    for m, e in zip(M.tolist(), E.tolist()):  # whole-number sums, divided once
        m2, m4 = sum(v * v for v in m) / (n * N ** 2), sum(v ** 4 for v in m) / (n * N ** 4)
        rows.append([sum(map(abs, m)) / (n * N), m2, m4, sum(e) / (n * N), sum(v * v for v in e) / (n * N ** 2),
                     1 - m4 / (3 * m2 * m2)])
    return {"M": M, "E": E, "moments": np.array(rows)}
