"""The work that users of this framework have it do, as timed cases.

A case is a dict of plain values.  ``listed()`` gives the fixed ones,
``draw(rng)`` another of the same ranges, ``prepare(case, seed)`` the state a
program holds before the call (points on the GPU, a prepared ``Lloyd``
workspace), ``run(state)`` one pass through the package's public entry points,
``work(case)`` the bytes and operations a pass cannot do without and
``exact(case, seed)`` the same outputs in 64 bits.

The points are seeded Gaussian mixtures, the package's own recipe (means
uniform in a box, one sigma per component, Dirichlet weights, rows in random
order; heavy-tailed outliers where a case says so), drawn on the GPU.
"""
import math

import numpy as np
import torch

import paper_1908_02136_gb300 as kpp

DEVICE = "cuda:0"
SPECIALISED = (2, 4, 8, 16, 32, 64, 128)
BYTES = {"f32": 4, "bf16": 2, "fp8": 1}


def listed():
    return [
        # k-means++ of a small two-dimensional set: the call's latency counts
        {"name": "seed_small", "kind": "seed", "N": 10_000, "d": 2, "K": 16, "dtype": "f32",
         "comps": 16, "box": 10.0, "sigma_lo": 1.0, "sigma_hi": 1.0, "equal": True,
         "outliers": 0.0},
        # k-means++ of a million points of a usual embedding width
        {"name": "seed_1e6_d32", "kind": "seed", "N": 1_000_000, "d": 32, "K": 256,
         "dtype": "f32", "comps": 256, "outliers": 0.0},
        # a width and a number of rows that are no power of two (d = 50 is a
        # common word-vector size)
        {"name": "seed_odd_d50", "kind": "seed", "N": 300_007, "d": 50, "K": 100,
         "dtype": "f32", "comps": 100, "outliers": 0.0},
        # k-means++ far beyond L2, FP32 and stored as BF16
        {"name": "seed_1e7_d64", "kind": "seed", "N": 10_000_000, "d": 64, "K": 1024,
         "dtype": "f32", "comps": 1024, "outliers": 0.0},
        {"name": "seed_1e7_d64_bf16", "kind": "seed", "N": 10_000_000, "d": 64, "K": 1024,
         "dtype": "bf16", "comps": 1024, "outliers": 0.0},
        # the largest set, stored as FP8 with row scales, a tenth of it
        # heavy-tailed outliers
        {"name": "seed_2e7_d128_fp8", "kind": "seed", "N": 20_000_000, "d": 128, "K": 2048,
         "dtype": "fp8", "comps": 2048, "outliers": 0.1},
        # hundreds of uneven problems in one call
        {"name": "batch_512", "kind": "batch", "n": 512, "table": 1000},
        # one Lloyd iteration of a clustering loop: a usual size, a ragged one
        # and a large one
        {"name": "lloyd_1e6_d32", "kind": "lloyd", "N": 1_000_000, "d": 32, "K": 256},
        {"name": "lloyd_odd_d100", "kind": "lloyd", "N": 250_007, "d": 100, "K": 77},
        {"name": "lloyd_1e7_d64", "kind": "lloyd", "N": 10_000_000, "d": 64, "K": 1024},
        # k-means|| as the initialisation of a medium and a large problem
        {"name": "kmpar_1e6_d32", "kind": "kmpar", "N": 1_000_000, "d": 32, "K": 256},
        {"name": "kmpar_1e7_d64", "kind": "kmpar", "N": 10_000_000, "d": 64, "K": 1024},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["seed", "seed", "seed", "batch", "lloyd", "lloyd", "kmpar"])
    if kind == "batch":
        return {"kind": "batch", "n": _log_int(rng, 16, 512), "table": rng.randrange(1 << 30)}
    if kind == "seed":
        d = rng.choice(SPECIALISED) if rng.random() < 0.6 else _log_int(rng, 3, 300)
        N = _log_int(rng, 1_000, 10_000_000)
        while N * d > 1_280_000_000:
            N = _log_int(rng, 1_000, 10_000_000)
        K = min(N, _log_int(rng, 4, 1024))
        # other widths than the specialised ones run slower: keep the cost of
        # a drawn case below the largest listed one
        most = 600_000_000_000 if d in SPECIALISED else 20_000_000_000
        K = max(2, min(K, most // (N * d)))
        return {"kind": "seed", "N": N, "d": d, "K": K, "dtype": rng.choice(["f32", "f32", "bf16", "fp8"]),
                "comps": max(1, int(K * rng.choice([0.25, 1.0, 1.0, 2.0]))),
                "outliers": rng.choice([0.0, 0.0, 0.1])}
    d = rng.choice(SPECIALISED) if rng.random() < 0.5 else rng.randint(2, 128)
    N = _log_int(rng, 5_000, 10_000_000)
    if kind == "lloyd":
        return {"kind": "lloyd", "N": N, "d": d, "K": _log_int(rng, 2, 2048)}
    return {"kind": "kmpar", "N": N, "d": d, "K": max(4, min(_log_int(rng, 8, 1024), N // 20))}


# ---------------------------------------------------------------------------
# Inputs.
# ---------------------------------------------------------------------------
def _mixture(N, d, comps, seed, box=50.0, sigma_lo=0.5, sigma_hi=2.0, equal=False, outliers=0.0):
    """Points [N, d] float32 of a seeded mixture, and a fresh draw of every
    component [comps, d] (one point near the middle of each cluster)."""
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)

    def uniform(*shape):
        return torch.rand(*shape, generator=g, device=DEVICE)

    means = (2 * uniform(comps, d) - 1) * box
    sig = sigma_lo + (sigma_hi - sigma_lo) * uniform(comps)
    w = torch.ones(comps, device=DEVICE) if equal else -torch.log(1 - uniform(comps))
    edges = torch.cumsum(w.double(), 0)
    edges = edges / edges[-1]
    x = torch.empty(N, d, device=DEVICE)
    step = max(1, (1 << 27) // d)
    for s in range(0, N, step):
        e = min(N, s + step)
        lab = torch.searchsorted(edges, uniform(e - s).double()).clamp_(max=comps - 1)
        z = x[s:e].normal_(generator=g)
        z.mul_(sig[lab, None]).add_(means[lab])
    if outliers:
        rows = torch.randperm(N, generator=g, device=DEVICE)[:int(outliers * N)]
        for part in rows.split(step):
            # 10 * Student-t(3), centred at the origin
            chi2 = torch.zeros(len(part), d, device=DEVICE)
            for _ in range(3):
                chi2 += torch.randn(len(part), d, generator=g, device=DEVICE).square()
            z = torch.randn(len(part), d, generator=g, device=DEVICE)
            x[part] = 10.0 * z / torch.sqrt(chi2 / 3.0)
    near = means + sig[:, None] * torch.randn(comps, d, generator=g, device=DEVICE)
    return x, near


def _seed_points(case, seed):
    return _mixture(case["N"], case["d"], case["comps"], seed, case.get("box", 50.0),
                    case.get("sigma_lo", 0.5), case.get("sigma_hi", 2.0),
                    case.get("equal", False), case["outliers"])[0]


def _batch_sizes(case):
    """(N, d, K) of every problem: N log-uniform in [1e3, 2e5], d from {8, 16,
    32, 64, 128}, K log-uniform in [8, 256]."""
    rng = np.random.default_rng(case["table"])
    out = []
    for _ in range(case["n"]):
        N = int(round(math.exp(rng.uniform(math.log(1_000), math.log(200_000)))))
        d = int((8, 16, 32, 64, 128)[rng.integers(5)])
        out.append((N, d, min(N, int(round(math.exp(rng.uniform(math.log(8), math.log(256))))))))
    return out


def _batch_points(case, seed):
    return [_mixture(N, d, K, seed * 100_003 + p)[0]
            for p, (N, d, K) in enumerate(_batch_sizes(case))]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "seed":
        x, scales = _seed_points(case, seed), None
        if case["dtype"] == "bf16":
            x = kpp.quantize(x, "bf16")
        elif case["dtype"] == "fp8":
            x, scales = kpp.quantize(x, "fp8")
        return {"kind": kind, "x": x, "scales": scales, "K": case["K"], "seed": seed}
    if kind == "batch":
        sizes = _batch_sizes(case)
        Ns, Ks = [N for N, _, _ in sizes], [K for _, _, K in sizes]
        # one buffer per kind of result, a slice of it for every problem
        flat = [torch.empty(sum(Ks), dtype=torch.int64, device=DEVICE),
                torch.empty(sum(Ns), dtype=torch.float32, device=DEVICE),
                torch.empty(len(sizes), dtype=torch.float64, device=DEVICE)]
        outs = list(zip(flat[0].split(Ks), flat[1].split(Ns), flat[2].split(1)))
        return {"kind": kind, "xs": _batch_points(case, seed), "Ks": Ks,
                "seeds": [seed] * len(sizes), "outs": outs, "flat": flat}
    if kind == "lloyd":
        x, centres = _mixture(case["N"], case["d"], case["K"], seed)
        return {"kind": kind, "lloyd": kpp.Lloyd(x, case["K"]), "centres": centres}
    x = _mixture(case["N"], case["d"], case["K"], seed)[0]
    return {"kind": kind, "x": x, "K": case["K"], "seed": seed}


def run(state):
    kind = state["kind"]
    if kind == "seed":
        return list(kpp.seed(state["x"], state["K"], state["seed"], row_scales=state["scales"]))
    if kind == "batch":
        kpp.seed_batched(state["xs"], state["Ks"], state["seeds"], outs=state["outs"])
        return state["flat"]
    if kind == "lloyd":
        return list(state["lloyd"].step(state["centres"]))
    r = kpp.kmeans_par(state["x"], state["K"], state["seed"])
    # the number of candidates varies with the data: fixed room for the lists
    return [r["idx"], _padded(r["cand"], state["K"]), _padded(r["weights"], state["K"]),
            r["labels"], r["d2"], r["phi"]]


def _padded(t, K):
    return torch.nn.functional.pad(t, (0, 16 * K + 64 - len(t)), value=-1)


def _seed_work(N, d, K, dtype):
    points = N * d * BYTES[dtype] + (4 * N if dtype == "fp8" else 0)
    return points + 4 * N + 8 * K + 8, 3 * N * d * K


def work(case):
    kind = case["kind"]
    if kind == "seed":
        b, f = _seed_work(case["N"], case["d"], case["K"], case["dtype"])
        return {"bytes": b, "flops": f}
    if kind == "batch":
        parts = [_seed_work(N, d, K, "f32") for N, d, K in _batch_sizes(case)]
        return {"bytes": sum(b for b, _ in parts), "flops": sum(f for _, f in parts)}
    N, d, K = case["N"], case["d"], case["K"]
    if kind == "lloyd":
        # points and centres in; labels, D^2, new centres, counts and phi out
        return {"bytes": 4 * N * d + 8 * K * d + 8 * N + 8 * K + 8,
                "flops": 2 * N * K * d + 4 * N * d}
    # five rounds of 2K expected candidates each, searched over all points,
    # then K draws over the candidates
    cand = 1 + 10 * K
    return {"bytes": 4 * N * d + 8 * N + 16 * cand + 8 * K + 8,
            "flops": 2 * N * cand * d + 3 * cand * K * d}


# ---------------------------------------------------------------------------
# The same outputs in 64 bits (torch and numpy alone).
# ---------------------------------------------------------------------------
def _uniforms(seed, n, counter1=0, counter2=0, stream=0):
    """u_0 .. u_{n-1}: word 0 of Philox4x64-10 at counters {i, counter1,
    counter2, 0}, key {seed, stream}.  numpy steps the counter before each block,
    so it starts one below {0, counter1, counter2, 0}."""
    c = ((counter1 << 64 | counter2 << 128) - 1) % (1 << 256)
    words = [(c >> (64 * i)) & (2**64 - 1) for i in range(4)]
    bits = np.random.Philox(key=np.array([seed, stream], dtype=np.uint64),
                            counter=np.array(words, dtype=np.uint64))
    w0 = bits.random_raw(4 * n)[::4]
    return torch.from_numpy((w0 >> np.uint64(11)).astype(np.float64) * 2.0**-53).to(DEVICE)


def _first(u0, N):
    return torch.clamp((u0 * N).floor().long(), max=N - 1)


def _sq_to(x, c):
    """Squared distances in 64 bits of the rows of x to the one centre c."""
    out = torch.empty(x.shape[0], dtype=torch.float64, device=x.device)
    step = max(1, (1 << 28) // x.shape[1])
    for s in range(0, x.shape[0], step):
        out[s:s + step] = (x[s:s + step] - c).square_().sum(1)
    return out


def _draw(values, u):
    """The first index whose prefix sum exceeds u times the total."""
    cum = torch.cumsum(values, 0)
    i = torch.searchsorted(cum, (u * cum[-1]).reshape(1), right=True)[0]
    return torch.clamp(i, max=len(values) - 1)


def _seeding64(x, K, seed, stream=0):
    u = _uniforms(seed, K, stream=stream)
    idx = [_first(u[0], x.shape[0])]
    d2 = _sq_to(x, x[idx[0]])
    for m in range(1, K):
        idx.append(_draw(d2, u[m]))
        d2 = torch.minimum(d2, _sq_to(x, x[idx[-1]]))
    return [torch.stack(idx), d2, d2.sum().reshape(1)]


def _stored64(x, dtype):
    """The stored values of the points, as 64-bit numbers."""
    if dtype == "f32":
        return x.double()
    if dtype == "bf16":
        return x.bfloat16().double()
    top = x.abs().amax(1)
    # a tensor divisor: torch multiplies by the rounded reciprocal of a number
    s = torch.where(top > 0, top / torch.full_like(top, 448.0), torch.ones_like(top))
    q = (x / s[:, None]).clamp_(-448.0, 448.0).to(torch.float8_e4m3fn)
    return q.double() * s.double()[:, None]


def _nearest64(x, c):
    """(index of the nearest row of c, squared distance to it), in 64 bits:
    the index from the expanded form, the distance from the difference."""
    lab = torch.empty(x.shape[0], dtype=torch.int64, device=x.device)
    d2 = torch.empty(x.shape[0], dtype=torch.float64, device=x.device)
    cn = c.square().sum(1)
    step = max(1, (1 << 28) // max(len(c), x.shape[1]))
    for s in range(0, x.shape[0], step):
        part = x[s:s + step].double()
        lab[s:s + step] = torch.addmm(cn, part, c.T, alpha=-2.0).argmin(1)
        d2[s:s + step] = (part - c[lab[s:s + step]]).square_().sum(1)
    return lab, d2


def _lloyd64(x, centres):
    K, c = centres.shape[0], centres.double()
    lab, d2 = _nearest64(x, c)
    counts = torch.bincount(lab, minlength=K)
    sums = torch.zeros_like(c)
    step = max(1, (1 << 27) // x.shape[1])
    for s in range(0, x.shape[0], step):
        sums.index_add_(0, lab[s:s + step], x[s:s + step].double())
    means = torch.where(counts[:, None] > 0, sums / counts.clamp(min=1)[:, None], c)
    return [lab.int(), d2, means, counts, d2.sum().reshape(1)]


def _kmpar64(x, K, seed):
    x = x.double()
    N, ell = x.shape[0], 2.0 * K
    cand = [_first(_uniforms(seed, 1)[0], N).reshape(1)]
    lab = torch.zeros(N, dtype=torch.int64, device=x.device)
    d2 = _sq_to(x, x[cand[0][0]])
    have = 1
    for r in range(5):
        new = torch.nonzero(_uniforms(seed, N, r + 1) < ell * d2 / d2.sum())[:, 0]
        cand.append(new)
        if len(new):
            near, dist = _nearest64(x, x[new])
            lab = torch.where(dist < d2, near + have, lab)
            d2 = torch.minimum(d2, dist)
            have += len(new)
    cand = torch.cat(cand)
    w = torch.bincount(lab, minlength=len(cand))
    u = _uniforms(seed, K, 0, 1)
    c = x[cand]
    pick = [_draw(w.double(), u[0])]
    near = _sq_to(c, c[pick[0]])
    for m in range(1, K):
        pick.append(_draw(w * near, u[m]))
        near = torch.minimum(near, _sq_to(c, c[pick[-1]]))
    return [cand[torch.stack(pick)], _padded(cand, K), _padded(w, K), lab.int(), d2,
            d2.sum().reshape(1)]


def _steady(sizes):
    """Whether a seeding's D^2 has one 64-bit value.  A draw changes when its
    threshold falls within the rounding of a 32-bit D^2 of a prefix boundary
    -- a chance of about 4e-8 sqrt(N) -- and every later draw with it."""
    return sum(K * math.sqrt(N) for N, _, K in sizes) * 4e-8 < 0.015


def exact(case, seed):
    kind = case["kind"]
    if kind == "seed":
        if not _steady([(case["N"], case["d"], case["K"])]):
            return None
        x = _stored64(_seed_points(case, seed), case["dtype"])
        return _seeding64(x, case["K"], seed)
    if kind == "batch":
        if not _steady(_batch_sizes(case)):
            return None
        # problem p draws from stream p
        parts = [_seeding64(x.double(), K, seed, p) for p, (x, (_, _, K)) in
                 enumerate(zip(_batch_points(case, seed), _batch_sizes(case)))]
        return [torch.cat(t) for t in zip(*parts)]
    N, d, K = case["N"], case["d"], case["K"]
    x, centres = _mixture(N, d, K, seed)
    if kind == "lloyd":
        return None if N * d * K > 2_000_000_000_000 else _lloyd64(x, centres)
    return None if N * d * K > 100_000_000_000 else _kmpar64(x, K, seed)
