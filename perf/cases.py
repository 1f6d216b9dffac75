"""What this framework's users have it do, as cases that can be timed.

Each case is one call a user's program makes again and again through the
public entry points: environmental selection of a merged population (one
call, or a batch of uneven populations), ranking, TensorHypE and TensorMOEA/D
selection, a whole generation on the device, the IGD of a population and the
dominance matrix. Inputs are seeded populations on the linear (sum f = 0.5)
and sphere (||f|| = 1) fronts of the package's workloads, made on the GPU.
"""
import math
import random

import numpy as np
import torch

from paper_2503_20286_gb300 import _binding as emo
from paper_2503_20286_gb300 import workloads as wl

SHAPES = {"linear": emo.EMO_SHAPE_LINEAR, "sphere": emo.EMO_SHAPE_SPHERE}


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the paper's small population (92 survivors, H = 12): the latency of one selection
        dict(name="select_184_m3", kind="select", n2=184, m=3, shape="linear", q=0, h=12, h2=0, keep=92, niche=0),
        # an everyday population: 10,000 survivors on 10,011 directions
        dict(name="select_20000_m3", kind="select", n2=20000, m=3, shape="sphere", q=0, h=140, h2=0, keep=10000,
             niche=0),
        # five objectives, an odd size, as many directions as survivors
        dict(name="select_39999_m5", kind="select", n2=39999, m=5, shape="linear", q=0, h=24, h2=0, keep=20000,
             niche=0),
        # many objectives on a coarse grid (ties and duplicates), two-layer directions, long niche lists
        dict(name="select_100000_m8_ties", kind="select", n2=100000, m=8, shape="sphere", q=64, h=3, h2=2,
             keep=50000, niche=0),
        # the largest: the benchmark's population
        dict(name="select_400000_m3", kind="select", n2=400000, m=3, shape="sphere", q=0, h=631, h2=0, keep=200000,
             niche=0),
        # 64 uneven populations in one call
        dict(name="batch_64", kind="batch", count=64, lo=1000, hi=40000, sizes=3),
        # complete non-dominated sorting of an odd-sized population
        dict(name="rank_20001_m3", kind="rank", n2=20001, m=3, shape="sphere", q=0, keep=0),
        # hypervolume-based selection with 10,000 Monte Carlo samples
        dict(name="hype_100001_m3", kind="hype", n2=100001, m=3, shape="sphere", q=0, samples=10000, keep=50000),
        # decomposition-based selection, 20 neighbours
        dict(name="moead_200028_m3", kind="moead", h=631, m=3, d=12, t=20, shape="sphere"),
        # one generation on the device (mating, SBX, mutation, evaluation, selection of 2N, gather)
        dict(name="generation_50000_m3", kind="generation", n=50000, m=3, d=12, shape="sphere", h=315, niche=0),
        # quality of a population against the true front
        dict(name="igd_200000_m3", kind="igd", n=200000, m=3, h=631, shape="sphere"),
        # the caller-order dominance matrix and counts
        dict(name="dominance_100000_m3", kind="dominance", n2=100000, m=3, shape="sphere", q=0, ws=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the same calls over their whole range of sizes."""
    kind = rng.choice(["select"] * 5 + ["batch", "rank", "hype", "moead", "generation", "igd", "dominance"])
    shape = rng.choice(["linear", "sphere"])
    if kind == "select":
        m = rng.choice([2, 3, 3, 3, 5, 8])
        n2 = _log_int(rng, 100, {2: 40000, 3: 400000, 5: 50000, 8: 100000}[m])
        keep = n2 // 2
        two = m == 8 and rng.random() < 0.5
        h, h2 = (3, 2) if two else (wl.h_for_count(min(keep, 1000) if m == 8 else keep, m), 0)
        q = 0 if rng.random() < 0.75 else (64 if m >= 5 else 1024)
        return dict(kind=kind, n2=n2, m=m, shape=shape, q=q, h=h, h2=h2, keep=keep, niche=int(rng.random() < 0.25))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(2, 64), lo=rng.choice([200, 1000]), hi=rng.choice([8000, 40000]),
                    sizes=rng.randint(10, 10**6))
    if kind == "rank":
        m = rng.choice([2, 3, 3, 5])
        n2 = _log_int(rng, 100, {2: 20000, 3: 100000, 5: 50000}[m])
        return dict(kind=kind, n2=n2, m=m, shape=shape, q=0 if rng.random() < 0.75 else 1024,
                    keep=rng.choice([0, n2 // 2]))
    if kind == "hype":
        n2 = _log_int(rng, 200, 120000)
        return dict(kind=kind, n2=n2, m=rng.choice([2, 3, 4]) if n2 < 20000 else 3, shape=shape, q=0,
                    samples=_log_int(rng, 500, 20000), keep=n2 // 2)
    if kind == "moead":
        m = rng.choice([2, 3, 3])
        return dict(kind=kind, h=wl.h_for_count(_log_int(rng, 100, 200000 if m == 3 else 20000), m), m=m,
                    d=m + 9, t=rng.randint(8, 24), shape=shape)
    if kind == "generation":
        n = _log_int(rng, 92, 150000)
        return dict(kind=kind, n=n, m=3, d=rng.choice([7, 12, 21]), shape=shape, h=wl.h_for_count(n, 3),
                    niche=int(rng.random() < 0.25))
    if kind == "igd":
        m = rng.choice([2, 3, 3, 5])
        n = _log_int(rng, 100, {2: 20000, 3: 200000, 5: 50000}[m])
        return dict(kind=kind, n=n, m=m, h=wl.h_for_count(_log_int(rng, 100, n), m), shape=shape)
    m = rng.choice([2, 3, 3, 5, 8])
    n2 = _log_int(rng, 100, 100000 if m <= 5 else 40000)
    # without a workspace the matrix is computed pair by pair
    ws = m <= 5 and (n2 > 40000 or rng.random() < 0.75)
    return dict(kind=kind, n2=n2, m=m, shape=shape, q=0 if rng.random() < 0.75 else 64, ws=ws)


# ------------------------------------------------------------------ inputs
def _gen(seed, stream=0):
    g = torch.Generator(device="cuda")
    g.manual_seed((seed * 1000003 + stream) & 0x7FFFFFFFFFFFFFFF)
    return g


def _decisions(n, d, seed, stream=0):
    return torch.rand(n, d, generator=_gen(seed, stream), device="cuda", dtype=torch.float32)


def _objectives(x, m, shape, q=0):
    """Stand-in objectives of decision vectors (FP64, rounded once to float32)."""
    x = x.double()
    g = ((x[:, m - 1:] - 0.5) ** 2).sum(1, keepdim=True)
    p = x[:, :m - 1]
    one = torch.ones_like(g)
    if shape == "sphere":
        a = p * (math.pi / 2)
        prod = torch.cat([one, torch.cumprod(torch.cos(a), 1)], 1)  # 1, cos a_0, cos a_0 cos a_1, ...
        s = torch.cat([prod[:, m - 1:], (prod[:, :m - 1] * torch.sin(a)).flip(1)], 1)
        f = (1.0 + g) * s
    else:
        rest = torch.cat([one, torch.cumprod(1.0 - p, 1)], 1)
        s = torch.cat([rest[:, :m - 1] * p, rest[:, m - 1:]], 1)
        f = 0.5 * (1.0 + 100.0 * g) * s
    if q:
        f = torch.round(f * q) / q
    return f.float().contiguous()


def _population(case, seed, stream=0):
    return _objectives(_decisions(case["n2"], case["m"] + 9, seed, stream), case["m"], case["shape"], case["q"])


def _lattice(h, m):
    """Compositions of h into m parts, lexicographic (int64 [n][m])."""
    rows, left = np.zeros((1, 0), np.int64), np.array([h], np.int64)
    for _ in range(m - 1):
        rep = left + 1
        first = np.repeat(np.cumsum(rep) - rep, rep)
        k = np.arange(rep.sum()) - first
        rows = np.concatenate([np.repeat(rows, rep, 0), k[:, None]], 1)
        left = np.repeat(left, rep) - k
    return np.concatenate([rows, left[:, None]], 1)


def _directions(h, m, h2=0):
    w = _lattice(h, m) / float(h)
    if h2:
        w = np.concatenate([w.astype(np.float32).astype(np.float64), 0.5 * (_lattice(h2, m) / float(h2)) + 0.5 / m])
    return torch.from_numpy(w.astype(np.float32)).cuda()


def _front(h, m, shape):
    w = torch.from_numpy(_lattice(h, m) / float(h)).cuda()
    return (0.5 * w if shape == "linear" else w / w.norm(dim=1, keepdim=True)).float().contiguous()


def _neighbours(h, m, t):
    """The t nearest weights of each lattice weight (m = 2 or 3), by squared
    distance, then offset; itself first."""
    c = torch.from_numpy(_lattice(h, m)).cuda()
    n = c.shape[0]
    if m == 2:
        off = [(a, -a) for a in range(-t, t + 1)]
    else:
        r = 12
        off = [(a, b, -a - b) for a in range(-r, r + 1) for b in range(-r, r + 1) if abs(a + b) <= r]
    off.sort(key=lambda o: (sum(v * v for v in o), o))
    off = torch.tensor(off, device="cuda")
    out = torch.empty(n, t, dtype=torch.int32, device="cuda")
    for lo in range(0, n, 32768):
        p = c[lo:lo + 32768, None, :] + off[None]
        ok = (p >= 0).all(2)
        pos = torch.where(ok, torch.arange(off.shape[0], device="cuda"), off.shape[0] * 2)
        near = p.gather(1, pos.sort(1).indices[:, :t, None].expand(-1, -1, m))  # the first t that exist
        i = near[..., 0]
        idx = i if m == 2 else i * (h + 1) - i * (i - 1) // 2 + near[..., 1]
        out[lo:lo + 32768] = idx.int()
    return out


def _batch_sizes(case):
    r = random.Random(case["sizes"])
    for b in range(case["count"]):
        n2 = 2 * round(math.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"]))) / 2)
        yield n2, r.choice([2, 3, 5]), ("linear", "sphere")[b % 2]


def prepare(case, seed):
    """What the user's program keeps between calls: inputs, outputs, a workspace."""
    dev, kind = "cuda", case["kind"]
    s = {"case": case, "seed": seed}
    if kind in ("select", "rank", "hype", "dominance"):
        s["F"] = _population(case, seed)
        n2, m = s["F"].shape
    if kind == "select":
        s["R"] = _directions(case["h"], m, case["h2"])
        s["survivors"] = torch.empty(case["keep"], dtype=torch.int32, device=dev)
        s["info"] = torch.zeros(8, dtype=torch.int32, device=dev)
        nbytes = emo.emo_workspace_size(emo.EMO_OP_NSGA3_SELECT, n2, m, s["R"].shape[0])
    elif kind == "batch":
        sizes = list(_batch_sizes(case))
        out = torch.empty(sum(n2 // 2 for n2, _, _ in sizes), dtype=torch.int32, device=dev)
        info = torch.zeros(len(sizes), 8, dtype=torch.int32, device=dev)
        s.update(survivors=out, info=info, problems=[])
        at = 0
        for b, (n2, m, shape) in enumerate(sizes):
            F = _population(dict(n2=n2, m=m, shape=shape, q=0), seed, stream=1000 + b)
            s["problems"].append(dict(F=F, R=_directions(wl.h_for_count(n2 // 2, m), m), n_keep=n2 // 2, seed=seed,
                                      generation=b, survivors=out[at:at + n2 // 2], info=info[b]))
            at += n2 // 2
        nbytes = emo.emo_batch_workspace_size(s["problems"])
    elif kind == "rank":
        s["rank"] = torch.empty(n2, dtype=torch.int32, device=dev)
        s["last"] = torch.empty(1, dtype=torch.int32, device=dev)
        nbytes = emo.emo_workspace_size(emo.EMO_OP_ND_RANK, n2, m, 0)
    elif kind == "hype":
        s["U"] = torch.rand(case["samples"], m, generator=_gen(seed, 7), device=dev)
        s["v_ref"] = (s["F"].max(0).values * 1.1).contiguous()
        s["survivors"] = torch.empty(case["keep"], dtype=torch.int32, device=dev)
        s["info"] = torch.zeros(8, dtype=torch.int32, device=dev)
        s["hv"] = torch.empty(n2, dtype=torch.float64, device=dev)
        nbytes = emo.emo_workspace_size(emo.EMO_OP_HYPE_SELECT, n2, m, case["samples"])
    elif kind == "moead":
        h, m, d, t = case["h"], case["m"], case["d"], case["t"]
        s["W"] = _directions(h, m)
        n = s["W"].shape[0]
        s["I"] = _neighbours(h, m, min(t, n))
        s["X"], s["O"] = _decisions(n, d, seed, 11), _decisions(n, d, seed, 12)
        s["F1"], s["F2"] = _objectives(s["X"], m, case["shape"]), _objectives(s["O"], m, case["shape"])
        s["z0"] = s["F1"].min(0).values.contiguous()
        s["z"] = s["z0"].clone()
        s["X_next"], s["F_next"] = torch.empty_like(s["X"]), torch.empty_like(s["F1"])
        s["winner"] = torch.empty(n, dtype=torch.int32, device=dev)
        s["status"] = torch.empty(1, dtype=torch.int32, device=dev)
        nbytes = emo.emo_workspace_size(emo.EMO_OP_MOEAD_SELECT, n, m, s["I"].shape[1])
    elif kind == "generation":
        n, m, d = case["n"], case["m"], case["d"]
        s["R"] = _directions(case["h"], m)
        s["X0"] = _decisions(n, d, seed, 5)
        s["F0"] = _objectives(s["X0"], m, case["shape"])
        s["X"], s["F"] = s["X0"].clone(), s["F0"].clone()
        s["info"] = torch.zeros(8, dtype=torch.int32, device=dev)
        nbytes = emo.emo_generation_workspace_size(n, d, m, s["R"].shape[0])
    elif kind == "igd":
        m = case["m"]
        s["F"] = _objectives(_decisions(case["n"], m + 9, seed), m, case["shape"])
        s["Ref"] = _front(case["h"], m, case["shape"])
        s["igd"] = torch.empty(1, dtype=torch.float64, device=dev)
        nbytes = emo.emo_workspace_size(emo.EMO_OP_IGD, s["Ref"].shape[0], m, 0)
    else:
        s["D"] = torch.empty(n2, (n2 + 31) // 32, dtype=torch.int32, device=dev)
        s["count"] = torch.empty(n2, dtype=torch.int32, device=dev)
        nbytes = emo.emo_workspace_size(emo.EMO_OP_DOMINANCE_WS, n2, m, 0) if case["ws"] else 0
    s["ws"] = torch.empty(max(nbytes, 256), dtype=torch.uint8, device=dev)
    return s


# ------------------------------------------------------------------ the calls
def run(s):
    case, seed, kind = s["case"], s["seed"], s["case"]["kind"]
    if kind == "select":
        emo.emo_nsga3_select(s["F"], s["R"], case["keep"], seed, 1, survivors=s["survivors"], info=s["info"],
                             ws=s["ws"], niche_mode=case["niche"])
        return {"survivors": s["survivors"], "info": s["info"]}
    if kind == "batch":
        emo.emo_nsga3_select_batch(s["problems"], ws=s["ws"])
        return {"survivors": s["survivors"], "info": s["info"]}
    if kind == "rank":
        emo.emo_nd_rank(s["F"], case["keep"], rank=s["rank"], last_rank=s["last"], ws=s["ws"])
        return {"rank": s["rank"], "last": s["last"]}
    if kind == "hype":
        emo.emo_hype_select(s["F"], s["v_ref"], s["U"], case["keep"], survivors=s["survivors"], info=s["info"],
                            hv=s["hv"], ws=s["ws"])
        return {"survivors": s["survivors"], "info": s["info"], "hv": s["hv"]}
    if kind == "moead":
        s["z"].copy_(s["z0"])  # z is updated in place: each pass starts from the same ideal point
        emo.emo_moead_select(s["X"], s["F1"], s["O"], s["F2"], s["z"], s["W"], s["I"], 5.0, X_next=s["X_next"],
                             F_next=s["F_next"], winner=s["winner"], status=s["status"], ws=s["ws"])
        return {"X_next": s["X_next"], "F_next": s["F_next"], "z": s["z"], "winner": s["winner"],
                "status": s["status"]}
    if kind == "generation":
        s["X"].copy_(s["X0"])  # the generation is in place: each pass starts from the same parents
        s["F"].copy_(s["F0"])
        emo.emo_nsga3_generation(s["X"], s["F"], s["R"], SHAPES[case["shape"]], seed, 1, niche_mode=case["niche"],
                                 info=s["info"], ws=s["ws"])
        return {"X": s["X"], "F": s["F"], "info": s["info"]}
    if kind == "igd":
        return {"igd": emo.emo_igd(s["F"], s["Ref"], out=s["igd"], ws=s["ws"])}
    if case["ws"]:
        emo.emo_dominance_ws(s["F"], D=s["D"], dom_count=s["count"], ws=s["ws"])
    else:
        emo.emo_dominance(s["F"], D=s["D"], dom_count=s["count"])
    return {"D": s["D"], "count": s["count"]}


# ------------------------------------------------------------------ least work
def work(case):
    """Inputs read once, outputs written once, and the operations no method
    does without: one comparison per point, objective and bit of its position
    for an order of the points, 3 m operations per distance that is reported
    or decided. Dominance bits, tiles and workspaces are the present code's
    own traffic and count as nothing (except where the matrix is the output)."""
    kind = case["kind"]

    def select(n2, m, n_r, keep):
        return 4 * (n2 * m + n_r * m + keep + 8), m * n2 * math.log2(max(n2, 2)) + 3 * m * keep

    def dirs(h, m):
        return wl.das_dennis_count(h, m)

    if kind == "select":
        n_r = dirs(case["h"], case["m"]) + (dirs(case["h2"], case["m"]) if case["h2"] else 0)
        b, f = select(case["n2"], case["m"], n_r, case["keep"])
    elif kind == "batch":
        b = f = 0
        for n2, m, _ in _batch_sizes(case):
            x = select(n2, m, dirs(wl.h_for_count(n2 // 2, m), m), n2 // 2)
            b, f = b + x[0], f + x[1]
    elif kind == "rank":
        n2, m = case["n2"], case["m"]
        b, f = 4 * (n2 * m + n2 + 1), m * n2 * math.log2(max(n2, 2))
    elif kind == "hype":
        n2, m, ns = case["n2"], case["m"], case["samples"]
        b = 4 * (n2 * m + ns * m + m + case["keep"] + 8) + 8 * n2
        f = m * (n2 + ns) * math.log2(max(n2, 2))
    elif kind == "moead":
        n, m, d = dirs(case["h"], case["m"]), case["m"], case["d"]
        b = 2 * n * d * 4 + 4 * n * m * 4 + n * case["t"] * 4 + 4 * n
        f = n * (12 * m + 6) + n * case["t"] * (8 * m + 4)
    elif kind == "generation":
        n, m, d = case["n"], case["m"], case["d"]
        x = select(2 * n, m, dirs(case["h"], m), n)
        b, f = x[0] + 4 * n * (5 * d + 4 * m), x[1] + 40 * n * d
    elif kind == "igd":
        n, m, nr = case["n"], case["m"], dirs(case["h"], case["m"])
        b, f = 4 * (n * m + nr * m) + 8, 3 * m * nr
    else:
        n2, m = case["n2"], case["m"]
        b = 4 * n2 * m + 4 * n2 * ((n2 + 31) // 32) + 4 * n2
        f = m * n2 * math.log2(max(n2, 2))
    return {"bytes": float(b), "flops": float(f)}


# ------------------------------------------------------------------ 64 bits
def _dominated(F):
    """Which rows are dominated by another row."""
    n, out = F.shape[0], torch.zeros(F.shape[0], dtype=torch.bool, device=F.device)
    for lo in range(0, n, 1024):
        q = F[lo:lo + 1024]
        le = torch.ones(q.shape[0], n, dtype=torch.bool, device=F.device)
        eq = torch.ones_like(le)
        for k in range(F.shape[1]):
            le &= F[None, :, k] <= q[:, k, None]
            eq &= F[None, :, k] == q[:, k, None]
        out[lo:lo + 1024] = (le & ~eq).any(1)
    return out


def _exact_hype(case, seed):
    s = prepare(case, seed)
    F, n2, m, keep = s["F"], s["F"].shape[0], s["F"].shape[1], case["keep"]
    alive, before = torch.arange(n2, device="cuda"), 0
    while True:  # fronts until `keep` points are ranked
        dom = _dominated(F[alive])
        last = alive[~dom]
        if before + last.numel() >= keep:
            break
        before, alive = before + last.numel(), alive[dom]
    k = before + last.numel() - keep
    fl = F.min(0).values
    S = fl + s["U"] * (s["v_ref"] - fl)  # the samples are float32 points
    c = torch.zeros(S.shape[0], dtype=torch.int64, device="cuda")
    for lo in range(0, n2, 4096):
        c += (F[lo:lo + 4096, None, :] <= S[None]).all(2).sum(0)
    alpha = torch.zeros(n2 + 2, dtype=torch.float64, device="cuda")
    if k >= 1:
        i = torch.arange(1, k, dtype=torch.float64, device="cuda")
        lam = torch.cat([torch.ones(1, dtype=torch.float64, device="cuda"), (k - i) / (n2 - i)])
        alpha[1:k + 1] = torch.cumprod(lam, 0) / torch.arange(1, k + 1, dtype=torch.float64, device="cuda")
    w = alpha[c]
    hv = torch.zeros(n2, dtype=torch.float64, device="cuda")
    vol = (s["v_ref"].double() - fl.double()).prod()
    for lo in range(0, last.numel(), 1024):
        p = last[lo:lo + 1024]
        d = (F[p][:, None, :] <= S[None]).all(2)
        hv[p] = torch.where(d, w, 0.0).sum(1) * vol / S.shape[0]
    return {"survivors": None, "info": None, "hv": hv}


def _exact_moead(case, seed):
    s = prepare(case, seed)
    n, t = s["I"].shape
    z = torch.minimum(s["z0"], s["F2"].min(0).values)
    W = s["W"].double()
    nw = W.norm(dim=1)

    def pbi(f, j):
        v, w = f.double() - z.double(), W[j]
        d1 = (v * w).sum(1).abs() / nw[j]
        return d1 + 5.0 * (v - (d1 / nw[j])[:, None] * w).norm(dim=1)

    own = pbi(s["F1"], torch.arange(n, device="cuda"))
    i = torch.arange(n, device="cuda").repeat_interleave(t)
    j = s["I"].reshape(-1).long()
    g = pbi(s["F2"][i], j)
    mark = g <= own[j]
    i, j, g = i[mark], j[mark], g[mark]
    best = torch.full((n,), math.inf, dtype=torch.float64, device="cuda").scatter_reduce_(0, j, g, "amin")
    at = g == best[j]
    first = torch.full((n,), n, dtype=torch.int64, device="cuda").scatter_reduce_(0, j[at], i[at], "amin")
    win = (best < own) | (first == 0)
    o = first.clamp(max=n - 1)[:, None]
    X = torch.where(win[:, None], s["O"].gather(0, o.expand(-1, s["O"].shape[1])), s["X"])
    F = torch.where(win[:, None], s["F2"].gather(0, o.expand(-1, s["F2"].shape[1])), s["F1"])
    return {"X_next": X.double(), "F_next": F.double(), "z": z.double(), "winner": None, "status": None}


def exact(case, seed):
    """The computed numbers in 64 bits; None for whole-number outputs, and for
    a generation, whose survivors follow from every step before them."""
    if case["kind"] == "hype":
        return _exact_hype(case, seed)
    if case["kind"] == "moead":
        return _exact_moead(case, seed)
    if case["kind"] == "igd":
        s = prepare(case, seed)
        F, Ref = s["F"].double(), s["Ref"].double()
        total = torch.zeros((), dtype=torch.float64, device="cuda")
        for lo in range(0, Ref.shape[0], 2048):
            r, d2 = Ref[lo:lo + 2048], 0.0
            for k in range(F.shape[1]):
                d2 = d2 + (r[:, k, None] - F[None, :, k]).square_()
            total += d2.min(1).values.sqrt().sum()
        return {"igd": (total / Ref.shape[0]).reshape(1)}
    return None
