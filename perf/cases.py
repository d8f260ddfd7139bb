"""What this framework's speed is measured on: one pass of each of its main paths, called as a
user's program calls them, with sizes from the repository's own workloads and the ranges around
them. Sizes follow the synthetic workloads of workloads/gen.py: kernels with 128-point spaces,
full 16,384-point spaces ("dense") and random subsets of the axes ("uneven", 64 to 16,384 points).
"""

import math

import numpy as np
import torch

import paper_1701_08547_gb300 as T
from paper_1701_08547_gb300.surrogate import Surrogate
from workloads import archs as A
from workloads import gen
from workloads import mlp

DEV = "cuda"
INF = float("inf")
ALL_ARCHS = "sm_20,sm_35,sm_52,sm_60,sm_100,sm_103"
FLOP_PER_ROW = 2 * (48 * 256 + 3 * 256 * 256 + 256)  # the surrogate's forward, one row and member


def listed():
    return [
        # An interactive tool ranks the 128-point spaces of one program's kernels: launch-bound.
        {"name": "eval_small", "kind": "eval", "n": 64, "space": "small", "k": 5, "chunk": 0},
        # The headline workload: full spaces of 100,000 kernels, ten best each.
        {"name": "eval_dense", "kind": "eval", "n": 100_000, "space": "dense", "k": 10, "chunk": 1},
        # A corpus of kernels with spaces of every size, through the work queue that tune_autotune picks.
        {"name": "eval_uneven", "kind": "eval", "n": 1_000_000, "space": "uneven", "k": 5, "chunk": 4},
        # Every point's occupancy and cost written out (plots, training labels).
        {"name": "points_uneven", "kind": "points", "n": 20_000, "space": "uneven", "k": 5},
        # One corpus against every GPU generation of the architecture table.
        {"name": "archs_uneven", "kind": "archs", "n": 50_000, "space": "uneven", "k": 5, "archs": ALL_ARCHS},
        # Ranking measured or predicted scores: one inference chunk (few long segments) ...
        {"name": "topk_few", "kind": "topk", "segments": 64, "shortest": 16_384, "longest": 16_384, "k": 10},
        # ... and a corpus of spaces of all sizes, ragged offsets.
        {"name": "topk_ragged", "kind": "topk", "segments": 20_000, "shortest": 64, "longest": 16_384, "k": 5},
        # Simplex search of the statically pruned spaces with a budget of 128 evaluations.
        {"name": "search_pruned", "kind": "search", "n": 100_000, "space": "dense", "method": "nelder_mead",
         "budget": 128, "prune": True},
        # The ensemble's forward over one inference chunk.
        {"name": "forward_bf16", "kind": "forward", "rows": 1 << 20, "members": 5, "mode": "bf16"},
        # The same on E4M3 codes, an odd number of rows.
        {"name": "forward_fp8", "kind": "forward", "rows": 100_003, "members": 5, "mode": "fp8"},
        # Training on 51,141 labels (the kept ones of 64,000 timed samples) for two epochs, the weights read at the end.
        {"name": "train", "kind": "train", "rows": 51_141, "members": 5, "batch": 8192, "epochs": 2},
        # Every point of 1,000 kernels ranked by the ensemble, analytic fallback where its members disagree.
        {"name": "infer_uneven", "kind": "infer", "n": 1000, "space": "uneven", "k": 5, "members": 5, "mode": "bf16"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "points", "archs", "topk", "topk", "search", "forward", "forward",
                       "train", "infer"])
    k = rng.randint(1, 16)
    if kind == "eval":
        space = rng.choice(["small", "dense", "uneven"])
        n = _log_int(rng, 1, {"small": 1_000_000, "dense": 100_000, "uneven": 1_000_000}[space])
        return {"kind": kind, "n": n, "space": space, "k": k, "chunk": rng.choice([0, 0, 1, 4, 16])}
    if kind == "points":
        space = rng.choice(["small", "dense", "uneven"])
        return {"kind": kind, "n": _log_int(rng, 16, {"small": 200_000, "dense": 6_000, "uneven": 20_000}[space]),
                "space": space, "k": k}
    if kind == "archs":
        names = ALL_ARCHS.split(",")
        rows = rng.sample(names, rng.randint(1, len(names)))
        return {"kind": kind, "n": _log_int(rng, 64, 50_000), "space": rng.choice(["dense", "uneven"]), "k": k,
                "archs": ",".join(rows)}
    if kind == "topk":
        segments = _log_int(rng, 1, 20_000)
        longest = _log_int(rng, 64, min(1 << 20, 100_000_000 // segments))
        return {"kind": kind, "segments": segments, "shortest": max(1, longest // rng.choice([1, 2, 16, 256])),
                "longest": longest, "k": k}
    if kind == "search":
        return {"kind": kind, "n": _log_int(rng, 64, 100_000), "space": rng.choice(["dense", "uneven"]),
                "method": rng.choice(["nelder_mead", "random"]), "budget": rng.randint(16, 128),
                "prune": rng.random() < 0.5}
    if kind == "forward":
        return {"kind": kind, "rows": _log_int(rng, 1, 1 << 20), "members": rng.randint(1, 5),
                "mode": rng.choice(["bf16", "fp8"])}
    if kind == "train":
        return {"kind": kind, "rows": _log_int(rng, 1000, 51_141), "members": rng.randint(1, 5),
                "batch": rng.choice([1024, 2048, 4096, 8192]), "epochs": rng.randint(1, 2)}
    return {"kind": kind, "n": _log_int(rng, 1, 1000), "space": rng.choice(["small", "uneven"]), "k": k,
            "members": rng.randint(2, 5), "mode": rng.choice(["bf16", "fp8"])}


# ---- inputs -------------------------------------------------------------------------------


def _rng(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _axis_masks(n, width, size, g):
    """n random subsets of `size` (tensor [n]) of `width` positions, as int64 bit masks."""
    rank = torch.rand((n, width), generator=g, device=DEV).argsort(1)
    bits = torch.where(rank < size[:, None], 1, 0) << torch.arange(width, device=DEV)
    return bits.sum(1)


def _fields(n, space, seed):
    """The synthetic descriptors' fields: counts log-uniform in [1e2, 1e6], r0 in [16, 96], s0 in
    [0, 48 KB], d in [0, 0.5), and the space's four axis masks (t, g, u, c)."""
    g = _rng(seed)
    u = torch.rand((n, 7), generator=g, device=DEV, dtype=torch.float64)
    f = {"counts": torch.exp(math.log(1e2) + (math.log(1e6) - math.log(1e2)) * u).round().float(),
         "r0": torch.randint(16, 97, (n,), generator=g, device=DEV),
         "s0": torch.randint(0, 49153, (n,), generator=g, device=DEV),
         "d": 0.5 * torch.rand(n, generator=g, device=DEV)}
    full = torch.ones(n, dtype=torch.int64, device=DEV)
    if space == "uneven":
        log_s = (6 + 10 * torch.rand(n, generator=g, device=DEV)).clamp(max=14.0)
        f["masks"] = [_axis_masks(n, w, torch.exp2(log_s * b / 14).round(), g)
                      for w, b in ((32, 5), (16, 4), (8, 3), (4, 2))]
    elif space == "dense":
        f["masks"] = [full * m for m in (0xFFFFFFFF, 0xFFFF, 0xFF, 0xF)]
    else:  # 32 thread counts x unroll {1, 2, 4, 8}
        f["masks"] = [full * m for m in (0xFFFFFFFF, 1 << 10, 0x8B, 1 << 3)]
    return f


def _descs(f):
    """The fields as 64-byte descriptor records (uint8 [n, 64])."""
    n = f["r0"].numel()
    t, g, u, c = f["masks"]
    rec = torch.zeros((n, 16), dtype=torch.int32, device=DEV)
    rec[:, :7] = f["counts"].view(torch.int32)
    rec[:, 7], rec[:, 8] = f["r0"].int(), f["s0"].int()
    rec[:, 9] = f["d"].view(torch.int32)
    rec[:, 10] = torch.where(t >= 1 << 31, t - (1 << 32), t).int()
    rec[:, 11] = (g | (u << 16) | (c << 24)).int()
    return rec.view(torch.uint8)


def _count(mask, width):
    return ((mask[:, None] >> torch.arange(width, device=DEV)) & 1).sum(1)


def _sizes(f):
    t, g, u, c = f["masks"]
    return _count(t, 32) * _count(g, 16) * _count(u, 8) * _count(c, 4)


def _offsets(sizes):
    off = torch.zeros(sizes.numel() + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(sizes, 0, out=off[1:])
    return off


def _room(case):
    """Points that a program keeps room for (the spaces' total differs from corpus to corpus)."""
    n = case["n"]
    most = n * (128 if case["space"] == "small" else 16384)
    return most if case["space"] != "uneven" else min(most, int(n * _mean_space("uneven")[0] + 40_000 * math.sqrt(n)))


def _segments(case, seed):
    """Segment offsets with lengths log-uniform in [shortest, longest]."""
    g = _rng(seed)
    lo, hi = math.log2(case["shortest"]), math.log2(case["longest"])
    u = torch.rand(case["segments"], generator=g, device=DEV)
    return _offsets(torch.exp2(lo + (hi - lo) * u).round().long()), g


def _weights(members, seed):
    """An ensemble whose members agree up to a few percent, as trained ones do."""
    base = mlp.init_params(1, [seed % 100_000])
    rng = np.random.default_rng(seed + 1)
    noise = mlp.init_params(members, [int(s) for s in rng.integers(1 << 30, size=members)])
    return (np.tile(base, members) + np.float32(0.05) * noise).astype(np.float32)


def _samples(rows, seed):
    """rows random points of dense kernels: features, and the logarithm of their analytic cost, standardised."""
    n = 256
    f = _fields(n, "dense", seed)
    d = _descs(f)
    arch, ax = A.arch("sm_103"), gen.axes()
    cost = torch.empty(n * 16384, dtype=torch.float32, device=DEV)
    T.tune_eval(arch, ax, d, 1, flags=T.TUNE_EMIT_POINTS, pt_cost=cost, pt_offsets=_offsets(_sizes(f)))
    valid = torch.isfinite(cost).nonzero().flatten()
    pick = valid[torch.randint(valid.numel(), (rows,), generator=_rng(seed + 1), device=DEV)]
    feats = T.tune_features(arch, ax, d, pick // 16384, (pick % 16384).int())
    lab = torch.log(cost[pick])
    return feats, ((lab - lab.mean()) / lab.std()).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind, "case": case, "arch": A.arch("sm_103"), "axes": gen.axes()}
    if kind in ("eval", "points", "archs", "search", "infer"):
        f = _fields(case["n"], case["space"], seed)
        st["descs"] = _descs(f)
    if kind == "eval":
        chunk = case["chunk"]
        st["flags"] = T.TUNE_SCHED_WARP | (T.TUNE_SCHED_CHUNK(chunk.bit_length() - 1) if chunk else 0)
    elif kind == "points":
        st["off"] = _offsets(_sizes(f))
        n = _room(case)
        st["pt"] = [torch.zeros(n, dtype=dt, device=DEV) for dt in (torch.int32, torch.int32, torch.float32)]
    elif kind == "archs":
        st["archs"] = [A.arch(name) for name in case["archs"].split(",")]
    elif kind == "topk":
        st["off"], g = _segments(case, seed)
        n = int(st["off"][-1])
        st["scores"] = torch.exp(math.log(1e6) * torch.rand(n, generator=g, device=DEV))
    elif kind == "search":
        st["keep"] = T.tune_suggest(st["arch"], st["axes"], st["descs"])["t_star"] if case["prune"] else None
        st["seed"] = seed
    elif kind in ("forward", "infer"):
        st["sur"] = Surrogate(members=case["members"], batch=128)
        st["sur"].set_params(_weights(case["members"], seed))
        st["sur"].set_forward_mode({"bf16": Surrogate.FWD_FUSED_BF16, "fp8": Surrogate.FWD_FUSED_FP8}[case["mode"]])
        if kind == "forward":
            st["feats"] = _samples(case["rows"], seed)[0]
        else:
            st["off"] = _offsets(_sizes(f)).cpu().numpy()
    elif kind == "train":
        st["feats"], st["labels"] = _samples(case["rows"], seed)
        g = _rng(seed + 2)
        order = [torch.randperm(case["rows"], generator=g, device=DEV) for _ in range(case["epochs"])]
        st["order"] = torch.cat(order).int()
        st["sur"] = Surrogate(members=case["members"], batch=case["batch"])
        st["sur"].set_params(mlp.init_params(case["members"], [seed % 1000 + m for m in range(case["members"])]))
        steps = -(-case["rows"] // case["batch"])
        st["trace"] = torch.zeros((case["epochs"], steps, case["members"]), dtype=torch.float32, device=DEV)
    return st


def run(st):
    kind, case = st["kind"], st["case"]
    if kind == "eval":
        return T.tune_eval(st["arch"], st["axes"], st["descs"], case["k"], flags=st["flags"])
    if kind == "points":
        b, w, c = st["pt"]
        top = T.tune_eval(st["arch"], st["axes"], st["descs"], case["k"], flags=T.TUNE_EMIT_POINTS, pt_blocks=b,
                          pt_warps=w, pt_cost=c, pt_offsets=st["off"])
        return top[0], top[1], b, w, c
    if kind == "archs":
        return T.tune_eval_archs(st["archs"], st["axes"], st["descs"], case["k"])
    if kind == "topk":
        return T.tune_topk(st["scores"], st["off"], case["k"])
    if kind == "search":
        return T.tune_search(st["arch"], st["axes"], st["descs"], case["method"], case["budget"], st["seed"],
                             t_keep=st["keep"])
    if kind == "forward":
        return st["sur"].forward(st["feats"])
    if kind == "train":
        st["sur"].train(st["feats"], st["labels"], st["order"], case["epochs"], st["trace"])
        return st["trace"], st["sur"].get(Surrogate.GET_PARAMS)
    return st["sur"].infer(st["arch"], st["axes"], st["descs"], st["off"], case["k"], 0.1)


# ---- the least work of a pass --------------------------------------------------------------


def _mean_space(space):
    """Mean points and (T, U, C) triples of a kernel's space."""
    if space == "dense":
        return 16384.0, 1024.0
    if space == "small":
        return 128.0, 128.0
    log_s = np.minimum(6 + 10 * (np.arange(4000) + 0.5) / 4000, 14.0)
    t, g, u, c = (np.rint(np.exp2(log_s * b / 14)) for b in (5, 4, 3, 2))
    return float((t * g * u * c).mean()), float((t * u * c).mean())


def _mean_segment(case):
    lo, hi = case["shortest"], case["longest"]
    return float(lo) if lo == hi else (hi - lo) / math.log(hi / lo)


def work(case):
    kind = case["kind"]
    if kind in ("eval", "archs", "points"):
        rows = len(case["archs"].split(",")) if kind == "archs" else 1
        points, triples = _mean_space(case["space"])
        b = case["n"] * (64 + rows * 8 * case["k"])
        # eight operations rank a (T, U, C) triple: block limit, warps, latency factor, cost, bound
        fl = case["n"] * rows * triples * 8
        if kind == "points":
            b += case["n"] * (points * 12 + 8)
            fl += case["n"] * points
        return {"bytes": b, "flops": fl}
    if kind == "topk":
        n = case["segments"] * _mean_segment(case)
        return {"bytes": 4 * n + case["segments"] * (8 + 8 * case["k"]), "flops": n}
    if kind == "search":
        return {"bytes": case["n"] * (64 + 12 + (4 if case["prune"] else 0)), "flops": case["n"] * case["budget"] * 40}
    params = case["members"] * mlp.P * 4
    if kind == "forward":
        return {"bytes": case["rows"] * (128 + 4 * case["members"]) + params,
                "flops": case["rows"] * case["members"] * FLOP_PER_ROW}
    if kind == "train":
        n = case["rows"] * case["epochs"]
        return {"bytes": n * 136 + 2 * params, "flops": 3 * n * case["members"] * FLOP_PER_ROW}
    points = case["n"] * _mean_space(case["space"])[0]
    return {"bytes": case["n"] * (64 + 8 + 8 * case["k"] + 1) + params,
            "flops": points * (8 + case["members"] * FLOP_PER_ROW)}


# ---- the same results in 64 bits, in plain torch --------------------------------------------


def _costs64(arch, ax, f, rows):
    """Cost of every point of the full axes for kernels `rows` of the fields, [n, T, G, U, C], +inf
    where no block fits or the point is outside the kernel's space."""
    ten = {k: torch.tensor(v, device=DEV) for k, v in ax.items()}
    n = rows.numel()
    cnt, d = f["counts"][rows].double(), f["d"][rows].double()
    r0, s0 = f["r0"][rows], f["s0"][rows]
    wb = (ten["t"] + 31) // 32
    gw = torch.where(ten["t"] <= arch["max_threads_block"],
                     (arch["max_warps_sm"] // wb).clamp(max=arch["max_blocks_sm"]), 0)
    R = r0[:, None] + 4 * (ten["u"] - 1)                                   # [n, U]
    unit = arch["reg_alloc_unit"]
    if arch["reg_alloc_mode"] == 0:
        rpw = ((R * 32 + unit - 1) // unit * unit).clamp(min=1)
        gran = arch["warp_alloc_gran"]
        warps = arch["regs_sm"] // rpw // gran * gran
        gr = torch.where(rpw[:, None] * wb[:, None] > arch["regs_block_max"], 0, warps[:, None] // wb[:, None])
    else:
        rpb = ((R[:, None] * 32 * wb[:, None] + unit - 1) // unit * unit).clamp(min=1)
        gr = torch.where(rpb > arch["regs_block_max"], 0, arch["regs_sm"] // rpb)
    gr = torch.where((R > arch["regs_thread_max"])[:, None], 0, gr)         # [n, T, U]
    al = arch["smem_alloc_unit"]
    s_alloc = (s0 + arch["smem_reserved_block"] + al - 1) // al * al
    gs = torch.zeros((n, ten["c"].numel()), dtype=torch.int64, device=DEV)
    for cap in reversed(arch["smem_caps"]):                                 # the smallest that serves wins
        ok = (100 * cap >= ten["c"] * arch["smem_caps"][-1])[None] & (cap >= s_alloc)[:, None]
        gs = torch.where(ok, (cap // s_alloc.clamp(min=1))[:, None], gs)
    gs = torch.where((s_alloc == 0)[:, None], arch["max_blocks_sm"], gs)
    gs = torch.where((s0 > arch["smem_block_max"])[:, None], 0, gs)
    B = torch.minimum(torch.minimum(gw[None, :, None], gr)[..., None], gs[:, None, None])  # [n, T, U, C]
    ok = B > 0
    Bp = B.clamp(min=1)
    c = [cnt[:, i] / arch["ipc"][i] for i in range(7)]
    dk = (1 + d) * arch["work_scale"]
    cm = ((c[3] + c[4]) * dk)[:, None, None, None]
    cnm = ((c[0] + c[1] + c[2] + c[6])[:, None] + c[5][:, None] / ten["u"]) * dk[:, None]
    hide = (arch["w_sat"] / (Bp * wb[:, None, None]).double()).clamp(min=1.0)
    lane = (32 * wb).double() / ten["t"]
    x = (cnm[:, None, :, None] + cm * hide) * lane[:, None, None]
    slots = arch["n_sm"] * Bp
    G = ten["g"][:, None, None]
    waves = (G + slots[:, :, None] - 1) // slots[:, :, None]
    cost = x[:, :, None] * (waves * slots[:, :, None]).double() / (arch["n_sm"] * G).double()
    m = [(f["masks"][i][rows][:, None] >> torch.arange(w, device=DEV)) & 1 for i, w in enumerate((32, 16, 8, 4))]
    inside = m[0][:, :, None, None, None] * m[1][:, None, :, None, None] * m[2][:, None, None, :, None] * \
        m[3][:, None, None, None]
    cost = torch.where(ok[:, :, None], cost, INF)
    return cost, inside.bool()


def _exact_eval(arch, ax, f, k, points):
    top, every = [], []
    n = f["r0"].numel()
    for i in range(0, n, 512):
        cost, inside = _costs64(arch, ax, f, torch.arange(i, min(i + 512, n), device=DEV))
        if points:
            every.append(cost[inside])  # canonical order: T, G, U, C with C fastest
        cost = torch.where(inside, cost, INF).flatten(1)
        top.append(cost.topk(k, 1, largest=False, sorted=True).values)
    return torch.cat(top), torch.cat(every) if points else None


def _forward64(w, x):
    """One member's output and hidden values for rows x (64-bit), w: its weights."""
    h = x
    for layer in range(1, 5):
        h = torch.nn.functional.gelu(h @ w["W%d" % layer].T + w["b%d" % layer], approximate="tanh")
    return h @ w["w5"] + w["b5"]


def _members64(flat, members):
    return [{name: torch.tensor(v, dtype=torch.float64, device=DEV) for name, v in m.items()}
            for m in mlp.unpack(flat, members)]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("eval", "points", "archs"):
        rows = len(case["archs"].split(",")) if kind == "archs" else 1
        if case["n"] * rows > 120_000:  # over 20 seconds
            return None
        f = _fields(case["n"], case["space"], seed)
        names = case["archs"].split(",") if kind == "archs" else ["sm_103"]
        got = [_exact_eval(A.arch(name), gen.axes(), f, case["k"], kind == "points") for name in names]
        if kind == "archs":
            return None, torch.stack([t for t, _ in got])
        if kind == "eval":
            return None, got[0][0]
        every = torch.zeros(_room(case), dtype=torch.float64, device=DEV)
        every[:got[0][1].numel()] = got[0][1]
        return None, got[0][0], None, None, every
    if kind == "topk":
        off, g = _segments(case, seed)
        scores = torch.exp(math.log(1e6) * torch.rand(int(off[-1]), generator=g, device=DEV)).double()
        out = torch.full((case["segments"], case["k"]), INF, dtype=torch.float64, device=DEV)
        host = off.tolist()
        for s in range(case["segments"]):
            v = scores[host[s]:host[s + 1]]
            m = min(case["k"], v.numel())
            out[s, :m] = v.topk(m, largest=False, sorted=True).values
        return None, out
    if kind == "forward":
        x = _samples(case["rows"], seed)[0].double()
        out = torch.empty((case["members"], case["rows"]), dtype=torch.float64, device=DEV)
        if case["rows"] * case["members"] > 6_000_000:  # over 20 seconds of 64-bit products
            return None
        for m, w in enumerate(_members64(_weights(case["members"], seed), case["members"])):
            for i in range(0, case["rows"], 65536):
                out[m, i:i + 65536] = _forward64(w, x[i:i + 65536])
        return out
    if kind == "train":
        # Adam on the mean squared error, learning rate 1e-3, betas (0.9, 0.999), epsilon 1e-8
        feats, labels = _samples(case["rows"], seed)
        x, y = feats.double(), labels.double()
        g = _rng(seed + 2)
        order = [torch.randperm(case["rows"], generator=g, device=DEV) for _ in range(case["epochs"])]
        flat = mlp.init_params(case["members"], [seed % 1000 + m for m in range(case["members"])])
        steps = -(-case["rows"] // case["batch"])
        trace = torch.zeros((case["epochs"], steps, case["members"]), dtype=torch.float64, device=DEV)
        out = np.array(flat, dtype=np.float64)
        for m, w in enumerate(_members64(flat, case["members"])):
            for v in w.values():
                v.requires_grad_(True)
            opt = torch.optim.Adam(list(w.values()), lr=1e-3, betas=(0.9, 0.999), eps=1e-8)
            for e in range(case["epochs"]):
                for s in range(steps):
                    at = order[e][s * case["batch"]:(s + 1) * case["batch"]]
                    loss = ((_forward64(w, x[at]) - y[at]) ** 2).mean()
                    opt.zero_grad()
                    loss.backward()
                    opt.step()
                    trace[e, s, m] = loss.detach()
            views = mlp.unpack(out, case["members"])[m]
            for name, v in w.items():
                views[name][...] = v.detach().cpu().numpy()
        return trace, out
    return None  # a search's path, and a ranking by predicted times, turn on 32-bit comparisons
