"""The calls that a user of the sampler makes, as measurable cases.

A case is a dict of plain values: the graph (kind, size, edge probabilities),
the call (samples, row shape, schedule, launch form, model) and what the user
does with the RR sets (nothing more, a host copy, greedy seeds).  Graphs are the
synthetic stand-ins of the package's workloads (seeded R-MAT and Erdos-Renyi
graphs, weighted cascade, uniform or trivalency probabilities), drawn on the
GPU from the seed alone.
"""
import math

import numpy as np
import torch

import paper_2311_10201_gb300 as fbpt


def listed():
    return [
        # The smallest call: one word of 64 samples on a 1,024-vertex graph,
        # rows copied to the host, 4 seeds.  Launches and host work only.
        dict(name="er_1k_word", do="sample", graph="er", n=1024, m=8192, prob="uniform", p=0.1, samples=64, words=1,
             slots=0, schedule="push", launch="persistent", refill="lane", model="ic", order="none", k=4, host=True,
             rr=5),
        # A first call as the binding's defaults have it (persistent launch,
        # widest rows) on a sparse graph of odd sizes just below criticality.
        dict(name="er_odd_default", do="sample", graph="er", n=200003, m=1599989, prob="uniform", p=0.1,
             samples=50001, words=0, slots=0, schedule="push", launch="persistent", refill="lane", model="ic",
             order="none", k=0, host=False, rr=5),
        # The defaults on a mid-size social-network graph, weighted cascade:
        # 262,144 RR sets and 50 seeds.
        dict(name="wc_s20_default", do="sample", graph="rmat", scale=20, ef=16, prob="wc", p=0.0, samples=262144,
             words=0, slots=0, schedule="push", launch="persistent", refill="lane", model="ic", order="none", k=50,
             host=False, rr=20),
        # The plain fused form (512 colours a batch, run to completion).
        dict(name="wc_s20_plain_w8", do="sample", graph="rmat", scale=20, ef=16, prob="wc", p=0.0, samples=16384,
             words=8, slots=1, schedule="push", launch="graph", refill="batch", model="ic", order="none", k=0,
             host=False, rr=20),
        # The headline workload: 1,048,576 RR sets on a scale-22 graph in degree
        # order with sorted starts, widest rows, 100 seeds.
        dict(name="wc_s22_headline", do="sample", graph="rmat", scale=22, ef=16, prob="wc", p=0.0, samples=1 << 20,
             words=8, slots=8, schedule="push", launch="graph", refill="lane", model="ic", order="degree", k=100,
             host=False, rr=22),
        # Uniform p above criticality: RR sets of tens of thousands of vertices,
        # dense colours, narrow rows; schedule by the policy network.
        dict(name="uni_s18_learned", do="sample", graph="rmat", scale=18, ef=20, prob="uniform", p=0.06, samples=16384,
             words=8, slots=1, schedule="learned", launch="graph", refill="lane", model="ic", order="none", k=0,
             host=False, rr=12000),
        # Trivalency probabilities on a large graph: most sets stay at their
        # start, one in ten reaches the giant component.
        dict(name="tri_s22_learned", do="sample", graph="rmat", scale=22, ef=16, prob="tri", p=0.0, samples=2048,
             words=8, slots=1, schedule="learned", launch="graph", refill="lane", model="ic", order="none", k=0,
             host=False, rr=57000),
        # The linear-threshold model: one walk per sample, tiny frontiers, many
        # levels.
        dict(name="lt_s20", do="sample", graph="rmat", scale=20, ef=16, prob="wc", p=0.0, samples=131072, words=8,
             slots=8, schedule="push", launch="graph", refill="lane", model="lt", order="none", k=50, host=False,
             rr=40),
        # Many graphs of uneven size in one launch.
        dict(name="batched_8", do="batched", graphs=8, scale_lo=12, scale_hi=16, samples_lo=4096, samples_hi=16384,
             words=4, slots=2, schedule="learned", rr=1500),
        # Influence maximization end to end (estimation rounds, final sample,
        # greedy), as the sampler's consumer runs it.
        dict(name="imm_s18", do="imm", scale=18, ef=16, k=50, epsilon=0.3, words=8, slots=8, launch="graph", rr=20),
        # Seed selection alone over RR sets that are kept, for a large budget.
        dict(name="select_s20_k200", do="select", scale=20, ef=16, samples=524288, k=200, noalloc=False, rr=20),
        # The schedule network trained on level traces (rows of six features).
        dict(name="train_64k_rows", do="train", rows=65536, steps=50),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sample"] * 6 + ["batched", "imm", "select", "select", "train"])
    if kind == "batched":
        lo = rng.randint(10, 14)
        slo = _log_int(rng, 500, 6000)
        return dict(do="batched", graphs=rng.randint(2, 10), scale_lo=lo, scale_hi=rng.randint(lo, 16), samples_lo=slo,
                    samples_hi=slo + rng.randint(1, 8000), words=rng.choice([1, 2, 4, 8]), slots=rng.choice([1, 2, 4]),
                    schedule=rng.choice(["push", "learned", "heuristic"]), rr=1500)
    if kind == "imm":
        return dict(do="imm", scale=rng.randint(13, 18), ef=rng.randint(8, 20), k=rng.randint(5, 60),
                    epsilon=round(rng.uniform(0.3, 0.6), 3), words=8, slots=rng.choice([2, 4, 8]),
                    launch=rng.choice(["graph", "persistent"]), rr=20)
    if kind == "select":
        noalloc = rng.random() < 0.4
        return dict(do="select", scale=rng.randint(13, 18 if noalloc else 20), ef=rng.randint(8, 20),
                    samples=_log_int(rng, 3000, 80000 if noalloc else 524288), k=rng.randint(1, 200), noalloc=noalloc,
                    rr=20)
    if kind == "train":
        return dict(do="train", rows=_log_int(rng, 1000, 65536), steps=rng.randint(10, 50))
    words = rng.choice([1, 2, 4, 8])
    slots = rng.choice([s for s in (1, 2, 3, 8, 16, 32) if s * words <= 64])
    base = dict(do="sample", words=words, slots=slots, launch=rng.choice(["graph", "persistent"]), refill="lane",
                model="ic", order="none", host=rng.random() < 0.3)
    prob = rng.choice(["wc", "wc", "uniform_low", "uniform_high", "tri", "lt"])
    if prob in ("wc", "lt"):
        base.update(graph="rmat", scale=rng.randint(12, 20), ef=rng.randint(8, 24), prob="wc", p=0.0, rr=20,
                    samples=_log_int(rng, 100, min(1000 * 64 * words * slots // 20, 262144)),
                    schedule=rng.choice(["push", "push", "filtered", "learned"]), k=rng.choice([0, 7, 50]))
        if prob == "lt":
            base.update(model="lt", schedule="push", rr=40)
        elif rng.random() < 0.4:
            base.update(order=rng.choice(["degree", "rcm", "random"]))
        elif rng.random() < 0.3:
            base.update(refill="batch", samples=min(base["samples"], 20 * 64 * words * slots))
    elif prob == "uniform_low":
        n = _log_int(rng, 300, 300000)
        base.update(graph="er", n=n, m=n * rng.randint(4, 9) - rng.randint(0, 7), prob="uniform",
                    p=round(rng.uniform(0.02, 0.1), 4), samples=_log_int(rng, 30, 50 * 64 * words * slots),
                    schedule=rng.choice(["push", "learned"]), k=rng.choice([0, 5]), rr=5)
    elif prob == "uniform_high":
        scale = rng.randint(11, 17)
        base.update(graph="rmat", scale=scale, ef=rng.randint(8, 24), prob="uniform", p=round(rng.uniform(0.04, 0.1), 4),
                    samples=_log_int(rng, 100, 4096), schedule=rng.choice(["push", "learned", "heuristic"]), k=0,
                    rr=1 << max(scale - 3, 0))
    else:
        scale = rng.randint(16, 21)
        base.update(graph="rmat", scale=scale, ef=16, prob="tri", p=0.0, samples=_log_int(rng, 50, 1500),
                    schedule=rng.choice(["push", "learned"]), k=0, rr=1 << max(scale - 6, 0))
    return base


# ---- inputs -------------------------------------------------------------------------------


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _csr(n, src, dst):
    """In-edge CSR of the distinct non-loop edges src -> dst: (row_ptr, col)."""
    keep = src != dst
    key = torch.unique(dst[keep] * n + src[keep])  # sorted by (dst, src)
    row = key // n
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.bincount(row, minlength=n).cumsum(0)
    return row_ptr, (key - row * n).to(torch.int32)


def _rmat(scale, ef, gen):
    """R-MAT (a, b, c, d = 0.57, 0.19, 0.19, 0.05) with shuffled vertex ids."""
    n, e = 1 << scale, ef << scale
    src = torch.zeros(e, dtype=torch.int64, device="cuda")
    dst = torch.zeros_like(src)
    for _ in range(scale):
        r = torch.rand(e, generator=gen, device="cuda")
        src = src * 2 + (r >= 0.76)
        dst = dst * 2 + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    perm = torch.randperm(n, generator=gen, device="cuda")
    return (n, *_csr(n, perm[src], perm[dst]))


def _er(n, m, gen):
    src = torch.randint(n, (m,), generator=gen, device="cuda")
    dst = torch.randint(n, (m,), generator=gen, device="cuda")
    return (n, *_csr(n, src, dst))


def _bits32(x):
    return torch.where(x >= 1 << 31, x - (1 << 32), x).to(torch.int32)


def _thresholds(prob, p, row_ptr, col, gen):
    m = col.numel()
    if prob == "uniform":
        return _bits32(torch.full((m,), int(p * 2.0**32), dtype=torch.int64, device="cuda"))
    if prob == "tri":
        ps = torch.tensor([int(q * 2.0**32) for q in (0.1, 0.01, 0.001)], device="cuda")
        return _bits32(ps[torch.randint(3, (m,), generator=gen, device="cuda")])
    deg = row_ptr.diff()
    t = torch.where(deg > 1, (1 << 32) // deg.clamp(min=1), 0xFFFFFFFF)
    return _bits32(torch.repeat_interleave(t, deg))


def _size(case):
    return case["n"] if case["graph"] == "er" else 1 << case["scale"]


def _room(case, n, samples):
    """Entries of the buffer that a program keeps for the RR sets' vertices."""
    if case.get("model") == "lt" or case["prob"] == "wc":
        return 150 * samples + (1 << 20)
    if case["prob"] == "tri":
        return samples * n // 16 + (1 << 20)
    if case["graph"] == "er":
        return 40 * samples + (1 << 17)
    return samples * n // 2 + (1 << 16)  # reachable vertices have in- and out-edges: less than half of an R-MAT's


def _buffer(case, n, samples):
    return torch.zeros(_room(case, n, samples), dtype=torch.int32, device="cuda")


def _graph(case, gen):
    if case["graph"] == "er":
        n, row_ptr, col = _er(case["n"], case["m"], gen)
    else:
        n, row_ptr, col = _rmat(case["scale"], case["ef"], gen)
    thr = _thresholds(case["prob"], case["p"], row_ptr, col, gen)
    g = fbpt.Graph(n, row_ptr, col, thr)
    if case.get("order", "none") != "none":
        perm = fbpt.order_compute(n, row_ptr.cpu().numpy(), col.cpu().numpy(), case["order"], seed=1)
        g.set_order(perm, sorted_starts=True)
    return g


def _wc_graph(scale, ef, gen):
    return _graph(dict(graph="rmat", scale=scale, ef=ef, prob="wc", p=0.0), gen)


def _train_rows(rows, gen):
    """Trace-like rows: log2 features of levels, the action taken, its log2 time."""
    r = lambda lo, hi: lo + (hi - lo) * torch.rand(rows, generator=gen, device="cuda", dtype=torch.float64)  # noqa: E731
    units = r(0, 18)
    groups = units + r(0, 6)
    colours = units + r(0, 4)
    X = torch.stack([units, groups, colours, torch.minimum(colours, r(4, 12)), groups - 22, colours - units], 1)
    A = torch.randint(8, (rows,), generator=gen, device="cuda")
    Y = 14 + 0.3 * torch.relu(groups - 8 - 0.4 * A) + 0.2 * colours + 0.1 * r(-1, 1)
    return X.to(torch.float32), A, Y.to(torch.float32)


def _train_init(X, gen):
    """He weights, zero biases, the input mean and scale of the rows."""
    rnd = lambda k: torch.randn(k, generator=gen, device="cuda")  # noqa: E731
    X = X.double()
    parts = [X.mean(0).float(), X.std(0).clamp(min=1e-3).float(), rnd(192) * math.sqrt(2 / 6), torch.zeros(32, device="cuda"),
             rnd(1024) * math.sqrt(2 / 32), torch.zeros(32, device="cuda"), rnd(256) * math.sqrt(2 / 32),
             torch.full((8,), 16.0, device="cuda")]
    return torch.cat(parts)


def prepare(case, seed):
    gen = _gen(seed)
    do = case["do"]
    if do == "sample":
        buf = _buffer(case, _size(case), case["samples"])
        return dict(do=do, case=case, seed=seed, g=_graph(case, gen), buf=buf.cpu().numpy() if case["host"] else buf)
    if do == "batched":
        G, gs, bufs, S = case["graphs"], [], [], []
        for i in range(G):  # sizes spread over the case's ranges, small and large graphs and samples mixed
            at, other = i / max(G - 1, 1), (i * 7 % G) / max(G - 1, 1)
            c = dict(graph="rmat", scale=round(case["scale_lo"] + at * (case["scale_hi"] - case["scale_lo"])),
                     ef=8 + i * 5 % 17, prob="uniform", p=0.01 + 0.09 * ((i * 3 + 1) % G) / G)
            S.append(round(case["samples_lo"] + other * (case["samples_hi"] - case["samples_lo"])))
            gs.append(_graph(c, gen))
            bufs.append(_buffer(c, 1 << c["scale"], S[-1]))
        return dict(do=do, case=case, seeds=[seed + i for i in range(G)], S=S, gs=gs, bufs=bufs)
    if do == "imm":
        return dict(do=do, case=case, seed=seed, g=_wc_graph(case["scale"], case["ef"], gen))
    if do == "select":
        g = _wc_graph(case["scale"], case["ef"], gen)
        return dict(do=do, case=case, rr=fbpt.sample(g, seed, 0, case["samples"], launch="graph"))
    X, A, Y = _train_rows(case["rows"], gen)
    init = _train_init(X, gen)
    return dict(do=do, case=case, X=X.cpu().numpy(), A=A.to(torch.int32).cpu().numpy().view(np.uint32),
                Y=Y.cpu().numpy(), init=init.cpu().numpy())


# ---- one pass -----------------------------------------------------------------------------


class _Device:
    """A device array of an RRSets as torch sees it (keeps the RRSets alive)."""

    def __init__(self, rr, ptr, count, typestr):
        self.rr = rr
        self.__cuda_array_interface__ = dict(shape=(count,), typestr=typestr, data=(ptr, False), version=3)


def _rr_out(rr, buf):
    """The RR sets' index where it is (device tensors over the library's
    arrays), their vertices in the program's buffer, zeros behind them."""
    c = rr.c
    view = lambda p, n, t: torch.as_tensor(_Device(rr, p, n, t), device="cuda")  # noqa: E731
    buf[:rr.total].copy_(view(c.verts, rr.total, "<i4"))
    return dict(offsets=view(c.offsets, rr.S + 1, "<i8"), verts=buf, starts=view(c.starts, rr.S, "<i4"),
                vcount=view(c.vcount, int(c.n), "<i4"))


def run(state):
    case, do = state["case"], state["do"]
    if do == "sample":
        rr = fbpt.sample(state["g"], state["seed"], 0, case["samples"], words=case["words"], slots=case["slots"],
                         schedule=case["schedule"], launch=case["launch"], refill=case["refill"], model=case["model"])
        if case["host"]:
            off, verts, starts, vcount = rr.to_host()
            state["buf"][:verts.size] = verts.view(np.int32)
            out = dict(offsets=off.view(np.int64), verts=state["buf"], starts=starts.view(np.int32),
                       vcount=vcount.view(np.int32))
        else:
            out = _rr_out(rr, state["buf"])
        if case["k"]:
            seeds, gains = fbpt.select_seeds(rr, case["k"])
            out.update(seeds=seeds.view(np.int32), gains=gains.view(np.int64))
        return out
    if do == "batched":
        rrs, _ = fbpt.sample_batched(state["gs"], state["seeds"], [0] * len(state["gs"]), state["S"],
                                     words=case["words"], slots=case["slots"], schedule=case["schedule"])
        return [_rr_out(rr, buf) for rr, buf in zip(rrs, state["bufs"])]
    if do == "imm":
        seeds, gains, res, _ = fbpt.imm(state["g"], case["k"], case["epsilon"], 1.0, state["seed"], words=case["words"],
                                        slots=case["slots"], launch=case["launch"])
        return dict(seeds=seeds.view(np.int32), gains=gains.view(np.int64), samples=int(res["samples"]),
                    theta=int(res["theta"]), rounds=int(res["rounds"]))
    if do == "select":
        pick = fbpt.select_seeds_noalloc if case["noalloc"] else fbpt.select_seeds
        seeds, gains = pick(state["rr"], case["k"])
        return dict(seeds=seeds.view(np.int32), gains=gains.view(np.int64))
    # a training run: the trained parameters, and the loss and gradient there
    pol, loss = fbpt.policy_train(state["X"], state["A"], state["Y"], steps=case["steps"], lr=3e-3, init=state["init"])
    params = pol.params()
    loss2, grad = fbpt.policy_loss_grad(state["init"], state["X"], state["A"], state["Y"])
    return dict(params=params, loss=loss, start_loss=loss2, start_grad=grad)


# ---- what a pass cannot do without ------------------------------------------------------------


def _sample_bytes(n, m, samples, rr):
    """In-edges and thresholds read, RR sets with their index and counts written."""
    return 8.0 * (n + 1) + 8.0 * m + 4.0 * samples * rr + 12.0 * samples + 4.0 * n


def _select_bytes(n, samples, rr):
    """RR sets, index and counts read."""
    return 4.0 * samples * rr + 8.0 * samples + 4.0 * n


def work(case):
    do = case["do"]
    if do == "train":
        # forward 6-32-32-1 and twice that backward, a multiply and an add each
        return {"bytes": 32.0 * case["rows"], "flops": 6.0 * (6 * 32 + 32 * 32 + 32) * case["rows"] * (case["steps"] + 2)}
    if do == "batched":
        n = 2.0 ** ((case["scale_lo"] + case["scale_hi"]) / 2)
        S = (case["samples_lo"] + case["samples_hi"]) / 2
        return {"bytes": case["graphs"] * _sample_bytes(n, 16 * n, S, case["rr"]), "flops": 0.0}
    if do == "imm":
        n = 2.0 ** case["scale"]
        return {"bytes": _sample_bytes(n, case["ef"] * n, 0.02 * n / case["epsilon"], case["rr"]), "flops": 0.0}
    if do == "select":
        return {"bytes": _select_bytes(2.0 ** case["scale"], case["samples"], case["rr"]), "flops": 0.0}
    n = float(case["n"]) if case["graph"] == "er" else 2.0 ** case["scale"]
    m = float(case["m"]) if case["graph"] == "er" else case["ef"] * n
    b = _sample_bytes(n, m, case["samples"], case["rr"])
    if case["k"]:
        b += _select_bytes(n, case["samples"], case["rr"])
    return {"bytes": b, "flops": 0.0}


# ---- 64-bit results ----------------------------------------------------------------------------


_SHAPES = ((12, (32, 6)), (204, (32,)), (236, (32, 32)), (1260, (32,)), (1292, (8, 32)), (1548, (8,)))


def _loss(P, Xn, A, Y):
    W1, b1, W2, b2, W3, b3 = (P[o:o + math.prod(s)].reshape(s) for o, s in _SHAPES)
    h1 = torch.relu(Xn @ W1.T + b1)
    h2 = torch.relu(h1 @ W2.T + b2)
    out = (h2 @ W3.T + b3).gather(1, A[:, None])[:, 0]
    return (out - Y).square().mean()


def exact(case, seed):
    """Training in 64 bits (the parameters after the run, its loss, the first
    gradient); the sampler's outputs are whole numbers."""
    if case["do"] != "train":
        return None
    gen = _gen(seed)
    X, A, Y = _train_rows(case["rows"], gen)
    P0 = _train_init(X, gen).double()
    Xn, Y = (X.double() - P0[:6]) / P0[6:12], Y.double()
    lr, first = float(np.float32(3e-3)), None
    P, m, v = P0.clone(), torch.zeros_like(P0), torch.zeros_like(P0)
    for t in range(1, case["steps"] + 1):
        Q = P.clone().requires_grad_(True)
        loss = _loss(Q, Xn, A, Y)
        (g,) = torch.autograd.grad(loss, Q)
        if first is None:
            first = (float(loss.detach()), g)
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        P = P - lr * (m / (1 - 0.9**t)) / ((v / (1 - 0.999**t)).sqrt() + 1e-8)
        P[:12] = P0[:12]
    return dict(params=P, loss=float(_loss(P, Xn, A, Y)), start_loss=first[0], start_grad=first[1])
