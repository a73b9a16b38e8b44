"""What a user of the library has it do, as measurable cases.

Every case is one call (or the few calls that belong together) of the Python
binding, on systems drawn with the shapes of the repository's own workloads
(``paam_gen.CONFIGS``); the tables are made here with torch on the GPU, from
the seed alone.
"""
import math

import numpy as np
import torch

import paper_2404_06452_gb300 as paam
from paper_2404_06452_gb300 import _binding as B

# Shapes of the workloads: chains per system (uniform, or a geometric tail of
# probability g), callbacks per chain, executors, executors per core, total CPU
# utilisation, probability of an accelerator segment per callback, its WCET.
SHAPES = {
    "cfg1": dict(n=(4, 4), g=0.0, cb=(2, 4), x=(2, 2), per_core=2, u=(0.5, 0.5), p=0.3, a=(100_000, 2_000_000)),
    "cfg2": dict(n=(8, 16), g=0.0, cb=(3, 8), x=(4, 4), per_core=2, u=(0.3, 0.9), p=0.5, a=(100_000, 2_000_000)),
    "cfg3": dict(n=(2, 64), g=1.0 / 9.0, cb=(1, 12), x=(2, 8), per_core=2, u=(0.2, 0.95), p=0.5,
                 a=(100_000, 2_000_000)),
    "cfg4": dict(n=(16, 16), g=0.0, cb=(2, 4), x=(2, 2), per_core=2, u=(0.7, 0.7), p=0.3, a=(100_000, 2_000_000)),
    "cfg4s": dict(n=(16, 16), g=0.0, cb=(2, 4), x=(16, 16), per_core=1, u=(0.7, 0.7), p=0.3, a=(50_000, 1_000_000)),
}
PLAIN = dict(n_buckets=1, eps=0, kappa=0)                      # one bucket, no server overhead
LOADED = dict(n_buckets=2, eps=391_000, kappa=129_180)         # the paper's measured overheads, two buckets


def listed():
    return [
        # an admission test inside a control loop that may not allocate: tables already on the GPU
        dict(name="admit_noalloc_1k", call="noalloc", shape="cfg1", n_sys=1000, acc=1, safe=False, spin=0.0, **LOADED),
        # new systems (generated on the GPU by a design-space exploration): load, validate, analyse, free
        dict(name="load_analyze_200k", call="load", shape="cfg2", n_sys=200_000, acc=1, safe=False, spin=0.0, **PLAIN),
        # the batched analysis itself on a loaded batch, the headline workload
        dict(name="batch_1m", call="batch", shape="cfg2", n_sys=1_000_000, acc=1, safe=False, spin=0.0, **PLAIN),
        # the same for systems of very uneven size (2 to 64 chains)
        dict(name="batch_uneven_1m", call="batch", shape="cfg3", n_sys=1_000_000, acc=1, safe=False, spin=0.0, **PLAIN),
        # uneven systems with three accelerators each
        dict(name="batch_acc3_uneven_200k", call="batch", shape="cfg3", n_sys=200_000, acc=3, safe=False, spin=0.0,
             **PLAIN),
        # uneven systems under the safe reading of the blocking term, server overheads included
        dict(name="batch_safe_uneven_200k", call="batch", shape="cfg3", n_sys=200_000, acc=1, safe=True, spin=0.0,
             **LOADED),
        # systems that come from the host and whose results go back there
        dict(name="host_100k", call="host", shape="cfg2", n_sys=100_000, acc=1, safe=False, spin=0.0, **PLAIN),
        # priority search: every candidate order of every system
        dict(name="search_10k_x256", call="search", shape="cfg4s", n_sys=10_000, acc=1, safe=False, spin=0.0, K=256,
             early=False, **PLAIN),
        # priority search over uneven systems, stopping at the first admitted order
        dict(name="search_first_uneven_3k_x100", call="search", shape="cfg3", n_sys=3001, acc=1, safe=False, spin=0.0,
             K=100, early=True, **PLAIN),
        # a good first order for each system, lowest priority level first
        dict(name="seed_order_10k", call="audsley", shape="cfg4s", n_sys=10_000, acc=1, safe=False, spin=0.0, **PLAIN),
        # the network's ranking of candidate orders (inference), two pinned seeds
        dict(name="rank_10k_x256", call="rank", shape="cfg4s", n_sys=10_000, acc=1, safe=False, spin=0.0, K=256,
             top_k=16, n_pinned=2, **PLAIN),
        # one epoch of training on freshly analysed systems (forward, backward, update)
        dict(name="train_100k", call="train", shape="cfg2", n_sys=100_000, acc=1, safe=False, spin=0.0,
             batch_rows=8192, **PLAIN),
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    call = rng.choice(["noalloc", "load", "batch", "batch", "batch", "host", "search", "search", "audsley", "rank",
                       "train"])
    opts = dict(rng.choice([PLAIN, LOADED]))
    if rng.random() < 0.3:
        opts["n_buckets"] = rng.choice([1, 2, 3, 6])
    case = dict(call=call, acc=1, safe=False, spin=rng.choice([0.0, 0.0, 0.25]), **opts)
    if call in ("noalloc", "load", "host", "batch"):
        case["shape"] = rng.choice(["cfg1", "cfg2", "cfg3", "cfg4s"])
        kind = rng.choice(["plain", "plain", "acc", "safe"])
        if kind == "acc":
            case["acc"] = rng.choice([2, 3, 4])
        case["safe"] = kind == "safe"
        top = {"noalloc": 20_000, "load": 200_000, "host": 100_000,
               "batch": 1_000_000 if kind == "plain" else 200_000}[call]
        case["n_sys"] = _log(rng, 10, top)
    elif call == "search":
        case["shape"] = rng.choice(["cfg4s", "cfg4s", "cfg1", "cfg3"])  # shapes of which some systems are admitted
        case["early"] = rng.random() < 0.5
        case["K"] = rng.randint(2, 256)
        case["n_sys"] = _log(rng, 100, 3000 if case["shape"] == "cfg3" else 10_000)
        if case["shape"] == "cfg3":
            case["K"] = min(case["K"], 100)
    elif call == "audsley":
        case["shape"] = rng.choice(["cfg1", "cfg2", "cfg4", "cfg4s"])
        case["n_sys"] = _log(rng, 10, 10_000)
    elif call == "rank":
        case["shape"] = rng.choice(["cfg4s", "cfg2", "cfg3"])
        case["K"] = rng.randint(2, 256)
        case["n_sys"] = _log(rng, 10, 2000 if case["shape"] == "cfg3" else 10_000)
        if case["shape"] == "cfg3":
            case["K"] = min(case["K"], 64)
        case["top_k"] = rng.randint(1, min(case["K"], 64))
        case["n_pinned"] = rng.choice([0, 1, 2])
    else:
        case["shape"] = rng.choice(["cfg2", "cfg3", "cfg4s"])
        case["batch_rows"] = rng.choice([1024, 4096, 8192])
        case["n_sys"] = _log(rng, 1000, 12 * case["batch_rows"])
    return case


# ---- inputs ---------------------------------------------------------------
class Tables:
    """Device tables in the library's SoA / CSR layout (attribute per array)."""


def _off(counts):
    o = torch.zeros(counts.numel() + 1, dtype=torch.int64, device=counts.device)
    torch.cumsum(counts, 0, out=o[1:])
    return o


def _tables(case, seed):
    """Systems of the case's shape, drawn on the GPU from the seed.  Which chain counts occur is the same for
    every seed (their order is not), so results have one length."""
    sh, S, dev = SHAPES[case["shape"]], case["n_sys"], "cuda"
    g = torch.Generator(device=dev)

    def uni(n):
        return torch.rand(n, generator=g, device=dev, dtype=torch.float64)

    def ints(lo, hi, n):
        return torch.randint(lo, hi + 1, (n,), generator=g, device=dev, dtype=torch.int64)

    g.manual_seed(1)
    if sh["g"] > 0:
        n = sh["n"][0] + torch.floor(torch.log1p(-uni(S)) / math.log1p(-sh["g"])).to(torch.int64)
        n = n.clamp(sh["n"][0], sh["n"][1])
    else:
        n = ints(sh["n"][0], sh["n"][1], S)
    g.manual_seed(seed)
    n = n[torch.randperm(S, generator=g, device=dev)]
    nx = ints(sh["x"][0], sh["x"][1], S)
    t = Tables()
    t.sys_chain_off, t.sys_exec_off = _off(n), _off(nx)
    NC, NX = int(t.sys_chain_off[-1]), int(t.sys_exec_off[-1])
    sysid = torch.repeat_interleave(torch.arange(S, device=dev), n, output_size=NC)
    ncb = ints(sh["cb"][0], sh["cb"][1], NC)
    t.chain_cb_off = _off(ncb)
    NB = int(t.chain_cb_off[-1])
    has = (uni(NB) < sh["p"]).to(torch.int64)
    t.cb_seg_off = _off(has)
    NS = int(t.cb_seg_off[-1])
    # utilisation: a uniform split of the system's total over its chains (normalised exponentials)
    if case["shape"] == "cfg2":
        U = 0.3 + 0.1 * (torch.arange(S, device=dev) % 7).double()
    else:
        U = sh["u"][0] + (sh["u"][1] - sh["u"][0]) * uni(S)
    e = -torch.log1p(-uni(NC))
    tot = torch.zeros(S, dtype=torch.float64, device=dev).index_add_(0, sysid, e)
    t.T = torch.exp(math.log(1e7) + math.log(10.0) * uni(NC)).round().to(torch.int64)
    t.D = t.T.clone()
    per_cb = torch.floor(U[sysid] * e / tot[sysid] * t.T.double() / ncb.double()).to(torch.int64)
    chain_of_cb = torch.repeat_interleave(torch.arange(NC, device=dev), ncb, output_size=NB)
    t.E = per_cb[chain_of_cb]
    t.A = ints(sh["a"][0], sh["a"][1], NS)
    # distinct priorities: a random permutation of 0..n-1 per system
    order = torch.argsort(sysid.double() + uni(NC))
    local = torch.arange(NC, device=dev) - t.sys_chain_off[:-1][sysid]
    prio = torch.empty(NC, dtype=torch.int64, device=dev)
    prio[order] = local
    t.prio = prio.to(torch.int32)
    ex = torch.minimum((uni(NC) * nx[sysid]).to(torch.int64), nx[sysid] - 1)
    t.exec = ex.to(torch.int32)
    t.spin = (uni(NC) < case["spin"]).to(torch.uint8)
    # executors: per_core of them on each core, criticality-as-priority
    sys_of_x = torch.repeat_interleave(torch.arange(S, device=dev), nx, output_size=NX)
    lx = torch.arange(NX, device=dev) - t.sys_exec_off[:-1][sys_of_x]
    t.exec_core = (lx // sh["per_core"]).to(torch.int32)
    t.exec_prio = (-(lx + 1)).scatter_reduce(0, t.sys_exec_off[:-1][sysid] + ex, prio, "amax").to(torch.int32)
    # accelerators: worst fit over the units, approximated by dealing the segments of a
    # system to them back and forth by decreasing utilisation
    if case["acc"] > 1:
        sys_of_seg = sysid[chain_of_cb[has.bool()]]
        util = t.A.double() / t.T[chain_of_cb[has.bool()]].double()
        order = torch.argsort(sys_of_seg.double() + 0.999 * (1.0 - util / util.max().clamp(min=1e-300)))
        first = _off(torch.bincount(sys_of_seg, minlength=S))[:-1]
        k = (torch.arange(NS, device=dev) - first[sys_of_seg[order]]) % (2 * case["acc"])
        t.acc = torch.empty(NS, dtype=torch.int32, device=dev)
        t.acc[order] = torch.minimum(k, 2 * case["acc"] - 1 - k).to(torch.int32)
    else:
        t.acc = torch.zeros(NS, dtype=torch.int32, device=dev)
    return t, n


def _candidates(t, n, K, seed):
    """Rank rows [S, K, nmax]: slot 0 the system's own order, slot 1 deadline-monotonic, the others random."""
    S, nmax, dev = n.numel(), int(n.max()), "cuda"
    g = torch.Generator(device=dev)
    g.manual_seed(seed + 77)
    key = torch.rand((S, K, nmax), generator=g, device=dev)
    at = torch.arange(nmax, device=dev)
    real = at[None, :] < n[:, None]
    idx = (t.sys_chain_off[:-1, None] + at[None, :]).clamp(max=t.T.numel() - 1)
    key[:, 0] = 1.0 - t.prio[idx].float() / 64.0  # exact: priorities lie below 64
    key[:, 1] = torch.argsort(torch.argsort(torch.where(real, t.D[idx], 1 << 60), dim=1, stable=True), dim=1).float() / 64.0
    key.masked_fill_(~real[:, None, :], 2.0)
    by = torch.argsort(key, dim=2, stable=True)
    ranks = torch.empty((S, K, nmax), dtype=torch.int16, device=dev)
    ranks.scatter_(2, by, at.to(torch.int16).expand(S, K, nmax).contiguous())
    return ranks.masked_fill_(~real[:, None, :], -1)


def _weights(seed):
    """Parameters of a ranking network, in the library's order: uniform weights, zero biases."""
    g = torch.Generator()
    g.manual_seed(seed + 5)
    parts = []
    for fin, fout in SIZES:
        parts.append((torch.rand(fout * fin, generator=g) * 2 - 1) * math.sqrt(6.0 / fin))
        parts.append(torch.zeros(fout))
    return torch.cat(parts).numpy()


SIZES = [(1024, 256), (256, 256), (256, 256), (256, 64)]
LR, DECAY, BETA1, BETA2, ADAM_EPS = 2e-3, 1e-4, 0.9, 0.999, 1e-8
_ctx = []


def _context():
    if not _ctx:
        _ctx.append(paam.Context(0))
    return _ctx[0]


def _opts(case):
    return B.analysis_opts(case["n_buckets"], case["eps"], case["kappa"], 1 if case["safe"] else 0)


def prepare(case, seed):
    ctx, call = _context(), case["call"]
    t, n = _tables(case, seed)
    s = dict(case=case, ctx=ctx, opts=_opts(case))
    nc, ns = t.T.numel(), case["n_sys"]
    if call == "host":
        h = Tables()
        for f, a in vars(t).items():
            setattr(h, f, torch.empty(a.shape, dtype=a.dtype, pin_memory=True).copy_(a))
        s["tables"] = h
        s["out"] = [torch.empty(nc, dtype=torch.int64, pin_memory=True),
                    torch.empty(nc, dtype=torch.uint8, pin_memory=True),
                    torch.empty(ns, dtype=torch.uint8, pin_memory=True)]
        return s
    if call in ("noalloc", "load", "batch", "train"):
        s["out"] = [torch.empty(nc, dtype=torch.int64, device="cuda"),
                    torch.empty(nc, dtype=torch.uint8, device="cuda"),
                    torch.empty(ns, dtype=torch.uint8, device="cuda")]
    if call in ("noalloc", "load"):
        s["tables"] = t
        return s
    s["batch"] = B.paam_rta_load_systems(ctx, t)
    if call in ("search", "rank"):
        s["ranks"] = _candidates(t, n, case["K"], seed)
    if call == "search":
        s["first"] = torch.empty(ns, dtype=torch.int32, device="cuda")
        s["ok"] = None if case["early"] else torch.empty((ns, case["K"]), dtype=torch.uint8, device="cuda")
    if call == "audsley":
        s["seed_ranks"] = torch.empty((ns, int(n.max())), dtype=torch.int16, device="cuda")
    if call in ("rank", "train"):
        s["model"] = B.Model.create(ctx, 1)
        s["model"].set_params(_weights(seed))
    if call == "rank":
        s["ranked"] = torch.empty((ns, case["top_k"]), dtype=torch.int32, device="cuda")
        s["scores"] = torch.empty((ns, case["K"]), dtype=torch.float32, device="cuda")
    if call == "train":
        B.paam_rta_analyze_batch(ctx, s["batch"], s["opts"], *s["out"])
        s["loss"] = np.zeros(1, np.float32)
        s["train"] = B.train_opts(epochs=1, batch_rows=case["batch_rows"], lr=LR, weight_decay=DECAY, beta1=BETA1,
                                  beta2=BETA2, adam_eps=ADAM_EPS, seed=seed, n_buckets=case["n_buckets"],
                                  kappa=case["kappa"], epoch_loss=s["loss"])
    return s


def run(s):
    case, ctx, opts = s["case"], s["ctx"], s["opts"]
    call = case["call"]
    if call == "noalloc":
        B.paam_rta_analyze_noalloc(s["tables"], opts, *s["out"])
        return s["out"]
    if call == "load":
        batch = B.paam_rta_load_systems(ctx, s["tables"])
        B.paam_rta_analyze_batch(ctx, batch, opts, *s["out"])
        torch.cuda.current_stream().synchronize()  # a batch is freed only after the work that uses it
        batch.free()
        return s["out"]
    if call == "batch":
        B.paam_rta_analyze_batch(ctx, s["batch"], opts, *s["out"])
        return s["out"]
    if call == "host":
        B.paam_rta_analyze_host(ctx, s["tables"], opts, *s["out"])
        return s["out"]
    if call == "search":
        B.paam_rta_search_priorities(ctx, s["batch"], opts, s["ranks"], case["early"], s["ok"], s["first"])
        return [s["first"]] if s["ok"] is None else [s["first"], s["ok"]]
    if call == "audsley":
        B.paam_rta_audsley_order(ctx, s["batch"], opts, s["seed_ranks"])
        return s["seed_ranks"]
    if call == "rank":
        B.paam_surrogate_infer(ctx, s["model"], s["batch"], s["ranks"], case["top_k"], s["ranked"], s["scores"],
                               n_buckets=case["n_buckets"], kappa=case["kappa"], n_pinned=case["n_pinned"])
        return {"scores": s["scores"], "ranked": s["ranked"]}
    B.paam_surrogate_train(ctx, s["batch"], s["out"][0], s["out"][1], s["train"], s["model"])
    return {"params": s["model"].get_params(), "loss": s["loss"].copy()}


# ---- work -----------------------------------------------------------------
def work(case):
    """Each table read once and each result written once; the network's multiplications."""
    sh = SHAPES[case["shape"]]
    n = min(9.0 + 1.0, sh["n"][1]) if sh["g"] > 0 else sum(sh["n"]) / 2
    cb, x = sum(sh["cb"]) / 2, sum(sh["x"]) / 2
    nmax = sh["n"][1]
    tables = 16 + n * (8 + 16 + 4 + 4 + 1) + n * cb * (16 + sh["p"] * (8 + (4 if case["acc"] > 1 else 0))) + x * 8
    S, call = case["n_sys"], case["call"]
    if call in ("noalloc", "load", "batch", "host"):
        return {"bytes": S * (tables + n * 9 + 1), "flops": 0}
    if call == "search":
        return {"bytes": S * (tables + case["K"] * (2 * nmax + 1) + 4), "flops": 0}
    if call == "audsley":
        return {"bytes": S * (tables + 2 * nmax), "flops": 0}
    if call == "rank":
        kx = min(1024, (16 * nmax + 63) // 64 * 64)
        macs = kx * 256 + 2 * 256 * 256 + 256 * 64
        return {"bytes": S * (tables + case["K"] * (2 * nmax + 4) + 4 * case["top_k"]),
                "flops": 2.0 * macs * S * case["K"]}
    kx = 16 * n  # features that are not zero
    fwd = kx * 256 + 2 * 256 * 256 + 256 * 64
    return {"bytes": S * (tables + n * 9) + 3 * 4 * 410_000 * 2, "flops": 2.0 * S * (2 * fwd + 2 * 256 * 256 + 256 * 64)}


# ---- 64-bit values of the floating outputs -----------------------------------
def _chain_sums(t, kappa):
    """E, largest E, S*, M*, number of segments per chain, in float64."""
    NC, dev = t.T.numel(), "cuda"
    ncb = t.chain_cb_off[1:] - t.chain_cb_off[:-1]
    of_cb = torch.repeat_interleave(torch.arange(NC, device=dev), ncb)
    of_seg = torch.repeat_interleave(of_cb, t.cb_seg_off[1:] - t.cb_seg_off[:-1])

    def zero():
        return torch.zeros(NC, dtype=torch.float64, device=dev)

    a = t.A.double() + 2.0 * kappa
    return (zero().index_add_(0, of_cb, t.E.double()), zero().scatter_reduce_(0, of_cb, t.E.double(), "amax"),
            zero().index_add_(0, of_seg, a), zero().scatter_reduce_(0, of_seg, a, "amax"),
            zero().index_add_(0, of_seg, torch.ones_like(a)))


def _features(t, n, ranks, n_buckets, kappa, lo, hi):
    """The network's inputs of systems lo..hi-1 in float64: [systems, K, nmax, 16] (the header lists the ratios)."""
    dev, nmax = "cuda", int(n.max())
    if not hasattr(t, "sums"):
        t.sums = _chain_sums(t, kappa)
    at = torch.arange(nmax, device=dev)
    real = at[None, :] < n[lo:hi, None]
    idx = (t.sys_chain_off[lo:hi, None] + at[None, :]).clamp(max=t.T.numel() - 1)

    def pad(v, fill):
        return torch.where(real, v[idx].double(), fill)[:, None, :]  # [s, 1, nmax]

    T, D = pad(t.T, 1.0), pad(t.D, 1.0)
    E, Emax, S, M, dl = (pad(v, 0.0) for v in t.sums)
    ex = torch.where(real, t.exec[idx].long(), -1 - at[None, :])
    core = t.exec_core[(t.sys_exec_off[lo:hi, None] + ex.clamp(min=0)).clamp(max=t.exec_core.numel() - 1)].long()
    core = torch.where(real, core, -1 - at[None, :])
    num = n[lo:hi, None, None].double()
    if ranks is None:
        prio = torch.where(real, t.prio[idx].double(), -1.0)[:, None, :]
    else:
        prio = torch.where(real[:, None, :], num - 1.0 - ranks[lo:hi].double(), -1.0)
    both = (real[:, :, None] & real[:, None, :])[:, None]
    same_x = both & (ex[:, :, None] == ex[:, None, :])[:, None]
    same_k = both & (core[:, :, None] == core[:, None, :])[:, None] & ~same_x
    hi_ = both & (prio[:, :, None, :] > prio[:, :, :, None])  # [s, K, c, h]: h above c
    low = both & (prio[:, :, None, :] < prio[:, :, :, None])
    ep = torch.where(same_x, prio[:, :, None, :], -9.0).amax(3)
    user = dl > 0
    hps = hi_ & user[:, :, None, :]
    rank_u = hps.sum(3)
    n_user = user.sum(2, keepdim=True).clamp(min=1)
    bucket = torch.where(user, rank_u * n_buckets // n_user, -1)
    hp = hi_ & same_x
    hpp = same_k & (ep[:, :, None, :] > ep[:, :, :, None])
    blk_set = low & user[:, :, None, :] & (bucket[:, :, None, :] == bucket[:, :, :, None]) & user[:, :, :, None]

    def total(mask, v):
        return torch.einsum("skch,sjh->skc", mask.double(), v)

    def largest(mask, v):
        return torch.where(mask, v[:, :, None, :], 0.0).amax(3)

    Tmin = torch.where(real[:, None, :], T, 1e300).amin(2, keepdim=True)
    K = prio.shape[1]
    f = [E / T, S / T, D / T, torch.log2(T / Tmin) / 4, hi_.sum(3) / num, dl.clamp(max=16) / 16, Emax / D, M / D,
         total(hp, (E + S) / T), total(hpp, E / T), total(hps, S / T), largest(low & same_x, Emax) / D,
         largest(blk_set, M) / D, (E + S) / D, total(hp | hpp, E + S) / D, torch.ones_like(T)]
    f = torch.stack([v.expand(-1, K, -1) for v in f], 3).clamp(0.0, 8.0)
    return torch.where(real[:, None, :, None], f, 0.0)


def _layers(flat, width):
    out, o = [], 0
    for k, (fin, fout) in enumerate(SIZES):
        W = flat[o:o + fin * fout].view(fout, fin)
        o += fin * fout
        out.append([W[:, :width] if k == 0 else W, flat[o:o + fout]])
        o += fout
    return out


def _gelu(z):
    return 0.5 * z * (1 + torch.tanh(math.sqrt(2 / math.pi) * (z + 0.044715 * z ** 3)))


def _shuffled(n, total, seed):
    """The documented minibatch order of the first epoch of a new model: Fisher-Yates from the seed, padded with -1."""
    mask, x = (1 << 64) - 1, (seed ^ 0x5DEECE66D) & ((1 << 64) - 1)
    p = list(range(n))
    for i in range(n - 1, 0, -1):
        x = (x + 0x9E3779B97F4A7C15) & mask
        z = ((x ^ (x >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        z ^= z >> 31
        u = (z >> 11) * 2.0 ** -52 - 1.0
        j = int((u * 0.5 + 0.5) * float(i + 1)) % (i + 1)
        p[i], p[j] = p[j], p[i]
    return torch.tensor(p + [-1] * (total - n), device="cuda")


def exact(case, seed):
    """float64 values of the network's results; every other output is whole numbers, which have none."""
    call = case["call"]
    if call == "rank":
        t, n = _tables(case, seed)
        K, nmax = case["K"], int(n.max())
        ranks = _candidates(t, n, K, seed)
        W = _layers(torch.from_numpy(_weights(seed)).cuda().double(), 16 * nmax)
        scores = torch.empty((case["n_sys"], K), dtype=torch.float64, device="cuda")
        step = max(1, 40_000_000 // (K * nmax * nmax))
        for lo in range(0, case["n_sys"], step):
            hi = min(case["n_sys"], lo + step)
            h = _features(t, n, ranks, case["n_buckets"], case["kappa"], lo, hi).reshape((hi - lo) * K, -1)
            for k, (w, b) in enumerate(W):
                h = h @ w.T + b
                h = _gelu(h) if k < 3 else h
            own = torch.arange(64, device="cuda")[None, None, :] < n[lo:hi, None, None]
            scores[lo:hi] = torch.where(own, h.view(hi - lo, K, 64), 0.0).amax(2).clamp(min=0.0)
        return {"scores": scores, "ranked": None}
    if call == "train":
        t, n = _tables(case, seed)
        S, rows, nmax = case["n_sys"], case["batch_rows"], int(n.max())
        R, status, _ = prepare(case, seed)["out"]  # the labels are the training's inputs
        torch.cuda.synchronize()
        at = torch.arange(64, device="cuda")
        real = at[None, :] < n[:, None]
        idx = (t.sys_chain_off[:-1, None] + at[None, :]).clamp(max=t.T.numel() - 1)
        y = torch.where(status[idx] == 0, (R[idx].double() / t.D[idx].double()).clamp(max=2.0), 2.0)
        X = torch.empty((S, nmax * 16), dtype=torch.float64, device="cuda")
        step = max(1, 40_000_000 // (nmax * nmax))
        for lo in range(0, S, step):
            hi = min(S, lo + step)
            X[lo:hi] = _features(t, n, None, case["n_buckets"], case["kappa"], lo, hi).reshape(hi - lo, -1)
        flat = torch.from_numpy(_weights(seed)).cuda().double()
        m, v = torch.zeros_like(flat), torch.zeros_like(flat)
        decay = torch.zeros_like(flat)
        for k, (w, _) in enumerate(_layers(decay, 1024)):
            w.fill_(DECAY)
        steps = (S + rows - 1) // rows
        order = _shuffled(S, steps * rows, seed)
        loss = 0.0
        for k in range(steps):
            pick = order[k * rows:(k + 1) * rows]
            pick = pick[pick >= 0]
            p = flat.clone().requires_grad_()
            h = X[pick]
            for j, (w, b) in enumerate(_layers(p, nmax * 16)):
                h = h @ w.T + b
                h = _gelu(h) if j < 3 else h
            one = (torch.where(real[pick], h - y[pick], 0.0) ** 2).sum() / real[pick].sum().clamp(min=1)
            one.backward()
            loss += float(one)
            m = BETA1 * m + (1 - BETA1) * p.grad
            v = BETA2 * v + (1 - BETA2) * p.grad ** 2
            c1, c2 = 1 - BETA1 ** (k + 1), 1 - BETA2 ** (k + 1)
            flat = flat - LR * ((m / c1) / ((v / c2).sqrt() + ADAM_EPS) + decay * flat)
        return {"params": flat, "loss": torch.tensor([loss / steps], dtype=torch.float64)}
    return None
