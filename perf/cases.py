"""The work that programs using this package have it do, as sized cases.

Each kind of case is one use of the public entry points:
  whole    the initializer from a netlist in device memory to a scored
           placement: pl_build_graph (in place), pl_filter_init, pl_hpwl;
  gsp      the GSP start alone (a placer that brings its own refinement):
           pl_build_graph, pl_init_signal, pl_gift;
  refine   one round of Algorithm 1 at a given placement: pl_build_hints,
           pl_filter_apply;
  learned  the same round with the learned filter: pl_build_hints,
           pl_learned_apply;
  batch    many designs' initializers at once: pl_filter_init_batch;
  hpwl     the score of a placement, as a placement loop asks for it;
  density  the scheduled macro charge on a placer's bin grid, once per
           iteration of global placement;
  train    epochs of the learned filter's training on collected records.

Netlists follow the recipe of the package's synthetic netlists (cell sizes, net
degrees, macro share, boundary pins, index locality), drawn here with torch on
the device so that many of them can be made quickly; macros sit one in a slot of
a uniform grid.  `exact` states the same results in plain torch, FP64.
"""
import json
import math
import os
from types import SimpleNamespace

import numpy as np
import torch

import paper_2511_10073_gb300 as pl

DEV = "cuda"
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
GIFT_BANDS = ((4, 4.0, 0.7), (2, 4.0, 0.2), (2, 2.0, 0.1))  # (k, sigma, alpha), the defaults
GAMMA, T_HINT, CAPACITY, MU, DET_RATIO, CLIQUE = 0.5, 3, 1.0, 4.0, 0.1, 16
RHO_MODELS = ("gauss", "exp", "linear", "sigmoid")


def _design(cells, macros, io, nets, cap, shuffled=False):
    return dict(cells=cells, macros=macros, io=io, nets=nets, cap=cap, shuffled=shuffled)


SMALL = _design(2_000, 20, 64, 2_200, 64)
MEDIUM = _design(210_000, 550, 1_000, 220_000, 2_000)
HALF = _design(1_100_000, 4_000, 4_000, 1_125_000, 5_000)
LARGE = _design(2_200_000, 8_000, 8_000, 2_250_000, 10_000)


def listed():
    fp32 = dict(bins=32, wdtype="fp32", taps="8", pin=False)
    bf16 = dict(bins=32, wdtype="bf16", taps="2,4,8", pin=False)
    return [
        # a block of a few thousand cells, initialized interactively: launches and host reads count
        dict(name="whole_2k", kind="whole", **SMALL, **{**fp32, "bins": 16}),
        # a full chip, from netlist to score
        dict(name="whole_2200k", kind="whole", **LARGE, **bf16),
        # the GSP start of a mid-size design, filtered about the region's centre
        dict(name="gsp_210k", kind="gsp", **MEDIUM, **fp32, center=True),
        # one refinement round of the full chip, the step that Algorithm 1 repeats
        dict(name="refine_2200k", kind="refine", **LARGE, **bf16),
        # a mid-size round in FP32 weights, fixed nodes re-pinned after every power
        dict(name="refine_210k_fp32", kind="refine", **MEDIUM, **{**fp32, "pin": True}),
        # a small block on a fine bin grid (5 x 5 windows), cells in no particular order
        dict(name="refine_20k_64bins", kind="refine",
             **_design(20_011, 97, 101, 20_407, 2_000, True), **{**bf16, "bins": 64}),
        # a round of the learned filter on half a chip
        dict(name="learned_1100k", kind="learned", **HALF, **{**bf16, "pin": True}, model="k012"),
        # a serving batch of uneven designs, one worker stream each in turn
        dict(name="batch_32", kind="batch", designs=32, lo=5_000, hi=200_000, **bf16),
        # scoring the full chip
        dict(name="hpwl_2250k", kind="hpwl", **LARGE, offsets=True),
        # macro charge redistribution on a full chip's placement grid
        dict(name="density_gauss_512", kind="density", macros=8_000, bins=512, model="gauss", t=150),
        # macro charge restoration on a mid-size grid
        dict(name="density_sigmoid_256", kind="density", macros=550, bins=256, model="sigmoid", t=150),
        # training on one mid-size design's records
        dict(name="train_630k", kind="train", **MEDIUM, **{**bf16, "pin": True}, epochs=2),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["whole", "whole", "gsp", "refine", "refine", "learned", "batch", "hpwl",
                       "density", "train"])
    if kind == "density":
        return dict(kind=kind, macros=_log(rng, 20, 8_000), bins=_log(rng, 31, 512),
                    model=rng.choice(RHO_MODELS), t=rng.randrange(1, 300))
    opts = dict(bins=rng.choice([16, 24, 32, 32, 33, 48, 64]), wdtype=rng.choice(["fp32", "bf16"]),
                taps=rng.choice(["8", "4", "2,4,8", "1,3"]), pin=rng.random() < 0.4)
    if kind == "batch":
        lo = _log(rng, 2_000, 20_000)
        return dict(kind=kind, designs=rng.randrange(2, 33), lo=lo, hi=lo * rng.randrange(2, 11), **opts)
    cells = _log(rng, *{"hpwl": (2_000, 2_200_000), "train": (20_000, 210_000),
                        "learned": (20_000, 1_100_000)}.get(kind, (1_500, 2_000_000)))
    d = _design(cells, max(1, int(cells * rng.uniform(0.002, 0.01))), max(16, cells // 200),
                int(1.02 * cells), min(10_000, max(40, cells // 100)), rng.random() < 0.25)
    if kind == "hpwl":
        return dict(kind=kind, **d, offsets=rng.random() < 0.7)
    if kind == "train":
        return dict(kind=kind, **d, **{**opts, "pin": True}, epochs=rng.randrange(1, 4))
    if kind == "learned":
        return dict(kind=kind, **d, **{**opts, "pin": True}, model=rng.choice(["k012", "k024", "k036"]))
    if kind == "gsp":
        return dict(kind=kind, **d, **opts, center=rng.random() < 0.5)
    return dict(kind=kind, **d, **opts)


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)
    return g


def _uniform(g, n, lo=0.0, hi=1.0):
    return torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * (hi - lo) + lo


def _boundary(g, w, h):
    """A uniform point on the boundary of each w x h rectangle, from its lower-left corner."""
    t = _uniform(g, w.numel()) * 2 * (w + h)
    x = torch.where(t < w, t, torch.where(t < w + h, w, torch.where(t < 2 * w + h, t - w - h, 0 * t)))
    y = torch.where(t < w, 0 * t, torch.where(t < w + h, t - w, torch.where(t < 2 * w + h, h, t - 2 * w - h)))
    return x, y


def _macros(g, n, side):
    """n macros covering about 40% of a side x side die, one in a slot of a uniform grid."""
    ng = max(1, math.ceil(math.sqrt(n)))
    slot = side / ng
    rel = torch.exp(_uniform(g, n, 0.0, math.log(10.0)))
    area = rel / rel.sum() * 0.40 * side * side
    asp = _uniform(g, n, 0.7, 1.4)
    most = max(1.0, math.floor(0.94 * slot))
    w = torch.round(torch.sqrt(area * asp)).clamp(1.0, most)
    h = torch.round(torch.sqrt(area / asp)).clamp(1.0, most)
    at = torch.randperm(ng * ng, generator=g, device=DEV)[:n]
    x = (at % ng) * slot + _uniform(g, n) * (slot - w) + 0.5 * w
    y = (at // ng) * slot + _uniform(g, n) * (slot - h) + 0.5 * h
    return x, y, w, h, slot


def _netlist(case, seed):
    """A netlist of the case's sizes on the device, and its arrays on the host."""
    g = _gen(seed)
    n, nm, nio, nn, cap = (case[k] for k in ("cells", "macros", "io", "nets", "cap"))
    C = n + nm + nio
    sw = torch.randint(1, 5, (n,), generator=g, device=DEV).double()
    side = float(math.ceil(math.sqrt(float(sw.sum()) / 0.36)))
    mx, my, mw, mh, slot = _macros(g, nm, side)
    full = torch.full((nio,), side, device=DEV, dtype=torch.float64)
    iox, ioy = _boundary(g, full, full)
    one, zn, zi = torch.ones(n, device=DEV).double(), 0 * sw, 0 * full
    cell_w, cell_h = torch.cat([sw, mw, zi]), torch.cat([one, mh, zi])
    kind = torch.cat([zn, 0 * mw + 1, zi + 2]).to(torch.uint8)
    fx, fy = torch.cat([zn, mx, iox]), torch.cat([zn, my, ioy])
    # net degrees: 55% 2-pin, 20% 3-pin, 25% with P(d) ~ d^-2.5 on [4, cap]
    u = _uniform(g, nn)
    pmf = torch.arange(4, cap + 1, device=DEV, dtype=torch.float64) ** -2.5
    tail = 4 + torch.searchsorted(torch.cumsum(pmf, 0) / pmf.sum(), _uniform(g, nn))
    deg = torch.where(u < 0.55, 2, torch.where(u < 0.75, 3, tail)).clamp(max=cap)
    # locality: a seed cell, every other pin from a block of 32 * 2^l cells around it, P(l) ~ 2^-l
    root = torch.randint(0, n, (nn,), generator=g, device=DEV)
    net = torch.repeat_interleave(torch.arange(nn, device=DEV), deg - 1)
    depth = max(1, math.ceil(math.log2(max(2, n / 32)))) + 1
    lvl = torch.floor(-torch.log2(_uniform(g, net.numel()).clamp(min=1e-300))).clamp(max=depth).long()
    lo = (root[net] >> (5 + lvl)) << (5 + lvl)
    hi = (lo + (32 << lvl)).clamp(max=n)
    extra = torch.minimum(lo + (_uniform(g, net.numel()) * (hi - lo)).long(), hi - 1)
    pin_net, pin_cell = torch.cat([torch.arange(nn, device=DEV), net]), torch.cat([root, extra])
    pdx = _uniform(g, pin_cell.numel(), -0.4, 0.4) * sw[pin_cell]
    pdy = _uniform(g, pin_cell.numel(), -0.4, 0.4)
    # macro pins on the macros' boundaries and one pin per I/O, on random nets
    mcell = torch.repeat_interleave(torch.arange(nm, device=DEV),
                                    torch.round((mw + mh) / 4).clamp(8, 64).long())
    bx, by = _boundary(g, mw[mcell], mh[mcell])
    pin_net = torch.cat([pin_net, torch.randint(0, nn, (mcell.numel() + nio,), generator=g, device=DEV)])
    pin_cell = torch.cat([pin_cell, n + mcell, torch.arange(n + nm, C, device=DEV)])
    pdx = torch.cat([pdx, bx - 0.5 * mw[mcell], zi])
    pdy = torch.cat([pdy, by - 0.5 * mh[mcell], zi])
    order = torch.randperm(pin_net.numel(), generator=g, device=DEV)
    order = order[torch.argsort(pin_net[order], stable=True)]
    ptr = torch.zeros(nn + 1, device=DEV, dtype=torch.int64)
    ptr[1:] = torch.cumsum(torch.bincount(pin_net, minlength=nn), 0)
    pin_cell, pdx, pdy = pin_cell[order], pdx[order], pdy[order]
    if case.get("shuffled"):  # cells numbered in no particular order
        new = torch.randperm(C, generator=g, device=DEV)
        old = torch.argsort(new)
        pin_cell = new[pin_cell]
        cell_w, cell_h, kind, fx, fy = (a[old] for a in (cell_w, cell_h, kind, fx, fy))
    offs = case.get("offsets", True)
    dev = dict(net_ptr=ptr, pin_cell=pin_cell.int(), pin_dx=pdx.float() if offs else None,
               pin_dy=pdy.float() if offs else None, cell_w=cell_w.float(), cell_h=cell_h.float(),
               cell_kind=kind, fixed_x=fx.float(), fixed_y=fy.float())
    host = SimpleNamespace(region=(0.0, 0.0, side, side),
                           **{k: None if v is None else v.cpu().numpy() for k, v in dev.items()})
    return SimpleNamespace(C=C, M=nn, side=side, slot=slot, host=host, **dev)


def _placement(nl, seed):
    """Cell centres as the GSP start leaves them: most cells near the middle of the die (a
    standard deviation of a tenth of it, neighbours in a block of 32 somewhat together), a few
    anywhere; fixed cells at their places."""
    g = _gen(seed + 7919)
    C = nl.C
    block = torch.arange(C, device=DEV) // 32

    def axis():
        b = torch.randn(C // 32 + 1, generator=g, device=DEV, dtype=torch.float64)[block]
        p = 0.48 + 0.033 * b + 0.097 * torch.randn(C, generator=g, device=DEV, dtype=torch.float64)
        return torch.where(_uniform(g, C) < 0.02, _uniform(g, C), p).clamp(0.002, 0.998) * nl.side

    free = nl.cell_kind == 0
    return torch.stack([torch.where(free, axis().float(), nl.fixed_x),
                        torch.where(free, axis().float(), nl.fixed_y)], 1).contiguous()


def _taps(case):
    return [int(t) for t in case["taps"].split(",")]


def _params(case):
    k = _taps(case)
    n = len(k)
    return pl.params(nbx=case["bins"], nby=case["bins"],
                     wdtype=pl.PL_W_FP32 if case["wdtype"] == "fp32" else pl.PL_W_BF16, ntaps=n,
                     tap_k=tuple(k + [0] * (4 - n)), tap_alpha=tuple([1.0 / n] * n + [0.0] * (4 - n)),
                     pin_every_step=int(case["pin"]), gift_center=int(case.get("center", False)))


def _batch_sizes(case):
    n, lo, hi = case["designs"], case["lo"], case["hi"]
    cells = [int(round(lo * (hi / lo) ** ((i + 0.5) / n))) for i in range(n)]
    return [cells[(i * 5) % n] if n % 5 else cells[i] for i in range(n)]  # in no order of size


def _batch_designs(case):
    return [dict(**_design(c, max(1, c // 170), max(16, c // 200), int(1.02 * c), 2_000))
            for c in _batch_sizes(case)]


def _most_nodes(case):
    """Rows that hold any netlist's nodes: cells, macro pins, stars (a few percent of the nets),
    macro and bin nodes."""
    return (case["cells"] + case["macros"] + case["io"] + 64 * case["macros"] + case["nets"] // 8 + 64
            + case["macros"] + case["bins"] ** 2)


def _padded(case, x):
    return {"xy": torch.cat([x, x.new_zeros((_most_nodes(case) - x.shape[0], 2))])}


def _model(name):
    with open(os.path.join(ROOT, "paper_2511_10073_gb300", "weights", "learned_%s.json" % name)) as f:
        return json.load(f)


def _macro_case(case, seed):
    g = _gen(seed)
    side = math.ceil(math.sqrt(case["macros"] * 275 * 2.5 / 0.36))  # 275 cells a macro
    x, y, w, h, _ = _macros(g, case["macros"], float(side))
    return float(side), [t.float().contiguous() for t in (x, y, w, h)]


def prepare(case, seed):
    kind, s = case["kind"], SimpleNamespace(kind=case["kind"], seed=int(seed))
    if kind == "density":
        side, s.macros = _macro_case(case, seed)
        s.region, s.bins, s.t = (0.0, 0.0, side, side), case["bins"], case["t"]
        s.rp = pl.rho_params(model=RHO_MODELS.index(case["model"]))
        s.rho = torch.empty(s.bins * s.bins, dtype=torch.float64, device=DEV)
        return s
    if kind == "batch":
        s.prm = _params(case)
        nls = [_netlist(d, seed * 64 + i) for i, d in enumerate(_batch_designs(case))]
        s.graphs = [pl.pl_build_graph(pl.DeviceNetlist(nl.host), s.prm) for nl in nls]
        s.outs = [torch.empty(nl.C * 2, dtype=torch.float32, device=DEV) for nl in nls]
        s.seeds = [seed + i for i in range(len(nls))]
        s.streams = [torch.cuda.Stream() for _ in range(16)]
        s.opts = pl.batch_opts(union_products=0, streams=min(16, len(nls)))
        return s
    nl = _netlist(case, seed)
    s.dnl = pl.DeviceNetlist(nl.host)
    if kind in ("hpwl", "whole"):
        s.ws = pl.hpwl_workspace(nl.M)
        s.hpwl = torch.empty(1, dtype=torch.float64, device=DEV)
    if kind == "hpwl":
        s.xy = _placement(nl, seed)
        return s
    s.prm = _params(case)
    s.g = pl.pl_build_graph(s.dnl, s.prm)
    N = s.g.info()["N"]
    if kind == "whole":
        s.out = torch.empty((nl.C, 2), dtype=torch.float32, device=DEV)
        return s
    s.xy = torch.empty((N, 2), dtype=torch.float32, device=DEV)
    # the node coordinates head a buffer whose size depends on the case alone
    s.nodes = torch.zeros((_most_nodes(case), 2), dtype=torch.float32, device=DEV)
    s.out = s.nodes[:N]
    if kind == "gsp":
        return s
    pl.pl_init_signal(s.g, s.seed, _placement(nl, seed), s.xy)
    if kind == "learned":
        s.model = pl.LearnedModel.from_host(_model(case["model"]))
    if kind == "train":
        pl.pl_build_hints(s.g, s.prm, s.xy)
        n = pl.pl_learned_collect(s.g, s.prm, (0, 1, 2), 0, s.xy, None)
        s.rec = torch.empty((3 * n, pl.LEARNED_REC), dtype=torch.float32, device=DEV)
        s.nrec = 0
        for r in range(3):  # the trajectory's three rounds
            if r:
                pl.pl_build_hints(s.g, s.prm, s.xy)
            s.nrec += pl.pl_learned_collect(s.g, s.prm, (0, 1, 2), r, s.xy, s.rec[s.nrec:])
            pl.pl_filter_apply(s.g, s.prm, s.xy, s.out)
            s.xy, s.out = s.out, s.xy
        s.g.destroy()
        del s.g
        s.model = pl.learned_init((0, 1, 2), s.seed)
        s.w0 = s.model.w.clone()
        s.opts = pl.train_opts(epochs=case["epochs"], seed=s.seed)
        s.tws = pl.learned_train_workspace(s.nrec)
    return s


def run(s):
    if s.kind == "whole":
        pl.pl_build_graph(s.dnl, s.prm, graph=s.g)
        pl.pl_filter_init(s.g, s.prm, s.seed, None, s.out)
        pl.pl_hpwl(s.dnl, s.out, s.hpwl, s.ws)
        return {"xy": s.out, "hpwl": s.hpwl}
    if s.kind == "gsp":
        pl.pl_build_graph(s.dnl, s.prm, graph=s.g)
        pl.pl_init_signal(s.g, s.seed, None, s.xy)
        pl.pl_gift(s.g, s.prm, s.xy, s.out)
        return {"xy": s.nodes}
    if s.kind == "refine":
        pl.pl_build_hints(s.g, s.prm, s.xy)
        pl.pl_filter_apply(s.g, s.prm, s.xy, s.out)
        return {"xy": s.nodes}
    if s.kind == "learned":
        pl.pl_build_hints(s.g, s.prm, s.xy)
        pl.pl_learned_apply(s.g, s.prm, s.model, 0, s.xy, s.out)
        return {"xy": s.nodes}
    if s.kind == "batch":
        pl.pl_filter_init_batch(s.graphs, s.prm, s.seeds, s.outs, s.streams, s.opts)
        return s.outs
    if s.kind == "hpwl":
        pl.pl_hpwl(s.dnl, s.xy, s.hpwl, s.ws)
        return {"hpwl": s.hpwl}
    if s.kind == "density":
        pl.pl_macro_density(s.rp, s.t, *s.macros, s.region, s.bins, s.bins, s.rho)
        return {"rho": s.rho}
    s.model.w.copy_(s.w0)
    loss = pl.pl_learned_train(s.rec, s.nrec, s.model, s.opts, s.tws)
    return {"w": s.model.w, "loss": np.asarray(loss)}


# ------------------------------------------------------------------- work
def _expected(d):
    """About how many pins, static entries and nodes a netlist of these sizes has."""
    k = np.arange(4, d["cap"] + 1, dtype=np.float64)
    p = k ** -2.5 / np.sum(k ** -2.5)
    pins = d["nets"] * (0.55 * 2 + 0.2 * 3 + 0.25 * float(np.sum(p * k)))
    per = math.sqrt(0.40 * d["cells"] * 2.5 / 0.36 / d["macros"])  # a macro's side
    mpins = d["macros"] * min(64.0, max(8.0, per / 2))
    nnz = d["nets"] * (0.55 * 2 + 0.2 * 6 + 0.25 * float(np.sum(p * np.where(k <= CLIQUE, k * (k - 1), 2 * k))))
    stars = d["nets"] * 0.25 * float(np.sum(p[k > CLIQUE]))
    C = d["cells"] + d["macros"] + d["io"]
    return SimpleNamespace(pins=pins + mpins + d["io"], nnz=nnz + 4 * mpins, C=C, N=C + mpins + stars)


def _netlist_bytes(e, nets):
    return e.pins * 12 + nets * 8 + e.C * 17


def work(case):
    kind = case["kind"]
    if kind == "density":
        b = case["bins"]
        pairs = case["macros"] * (0.63 * b / math.sqrt(case["macros"]) + 1) ** 2  # macro-bin overlaps
        return {"bytes": case["macros"] * 16 + b * b * 8,
                "flops": pairs * {"gauss": 100, "exp": 64 * 40}.get(case["model"], 1024 * 12)}
    if kind == "batch":
        each = [work(dict(case, kind="whole", **d)) for d in _batch_designs(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    e = _expected(case)
    if kind == "hpwl":
        return {"bytes": e.pins * (12 if case["offsets"] else 4) + case["nets"] * 8 + e.C * 8 + 8,
                "flops": e.pins * 6}
    if kind == "train":
        rec = 3 * case["cells"]
        return {"bytes": rec * 96 + pl.LEARNED_SIZE * 8,
                "flops": case["epochs"] * rec * 6 * (16 * 64 + 64 * 4)}
    win = (2 * ((max(1, int(DET_RATIO * case["bins"])) - 1) // 2) + 1) ** 2
    power = {"learned": {"k012": 2, "k024": 4, "k036": 6}.get(case.get("model"), 0)}.get(kind, max(_taps(case)))
    product = 4 * (e.nnz + 2 * win * case["cells"]) * power
    gift = 4 * e.nnz * sum(max(k for k, s, _ in GIFT_BANDS if s == q) for q in {s for _, s, _ in GIFT_BANDS})
    if kind == "whole":
        return {"bytes": _netlist_bytes(e, case["nets"]) + e.C * 8 + 8, "flops": gift + T_HINT * product}
    if kind == "gsp":
        return {"bytes": _netlist_bytes(e, case["nets"]) + e.N * 8, "flops": gift}
    sw = 4 if case["wdtype"] == "fp32" else 2
    mlp = e.N * 2 * (16 * 64 + 64 * 4) if kind == "learned" else 0
    return {"bytes": e.nnz * (4 + sw) + e.N * 4 + e.C * 16 + e.N * 16, "flops": product + mlp}


# ------------------------------------------- the same results in plain FP64
def _store(w, wdtype):
    """FP64 weights rounded once to the storage type (nearest even), as FP64."""
    if wdtype == "fp32":
        return w.float().double()
    m, e = torch.frexp(w)
    return torch.ldexp(torch.round(m * 256) / 256, e)


def _static(nl, wdtype):
    """The static graph: merged clique and star edges, mean row weights, node tables."""
    C, M = nl.C, nl.M
    cell = nl.pin_cell.long()
    mac = nl.cell_kind[cell] == 1
    rank = torch.cumsum(mac.long(), 0) - 1
    Pm = int(mac.sum())
    node = torch.where(mac, C + rank, cell)
    top = C + Pm
    net = torch.repeat_interleave(torch.arange(M, device=DEV), nl.net_ptr[1:] - nl.net_ptr[:-1])
    key = torch.unique(net * top + node)
    unet, unode = key // top, key % top
    p = torch.bincount(unet, minlength=M)
    start = torch.cumsum(p, 0) - p
    rows, cols, lat = [], [], []
    for q in range(2, CLIQUE + 1):
        nets = torch.nonzero(p == q)[:, 0]
        nd = unode[start[nets][:, None] + torch.arange(q, device=DEV)]
        i, j = torch.nonzero(~torch.eye(q, dtype=torch.bool, device=DEV), as_tuple=True)
        rows.append(nd[:, i].reshape(-1))
        cols.append(nd[:, j].reshape(-1))
        lat.append(torch.full_like(rows[-1], 360360 // (q - 1)))
    big = torch.nonzero(p > CLIQUE)[:, 0]
    S = big.numel()
    Nst = top + S
    pair, inv = torch.unique(torch.cat(rows) * Nst + torch.cat(cols), return_inverse=True)
    w = torch.zeros(pair.numel(), device=DEV, dtype=torch.int64).index_add_(0, inv, torch.cat(lat)).double() / 360360
    star_of = torch.full((M,), -1, device=DEV, dtype=torch.int64)
    star_of[big] = top + torch.arange(S, device=DEV)
    on = star_of[unet] >= 0
    sn, sc = star_of[unet][on], unode[on]
    sw = (p[unet][on].double() / (p[unet][on] - 1).double())
    row = torch.cat([pair // Nst, sc, sn])
    col = torch.cat([pair % Nst, sn, sc])
    w = torch.cat([w, sw, sw])
    total = torch.zeros(Nst, device=DEV, dtype=torch.float64).index_add_(0, row, w)
    count = torch.bincount(row, minlength=Nst)
    base = torch.where(count > 0, total / count.clamp(min=1), 0 * total)[:C]
    xy = torch.zeros((Nst, 2), device=DEV, dtype=torch.float64)
    xy[:C, 0], xy[:C, 1] = nl.fixed_x.double(), nl.fixed_y.double()
    mc = cell[mac]
    for a, (f, o) in enumerate(((nl.fixed_x, nl.pin_dx), (nl.fixed_y, nl.pin_dy))):
        xy[C:top, a] = (f[mc].double() + (0 if o is None else o[mac].double())).float().double()
    kind = torch.full((Nst,), 2, device=DEV)
    kind[:C] = torch.where(nl.cell_kind == 0, 0, 2)
    kind[top:] = 1
    half = torch.zeros((Nst, 2), device=DEV, dtype=torch.float64)
    half[:C] = torch.where((nl.cell_kind == 0)[:, None], 0.5 * torch.stack([nl.cell_w, nl.cell_h], 1).double(), 0.0)
    return SimpleNamespace(row=row, col=col, w=_store(w, wdtype), base=base, Nst=Nst, top=top, S=S, kind=kind,
                           fixed=xy, half=half, star=(sn, sc), side=nl.side)


def _apply(row, col, w, x):
    return torch.zeros_like(x).index_add_(0, row, w[:, None] * x[col])


def _finish(x, kind, fixed, half, side):
    """Fixed nodes at their places, movable centres and star nodes inside the region."""
    lo = half[: x.shape[0]]
    x = torch.minimum(torch.maximum(x, lo), side - lo)
    return torch.where((kind == 2)[:, None], fixed, x)


def _splitmix(seed, n):
    c = np.arange(n, dtype=np.uint64)
    with np.errstate(over="ignore"):
        z = np.uint64(seed & 0xFFFFFFFFFFFFFFFF) + (c + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return (z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53


def _signal(nl, G, seed, xy0):
    """The initial node coordinates (static nodes)."""
    x = G.fixed.clone()
    if xy0 is None:
        xy0 = torch.from_numpy(_splitmix(seed, 2 * nl.C)).to(DEV).view(-1, 2) * nl.side
    free = (G.kind == 0)[: nl.C]
    x[: nl.C] = torch.where(free[:, None], xy0.double(), x[: nl.C])
    sn, sc = G.star
    sums = torch.zeros_like(x).index_add_(0, sn, x[sc])
    cnt = torch.bincount(sn, minlength=G.Nst).clamp(min=1)
    x[G.top:] = (sums / cnt[:, None])[G.top:]
    return x


def _gift(G, x, center):
    deg = torch.zeros(G.Nst, device=DEV, dtype=torch.float64).index_add_(0, G.row, G.w)
    c = 0.5 * G.side if center else 0.0
    out = torch.zeros_like(x)
    for k, sigma, alpha in GIFT_BANDS:
        r = torch.sqrt(deg + sigma)[:, None]
        u = x - c
        for _ in range(k):
            u = (sigma * u / r + _apply(G.row, G.col, G.w, u / r)) / r
        out += alpha * u
    return _finish(out + c, G.kind, G.fixed, G.half, G.side)


def _hints(nl, G, case, x):
    """The augmented graph at node coordinates x: all its edges, degrees, lambda_up, and
    tables over its N nodes (static, macro and bin nodes)."""
    nb, C, side = case["bins"], nl.C, nl.side
    f32 = dict(device=DEV, dtype=torch.float32)
    wb = side / nb
    hw = ((max(1, int(DET_RATIO * nb)) - 1) // 2)
    scale = torch.tensor(nb / side, **f32)
    free = nl.cell_kind == 0
    xf = x[:C].float()
    bxy = torch.floor(xf * scale).clamp(0, nb - 1).long()
    own = bxy[:, 1] * nb + bxy[:, 0]
    area = torch.where(free, nl.cell_w.double() * nl.cell_h.double(), 0.0)
    D = torch.zeros(nb * nb, device=DEV, dtype=torch.float64).index_add_(0, own, area) / (wb * wb)
    macs = torch.nonzero(nl.cell_kind == 1)[:, 0]
    mg = torch.stack([t[macs] for t in (nl.fixed_x, nl.fixed_y, nl.cell_w, nl.cell_h)], 1)
    m64 = mg.double()
    edge = torch.arange(nb + 1, device=DEV, dtype=torch.float64) * wb

    def cover(c, w):  # overlap length of each macro with each bin column
        return (torch.minimum(edge[1:], (c + 0.5 * w)[:, None]) - torch.maximum(edge[:-1], (c - 0.5 * w)[:, None])).clamp(min=0)

    amac = (cover(m64[:, 1], m64[:, 3]).T @ cover(m64[:, 0], m64[:, 2])).reshape(-1)
    cap = CAPACITY * (wb * wb - amac) / (wb * wb)
    phi = 2 / (1 + torch.exp(-MU * (D - cap))) - 1
    hint = free & (G.base > 0)
    cells = torch.nonzero(hint)[:, 0]
    mv0, bn0 = G.Nst, G.Nst + macs.numel()
    # macros over each cell: those of the cell's slot of the macro grid and the slots around it
    ng = round(side / nl.slot)
    at = (m64[:, 1] / nl.slot).long() * ng + (m64[:, 0] / nl.slot).long()
    slots = torch.full(((ng + 2) * (ng + 2),), -1, device=DEV, dtype=torch.int64)
    slots[(at // ng + 1) * (ng + 2) + at % ng + 1] = torch.arange(macs.numel(), device=DEV)
    kx, ky = ((xf[cells, a].double() / nl.slot).long().clamp(0, ng - 1) for a in (0, 1))
    near = torch.stack([slots[(ky + 1 + dy) * (ng + 2) + kx + 1 + dx] for dy in (-1, 0, 1) for dx in (-1, 0, 1)], 1)
    q = mg[near.clamp(min=0)]
    half = torch.tensor(0.5, **f32)
    hit = (near >= 0) & ((xf[cells, 0:1] - q[..., 0]).abs() < half * (nl.cell_w[cells][:, None] + q[..., 2])) \
        & ((xf[cells, 1:2] - q[..., 1]).abs() < half * (nl.cell_h[cells][:, None] + q[..., 3]))
    ci, cj = torch.nonzero(hit, as_tuple=True)
    i, m = cells[ci], near[ci, cj]
    r = torch.maximum((x[i, 0] - m64[m, 0]).abs() / (0.5 * m64[m, 2]), (x[i, 1] - m64[m, 1]).abs() / (0.5 * m64[m, 3]))
    rows, cols, ws = [i], [mv0 + m], [_store(-torch.exp(-r) * G.base[i], case["wdtype"])]
    for dy in range(-hw, hw + 1):
        for dx in range(-hw, hw + 1):
            bx, by = bxy[cells, 0] + dx, bxy[cells, 1] + dy
            ok = (bx >= 0) & (by >= 0) & (bx < nb) & (by < nb)
            i, bx, by = cells[ok], bx[ok], by[ok]
            r = torch.maximum((x[i, 0] - (bx.double() + 0.5) * wb).abs(), (x[i, 1] - (by.double() + 0.5) * wb).abs()) / (0.5 * wb)
            rows.append(i)
            cols.append(bn0 + by * nb + bx)
            ws.append(_store(-torch.exp(-r) * phi[by * nb + bx] * G.base[i], case["wdtype"]))
    i, v, w = torch.cat(rows), torch.cat(cols), torch.cat(ws)
    N = bn0 + nb * nb
    row, col, w = torch.cat([G.row, i, v]), torch.cat([G.col, v, i]), torch.cat([G.w, w, w])
    deg = torch.zeros(N, device=DEV, dtype=torch.float64).index_add_(0, row, w)
    pos = torch.zeros_like(deg).index_add_(0, row, w.clamp(min=0))
    c = ((torch.arange(nb, device=DEV).double() + 0.5) * wb).float().double()
    bins = torch.stack([c.repeat(nb), c.repeat_interleave(nb)], 1)
    fixed = torch.cat([G.fixed, m64[:, :2], bins])
    kind = torch.cat([G.kind, torch.full((N - G.Nst,), 2, device=DEV)])
    halfs = torch.cat([G.half, torch.zeros((N - G.Nst, 2), device=DEV, dtype=torch.float64)])
    return SimpleNamespace(row=row, col=col, w=w, deg=deg, pos=pos, lam=2 * pos.max(), N=N, fixed=fixed, kind=kind,
                           half=halfs, own=own, phi=phi, hint=hint, wb=wb)


def _powers(H, x, kmax, pin):
    for _ in range(kmax):
        x = ((H.lam - H.deg)[:, None] * x + _apply(H.row, H.col, H.w, x)) / H.lam
        if pin:
            x = torch.where((H.kind == 2)[:, None], H.fixed, x)
        yield x


def _relax(H, x, g, side):
    fix = (H.kind == 2)[:, None]
    return _finish((1 - GAMMA) * x + GAMMA * torch.where(fix, H.fixed, g), H.kind, H.fixed, H.half, side)


def _refine(nl, G, case, x):
    """One round of Algorithm 1 from static-node coordinates x; all N nodes."""
    H = _hints(nl, G, case, x)
    x = torch.cat([x, H.fixed[G.Nst:]])
    taps = _taps(case)
    g = torch.zeros_like(x)
    for k, y in enumerate(_powers(H, x, max(taps), case["pin"]), 1):
        if k in taps:
            g += y / len(taps)
    return _relax(H, x, g, nl.side)


def _bf16(a):
    return a.float().bfloat16().double()


def _learned(nl, G, case, x):
    H = _hints(nl, G, case, x)
    x = torch.cat([x, H.fixed[G.Nst:]])
    d = _model(case["model"])
    w = torch.tensor(d["w"], dtype=torch.float32, device=DEV).double()
    t = {0: x}
    for k, y in enumerate(_powers(H, x, max(d["k"]), case["pin"]), 1):
        if k in d["k"]:
            t[k] = y
    c = 0.5 * nl.side
    g0, g1, g2 = ((t[k] - c) / H.wb for k in d["k"])
    C, z = nl.C, torch.zeros(H.N, device=DEV, dtype=torch.float64)
    own_phi, is_hint, area = z.clone(), z.clone(), z.clone()
    own_phi[:C] = torch.where(H.hint, H.phi[H.own], 0.0)
    is_hint[:C] = H.hint.double()
    area[:C] = torch.where(nl.cell_kind == 0, nl.cell_w.double() * nl.cell_h.double() / (H.wb * H.wb), 0.0)
    f = torch.stack([(g1 - g0)[:, 0], (g1 - g0)[:, 1], (g2 - g0)[:, 0], (g2 - g0)[:, 1], H.deg / H.lam,
                     (2 * H.pos - H.deg) / H.lam, (H.deg - H.pos) / H.lam, own_phi, is_hint,
                     (H.kind == 1).double(), area, z, z, z, z, z], 1)
    f = _bf16((f - w[0:16]) * w[16:32])
    th, W1, b1 = w[32:35], _bf16(w[35:1059]).view(64, 16), w[1059:1123]
    W2, b2 = _bf16(w[1123:1379]).view(4, 64), w[1379:1383]
    o = _bf16(torch.relu(f @ W1.T + b1)) @ W2.T + b2
    p = th[0] * g0 + th[1] * g1 + th[2] * g2 + o[:, 0:1] * (g1 - g0) + o[:, 1:2] * (g2 - g0) + o[:, 2:4]
    return _relax(H, x, c + H.wb * p, nl.side)


def _hpwl(nl, xy):
    net = torch.repeat_interleave(torch.arange(nl.M, device=DEV), nl.net_ptr[1:] - nl.net_ptr[:-1])
    total = 0.0
    for a, o in ((0, nl.pin_dx), (1, nl.pin_dy)):
        q = xy[nl.pin_cell.long(), a].double() + (0 if o is None else o.double())
        big = torch.full((nl.M,), 1e300, device=DEV, dtype=torch.float64)
        lo, hi = big.scatter_reduce(0, net, q, "amin"), (-big).scatter_reduce(0, net, q, "amax")
        total = total + torch.where(hi >= lo, hi - lo, 0.0).sum()
    return total.view(1)


def _rho(case, seed):
    side, (mx, my, mw, mh) = _macro_case(case, seed)
    mx, my, mw, mh = (t.double() for t in (mx, my, mw, mh))
    n, T, t = case["bins"], 300, case["t"]
    wb, a, model = side / n, t / T, case["model"]
    k0 = [((c - 0.5 * w) / wb).floor().long().clamp(0, n - 1) for c, w in ((mx, mw), (my, mh))]
    k1 = [((c + 0.5 * w) / wb).floor().long().clamp(0, n - 1) for c, w in ((mx, mw), (my, mh))]
    nx, ny = k1[0] - k0[0] + 1, k1[1] - k0[1] + 1
    cnt = nx * ny
    m = torch.repeat_interleave(torch.arange(mx.numel(), device=DEV), cnt)
    j = torch.arange(m.numel(), device=DEV) - torch.repeat_interleave(torch.cumsum(cnt, 0) - cnt, cnt)
    bx, by = (k0[0][m] + j % nx[m]).double(), (k0[1][m] + j // nx[m]).double()
    ax, cx = torch.maximum(bx * wb - mx[m], -0.5 * mw[m]), torch.minimum((bx + 1) * wb - mx[m], 0.5 * mw[m])
    ay, cy = torch.maximum(by * wb - my[m], -0.5 * mh[m]), torch.minimum((by + 1) * wb - my[m], 0.5 * mh[m])
    ok = (ax < cx) & (ay < cy)
    m, b = m[ok], (by * n + bx)[ok].long()
    ax, cx, ay, cy, w, h = ax[ok], cx[ok], ay[ok], cy[ok], mw[m], mh[m]
    if model == "gauss":
        ea = math.sqrt(-2 * ((1 - a) * math.log(0.05) + a * math.log(0.9)))
        eb = math.sqrt(2 * math.log(2)) / (0.25 + 1.25 * a)
        z = min(1.0, max(0.0, (a - 0.3) / 0.4))
        s = 3 * z * z - 2 * z ** 3
        eta = eb ** (1 - s) * ea ** s
        c = math.sqrt(2) * eta
        A = 2 * eta * eta / (math.pi * math.erf(eta / math.sqrt(2)) ** 2)

        def part(lo, hi, w):
            return w * math.sqrt(math.pi) / (2 * c) * (torch.erf(c * hi / w) - torch.erf(c * lo / w))

        v = A * part(ax, cx, w) * part(ay, cy, h)
    else:
        gx, gw = (torch.tensor(q, device=DEV) for q in np.polynomial.legendre.leggauss(8))
        node = (0.25 * (torch.arange(4, device=DEV).double()[:, None] + 0.5) + 0.125 * gx).reshape(-1)  # on [0, 1]
        wt = (0.125 * gw).repeat(4)
        v = torch.empty_like(ax)
        for i in range(0, ax.numel(), 20_000):
            e = slice(i, i + 20_000)
            u = (ax[e, None] + (cx - ax)[e, None] * node) / w[e, None]
            y = (ay[e, None] + (cy - ay)[e, None] * node) / h[e, None]
            box = (cx - ax)[e] * (cy - ay)[e]
            if model == "exp":
                q = 1 / (2 * (-0.002 * T * math.log(1 - a)) ** 2)
                v[e] = box * (torch.exp(-torch.tan(math.pi * u) ** 2 * q) @ wt) * (torch.exp(-torch.tan(math.pi * y) ** 2 * q) @ wt)
                continue
            rr = torch.sqrt(2 * (u[:, :, None] ** 2 + y[:, None, :] ** 2)) * (0.5 / math.tan(0.5 * math.pi * a))
            f = (1 - rr).clamp(min=0) if model == "linear" else 2 / (1 + torch.exp(rr))
            v[e] = box * ((f @ wt) @ wt)
    return torch.zeros(n * n, device=DEV, dtype=torch.float64).index_add_(0, b, v)


def exact(case, seed):
    """run()'s outputs in FP64 (weights rounded to the storage type that the case asks for).
    None where a whole path is long enough for its bin decisions to differ between any two
    roundings (large designs, batches, training)."""
    kind = case["kind"]
    if kind == "density":
        return {"rho": _rho(case, seed)}
    if kind in ("batch", "train") or (kind == "whole" and case["cells"] > 20_000):
        return None
    nl = _netlist(case, seed)
    if kind == "hpwl":
        return {"hpwl": _hpwl(nl, _placement(nl, seed))}
    G = _static(nl, case["wdtype"])
    if kind in ("whole", "gsp"):
        x = _signal(nl, G, int(seed), None)
        x = _gift(G, x if kind == "whole" else x.float().double(), case.get("center", False))
        if kind == "gsp":
            nb, macs = case["bins"], nl.cell_kind == 1
            c = ((torch.arange(nb, device=DEV).double() + 0.5) * (nl.side / nb)).float().double()
            return _padded(case, torch.cat([x, torch.stack([nl.fixed_x[macs], nl.fixed_y[macs]], 1).double(),
                                            torch.stack([c.repeat(nb), c.repeat_interleave(nb)], 1)]))
        for _ in range(T_HINT):
            x = _refine(nl, G, case, x)[: G.Nst]
        return {"xy": x[: nl.C], "hpwl": _hpwl(nl, x[: nl.C])}
    x = _signal(nl, G, int(seed), _placement(nl, seed)).float().double()
    return _padded(case, (_refine if kind == "refine" else _learned)(nl, G, case, x))
