"""The work that users of the library have it do, as cases that can be timed and compared.

Every case goes through the public binding (paper_2501_18054_gb300.pngf), on
the devices of paper_2501_18054_gb300.workloads: the 64 x 64-pixel dielectric
waveguide region ("guide", eps in {1, 10}), the 32 x 32-pixel lossy-metal
region ("metal") and the 10 x 10-pixel free-space region ("free").  A smaller
region is the centred w x h block of pixels of its device (a principal
sub-block of G: the same device with fewer pixels).  Each seed draws its own
start design, visiting order and pixels, as independent random starts on one
device do.

Kinds of case (the field "kind"):
  score     every flip scored with its ports, and the gradient: what an
            optimiser outside the library asks for between its own steps
  walk      from a saved state: a number of flips kept one call at a time, then
            every flip scored (an optimiser that takes its own decisions)
  factor    a start design factored and its state read back (every new start
            and every new design a user brings)
  search    from a factored state: one direct binary search, its trace, final
            design and state read back
  searches  several such searches side by side, each on its own stream with
            its share of the SMs
  batch     many runs of three region sizes in one batched call
  tiles     2 x 2 tile flips on one design shared by three frequencies
  pec       perfect-conductor pixels: the state built for a start design, then
            one search
"""
import functools
import types

import numpy as np
import torch

from paper_2501_18054_gb300 import pngf, workloads

DEVICES = {"guide": ("fdfd256", 64), "metal": ("fdfd128_metal", 32), "free": ("fdfd64", 10),
           "metal_l19": ("fdfd128_metal_l19", 32), "metal_l21": ("fdfd128_metal_l21", 32)}
# improvement threshold: the library's default where the decisions are clear of
# rounding; metal pixels that others shield change the objective at rounding
# level only, and metal searches set the threshold above that
TAU = {"guide": 1e-9, "free": 1e-9, "metal": 1e-6}
REFRESH, DELAY = 64, 64
BATCH_SIDES = (16, 24, 32)


def listed():
    return [
        # the smallest calls: a 100-pixel region scored (a few launches)
        {"name": "score_free_100", "kind": "score", "device": "free", "w": 10, "h": 10},
        # host-driven optimisation: 16 kept flips, one call each
        {"name": "walk_guide_2112", "kind": "walk", "device": "guide", "w": 48, "h": 44, "flips": 16},
        # a new start design on an odd-sized region, and on the largest region of the device
        {"name": "factor_guide_1517", "kind": "factor", "device": "guide", "w": 37, "h": 41, "precision": "fp64"},
        {"name": "factor_guide_4096", "kind": "factor", "device": "guide", "w": 64, "h": 64, "precision": "fp64"},
        # the three single-search configurations: 100 pixels in a shuffled order,
        # lossy metal at 1024, dielectric at 4096 (FP64 and mixed)
        {"name": "search_free_100", "kind": "search", "device": "free", "w": 10, "h": 10, "precision": "fp64",
         "mode": "first", "sweeps": 3, "shuffled": True},
        {"name": "search_metal_1024", "kind": "search", "device": "metal", "w": 32, "h": 32, "precision": "fp64",
         "mode": "first", "sweeps": 10, "shuffled": False},
        {"name": "search_guide_4096_fp64", "kind": "search", "device": "guide", "w": 64, "h": 64, "precision": "fp64",
         "mode": "first", "sweeps": 10, "shuffled": False},
        {"name": "search_guide_4096_mixed", "kind": "search", "device": "guide", "w": 64, "h": 64,
         "precision": "mixed", "mode": "first", "sweeps": 10, "shuffled": False},
        # the throughput configuration: eight mixed searches side by side
        {"name": "searches_8x4096_mixed", "kind": "searches", "device": "guide", "w": 64, "h": 64,
         "precision": "mixed", "runs": 8, "sweeps": 10},
        # many random starts of 256, 576 and 1024 metal pixels in one call
        {"name": "batch_96_metal", "kind": "batch", "runs": 96, "sweeps": 3},
        # tile flips with three frequency systems
        {"name": "tiles_3x1024_metal", "kind": "tiles", "w": 32, "h": 32, "systems": 3, "sweeps": 4},
        # the perfect-conductor system, state built from the design and searched
        {"name": "pec_1024", "kind": "pec", "device": "metal", "w": 32, "h": 32, "sweeps": 3},
    ]


def _side(rng, lo, hi):
    return int(round(np.exp(rng.uniform(np.log(lo), np.log(hi)))))


def draw(rng):
    kind = rng.choice(["score", "walk", "factor", "factor", "search", "search", "search", "searches", "batch",
                       "tiles", "pec"])
    if kind == "score":
        dev = rng.choice(["free", "metal", "guide"])
        top = DEVICES[dev][1]
        return {"kind": kind, "device": dev, "w": _side(rng, 4, top), "h": _side(rng, 4, top)}
    if kind == "walk":
        return {"kind": kind, "device": "guide", "w": _side(rng, 6, 64), "h": _side(rng, 6, 64),
                "flips": rng.randint(1, 16)}
    if kind == "factor":
        dev = rng.choice(["metal", "guide", "guide"])
        top = DEVICES[dev][1]
        return {"kind": kind, "device": dev, "w": _side(rng, 5, top), "h": _side(rng, 5, top),
                "precision": rng.choice(["fp64", "mixed"]) if dev == "guide" else "fp64"}
    if kind == "search":
        dev = rng.choice(["metal", "guide", "guide"])
        top = DEVICES[dev][1]
        return {"kind": kind, "device": dev, "w": _side(rng, 6, top), "h": _side(rng, 6, top),
                "precision": rng.choice(["fp64", "mixed"]) if dev == "guide" else "fp64",
                "mode": rng.choice(["first", "first", "best"]), "sweeps": rng.randint(2, 10),
                "shuffled": rng.random() < 0.5}
    if kind == "searches":
        return {"kind": kind, "device": "guide", "w": _side(rng, 16, 64), "h": _side(rng, 16, 64),
                "precision": rng.choice(["fp64", "mixed"]), "runs": rng.randint(2, 8), "sweeps": rng.randint(2, 6)}
    if kind == "batch":
        return {"kind": kind, "runs": rng.randint(8, 96), "sweeps": rng.randint(1, 3)}
    if kind == "tiles":
        return {"kind": kind, "w": 2 * rng.randint(3, 16), "h": 2 * rng.randint(3, 16), "systems": rng.randint(1, 3),
                "sweeps": rng.randint(1, 4)}
    return {"kind": kind, "device": "metal", "w": _side(rng, 6, 32), "h": _side(rng, 6, 32),
            "sweeps": rng.randint(1, 3)}


# ---------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=None)
def _device_arrays(dev):
    c = workloads.get_case(DEVICES[dev][0])
    t = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to("cuda", torch.complex128)  # noqa: E731
    return c, t(c.G_dd), t(c.G_od), t(c.c_d), t(c.c_o), t(c.dv)


def _region(dev, w, h):
    """The centred w x h block of a device: (what DbsContext reads from a Case, inputs on the GPU)."""
    side = DEVICES[dev][1]
    c, G, God, cd, co, dv = _device_arrays(dev)
    x0, y0 = (side - w) // 2, (side - h) // 2
    idx = (torch.arange(x0, x0 + w, device="cuda")[:, None] * side + torch.arange(y0, y0 + h, device="cuda")).reshape(-1)
    case = types.SimpleNamespace(n_d=w * h, n_o=c.n_o, obj_kind=c.obj_kind, obj_weights=c.obj_weights,
                                 s_off=c.s_off, s_scale=c.s_scale)
    if w == side and h == side:
        inputs = tuple(t.clone() for t in (G, God, cd, co, dv))
    else:
        inputs = (G[idx][:, idx].contiguous(), God[:, idx].contiguous(), cd[idx].clone(), co.clone(), dv[idx].clone())
    return case, inputs


def _start(n, seed):
    return torch.from_numpy(workloads.random_design(n, seed)).cuda()


def _context(region, precision="fp64", mode="first", tau=1e-9, n_ctas=0, stream=None):
    case, inputs = region
    prec = {"fp64": pngf.PNGF_FP64, "mixed": pngf.PNGF_MIXED, "pec": pngf.PNGF_PEC}[precision]
    return pngf.DbsContext(case, precision=prec, mode=pngf.PNGF_BEST_IMPROVEMENT if mode == "best" else
                           pngf.PNGF_FIRST_IMPROVEMENT, tau=tau, refresh_k=REFRESH, delay_r=DELAY, n_ctas=n_ctas,
                           stream=stream, inputs_on_device=inputs, tensor_fold=1 if precision == "mixed" else 0)


def _state_buffers(n, n_o, with_W=False, runs=None):
    lead = () if runs is None else (runs,)
    z = lambda *s: torch.zeros(lead + s, dtype=torch.complex128, device="cuda")  # noqa: E731
    out = {"diag": z(n), "e": z(n), "T": z(n_o, n), "o": z(n_o)}
    if with_W:
        out["W"] = z(n, n)
    return out


def _search_buffers(n, cap, runs=None):
    lead = () if runs is None else (runs,)
    return {"trace": torch.zeros(lead + (cap, 4), dtype=torch.int32, device="cuda"),
            "trace_f": torch.zeros(lead + (cap,), dtype=torch.float64, device="cuda"),
            "counters": torch.zeros(lead + (8,), dtype=torch.int64, device="cuda"),
            "design": torch.zeros(lead + (n,), dtype=torch.uint8, device="cuda")}


def _read_state(ctx, b, r=None):
    g = lambda k: (b[k] if r is None else b[k][r]).data_ptr() if k in b else None  # noqa: E731
    pngf.pngf_get_state(ctx.ctx, g("W"), g("diag"), g("e"), g("T"), g("o"))


def _tau(case):
    return TAU[case.get("device", "metal")]


def prepare(case, seed):
    torch.cuda.set_device(0)
    kind = case["kind"]
    if kind in ("score", "walk", "factor", "search", "searches", "pec"):
        region = _region(case["device"], case["w"], case["h"])
        n, n_o = region[0].n_d, region[0].n_o
    if kind in ("score", "walk"):
        ctx = _context(region)
        ctx.factor(_start(n, seed))
        s = {"ctx": ctx, "n": n, "all": torch.arange(n, dtype=torch.int32, device="cuda"),
             "f": torch.zeros(n, dtype=torch.float64, device="cuda"),
             "ports": torch.zeros((n, n_o), dtype=torch.complex128, device="cuda")}
        if kind == "score":
            s["grad"] = torch.zeros(n, dtype=torch.float64, device="cuda")
            s["dodrho"] = torch.zeros((n_o, n), dtype=torch.complex128, device="cuda")
        else:
            s["pixels"] = [int(k) for k in _walk_pixels(n, case["flips"], seed)]
            s["state"] = _state_buffers(n, n_o, with_W=True)
            s["design"] = torch.zeros(n, dtype=torch.uint8, device="cuda")
            ctx.snapshot()
    elif kind == "factor":
        fp64 = case["precision"] == "fp64"
        s = {"ctx": _context(region, case["precision"]), "b": _start(n, seed), "state": _state_buffers(n, n_o, with_W=fp64)}
    elif kind == "search":
        ctx = _context(region, case["precision"], case["mode"], _tau(case))
        ctx.factor(_start(n, seed))
        ctx.snapshot()
        order = None
        if case["shuffled"] and case["mode"] == "first":
            order = torch.from_numpy(workloads.shuffled_order(n, case["sweeps"], seed)).cuda()
        s = {"ctx": ctx, "order": order, "cap": _cap(case, n), **_search_buffers(n, _cap(case, n)),
             "state": _state_buffers(n, n_o)}
    elif kind == "searches":
        runs = case["runs"]
        n_sm = torch.cuda.get_device_properties(0).multi_processor_count
        cap = _cap(case, n)
        s = {"cap": cap, "runs": [], **_search_buffers(n, cap, runs), "state": _state_buffers(n, n_o, runs=runs)}
        here = torch.cuda.current_stream()
        for r in range(runs):
            st = torch.cuda.Stream()
            st.wait_stream(here)
            ctx = _context(region, case["precision"], n_ctas=n_sm // runs, stream=st)
            with torch.cuda.stream(st):
                ctx.factor(_start(n, seed * 64 + r))
                ctx.snapshot()
            here.wait_stream(st)
            s["runs"].append((ctx, st))
    elif kind == "batch":
        runs, cap = case["runs"], case["sweeps"] * BATCH_SIDES[-1] ** 2
        regions = [_region("metal", q, q) for q in BATCH_SIDES]
        ctxs = []
        for r in range(runs):
            ctx = _context(regions[r % 3], tau=TAU["metal"])
            ctx.factor(_start(ctx.n_d, seed * 1024 + r))
            ctx.snapshot()
            ctxs.append(ctx)
        n, n_o = BATCH_SIDES[-1] ** 2, 2
        s = {"ctxs": ctxs, "cap": cap, **_search_buffers(n, cap, runs), "state": _state_buffers(n, n_o, runs=runs)}
        s["trace_p"] = [s["trace"][r].data_ptr() for r in range(runs)]
        s["trace_f_p"] = [s["trace_f"][r].data_ptr() for r in range(runs)]
        s["ws"] = torch.empty(pngf.pngf_batch_workspace_size(runs), dtype=torch.uint8, device="cuda")
    elif kind == "tiles":
        names = ("metal", "metal_l19", "metal_l21")[:case["systems"]]
        ctxs = [_context(_region(d, case["w"], case["h"]), tau=TAU["metal"]) for d in names]
        n, n_o = ctxs[0].n_d, ctxs[0].n_o
        for ctx in ctxs:
            ctx.factor(_start(n, seed))
            ctx.snapshot()
        search = pngf.TileSearch(ctxs, workloads.square_tiles(case["w"], case["h"], 2))
        cap = case["sweeps"] * search.n_tiles
        s = {"search": search, "cap": cap, **_search_buffers(n, cap),
             "state": _state_buffers(n, n_o, runs=len(ctxs))}
    else:
        cap = case["sweeps"] * n
        s = {"ctx": _context(region, "pec", tau=TAU["metal"]), "b": _start(n, seed), "cap": cap,
             **_search_buffers(n, cap), "state": _state_buffers(n, n_o)}
    s["kind"], s["sweeps"] = kind, case.get("sweeps")
    return s


def _cap(case, n):
    return case["sweeps"] * n if case.get("mode", "first") == "first" else case["sweeps"] * 32


def _steps(case):
    """n_sweeps of the call: passes (FIRST) or kept flips at most (BEST)."""
    return case["sweeps"] if case.get("mode", "first") == "first" else case["sweeps"] * 32


def _walk_pixels(n, flips, seed):
    return np.random.Generator(np.random.PCG64([seed, 1])).permutation(n)[:min(flips, n)]


# ---------------------------------------------------------------- one pass
_FOUND = ("trace", "trace_f", "counters", "design")


def run(s):
    kind = s["kind"]
    if kind == "score":
        c = s["ctx"].ctx
        pngf.pngf_score_flips(c, s["all"].data_ptr(), s["n"], s["f"].data_ptr(), s["ports"].data_ptr())
        pngf.pngf_gradient(c, s["grad"].data_ptr(), s["dodrho"].data_ptr())
        return {k: s[k] for k in ("f", "ports", "grad", "dodrho")}
    if kind == "walk":
        c = s["ctx"].ctx
        pngf.pngf_restore(c)
        for k in s["pixels"]:
            pngf.pngf_accept_flip(c, k)
        pngf.pngf_score_flips(c, s["all"].data_ptr(), s["n"], s["f"].data_ptr(), s["ports"].data_ptr())
        _read_state(s["ctx"], s["state"])
        pngf.pngf_get_design(c, s["design"].data_ptr())
        return {**s["state"], **{k: s[k] for k in ("f", "ports", "design")}}
    if kind == "factor":
        pngf.pngf_factor(s["ctx"].ctx, s["b"].data_ptr())
        _read_state(s["ctx"], s["state"])
        return s["state"]
    if kind == "search":
        c = s["ctx"].ctx
        pngf.pngf_restore(c)
        steps = s["sweeps"] if s["ctx"].cfg.mode == pngf.PNGF_FIRST_IMPROVEMENT else s["sweeps"] * 32
        pngf.pngf_dbs_sweep(c, steps, None if s["order"] is None else s["order"].data_ptr(), s["trace"].data_ptr(),
                            s["trace_f"].data_ptr(), s["cap"], s["counters"].data_ptr())
        pngf.pngf_get_design(c, s["design"].data_ptr())
        _read_state(s["ctx"], s["state"])
        return {**s["state"], **{k: s[k] for k in _FOUND}}
    if kind == "searches":
        here = torch.cuda.current_stream()
        for r, (ctx, st) in enumerate(s["runs"]):
            st.wait_stream(here)
            pngf.pngf_restore(ctx.ctx)
            pngf.pngf_dbs_sweep(ctx.ctx, s["sweeps"], None, s["trace"][r].data_ptr(), s["trace_f"][r].data_ptr(),
                                s["cap"], s["counters"][r].data_ptr())
            pngf.pngf_get_design(ctx.ctx, s["design"][r].data_ptr())
            _read_state(ctx, s["state"], r)
        for _, st in s["runs"]:
            here.wait_stream(st)
        return {**s["state"], **{k: s[k] for k in _FOUND}}
    if kind == "batch":
        for ctx in s["ctxs"]:
            pngf.pngf_restore(ctx.ctx)
        pngf.pngf_dbs_sweep_batch([ctx.ctx for ctx in s["ctxs"]], s["sweeps"], None, s["trace_p"], s["trace_f_p"],
                                  s["cap"], s["counters"].data_ptr(), s["ws"].data_ptr(), s["ws"].numel())
        b = s["state"]
        for r, ctx in enumerate(s["ctxs"]):  # a region of n pixels fills the first n (T: n_o x n) entries of its row
            pngf.pngf_get_design(ctx.ctx, s["design"][r].data_ptr())
            _read_state(ctx, b, r)
        return {**b, **{k: s[k] for k in _FOUND}}
    if kind == "tiles":
        t = s["search"]
        for ctx in t.ctxs:
            pngf.pngf_restore(ctx.ctx)
        pngf.pngf_dbs_sweep_tiles([ctx.ctx for ctx in t.ctxs], t.combine, t.tiles.data_ptr(), t.n_tiles, t.tile_m,
                                  s["sweeps"], None, s["trace"].data_ptr(), s["trace_f"].data_ptr(), s["cap"],
                                  s["counters"].data_ptr(), t.ws.data_ptr(), t.ws_bytes)
        pngf.pngf_get_design(t.ctxs[0].ctx, s["design"].data_ptr())
        for r, ctx in enumerate(t.ctxs):
            _read_state(ctx, s["state"], r)
        return {**s["state"], **{k: s[k] for k in _FOUND}}
    c = s["ctx"].ctx
    pngf.pngf_factor(c, s["b"].data_ptr())
    pngf.pngf_dbs_sweep(c, s["sweeps"], None, s["trace"].data_ptr(), s["trace_f"].data_ptr(), s["cap"],
                        s["counters"].data_ptr())
    pngf.pngf_get_design(c, s["design"].data_ptr())
    _read_state(s["ctx"], s["state"])
    return {**s["state"], **{k: s[k] for k in _FOUND}}


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    """Inputs read once and outputs written once; the arithmetic of the method
    at one complex multiply-add (8 real operations) per term: an LU
    factorisation and n right-hand sides for the pixels that are on (half of
    them), a score per pixel, and per kept flip (taken as a fifth of the
    pixels of a search) one column of the maintained inverse and its rank-1
    correction on one triangle."""
    kind = case["kind"]
    c16, n_o = 16.0, 2
    if kind == "batch":
        ns = [BATCH_SIDES[r % 3] ** 2 for r in range(case["runs"])]
    elif kind == "tiles":
        ns = [case["w"] * case["h"]] * case["systems"]
    elif kind == "searches":
        ns = [case["w"] * case["h"]] * case["runs"]
    else:
        ns = [case["w"] * case["h"]]
    b = f = 0.0
    for n in ns:
        state = c16 * n * (2 + n_o)
        if kind == "score":
            b += state + c16 * n * (1 + 2 * n_o) + 16.0 * n
            f += 8.0 * n * (4 + 2 * n_o)
        elif kind == "walk":
            b += 2 * c16 * n * n + 2 * state
            f += case["flips"] * 8.0 * n * n / 2
        elif kind == "factor":
            m = n / 2
            b += 2 * c16 * n * n + state
            f += 8.0 * (m ** 3 / 3 + m * m * n + (n - m) ** 2 * m / 2)
        else:
            w_bytes = 4.0 if case.get("precision") == "mixed" else 8.0
            flips = n / 5 if case.get("mode", "first") == "first" else min(case["sweeps"] * 32, n / 5)
            b += 2 * 2 * w_bytes * n * n / 2 + 2 * state
            f += flips * 8.0 * n * n / 2
            if kind == "pec":
                f += 8.0 * ((n / 2) ** 3 / 3 + (n / 2) ** 2 * n)
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------- the same in plain 64-bit torch
def _problem(region):
    case, (G, God, cd, co, dv) = region
    t = lambda x, d: torch.as_tensor(np.asarray(x)).to("cuda", d)  # noqa: E731
    return types.SimpleNamespace(n=case.n_d, n_o=case.n_o, G=G, God=God, cd=cd, co=co, dv=dv,
                                 w=t(case.obj_weights, torch.float64), off=t(case.s_off, torch.complex128),
                                 scale=t(case.s_scale, torch.complex128))


def _objective(p, o):
    """sum_p w_p |S_p|^2 over the last dimension (every device here maximises it)."""
    s = (o - p.off) * p.scale
    return (p.w * (s.real ** 2 + s.imag ** 2)).sum(-1)


def _solved(p, b):
    """W, e, T, o of design b by one LU solve and one step of refinement."""
    v = p.dv * b
    eye = torch.eye(p.n, dtype=torch.complex128, device="cuda")
    M = eye - p.G * v[None, :]
    rhs = torch.cat([p.G, p.cd[:, None]], 1)
    lu, piv = torch.linalg.lu_factor(M)
    x = torch.linalg.lu_solve(lu, piv, rhs)
    x = x + torch.linalg.lu_solve(lu, piv, rhs - M @ x)
    W, e = x[:, :p.n], x[:, p.n]
    T = p.God + (p.God * v[None, :]) @ W
    return W, e, T, p.co + p.God @ (v * e)


def _flip_ports(p, b, diag, e, T, o):
    """Ports after each flip, (n, n_o)."""
    delta = torch.where(b.bool(), -p.dv, p.dv)
    alpha = delta / (1.0 - delta * diag)
    return o[None, :] + (alpha * e)[:, None] * T.T, alpha


def _exact_search(p, b, tau, sweeps, best, order):
    """Plain direct binary search with the rank-1 update of W in 64 bits; final state solved anew."""
    W, e, T, o = _solved(p, b)
    b, f, trace = b.clone(), float(_objective(p, o)), []
    pos_all = torch.arange(p.n, device="cuda")
    s = t = kept = 0
    while True:
        ports, alpha = _flip_ports(p, b, W.diagonal(), e, T, o)
        gain = _objective(p, ports) - f
        good = gain > tau * max(abs(f), 1e-30)
        if best:
            k = int(gain.argmax())
            pos = 0
            ok = bool(good[k])
        else:
            seq = order[s] if order is not None else pos_all
            hit = good[seq] & (pos_all >= t)
            pos = int(hit.to(torch.uint8).argmax())
            ok = bool(hit[pos])
            k = int(seq[pos])
        if not ok:
            if best or kept == 0:
                break
            s, t, kept = s + 1, 0, 0
            if s >= sweeps:
                break
            continue
        c = W[:, k].clone()
        a, ek, Tk = alpha[k].clone(), e[k].clone(), T[:, k].clone()
        W.addr_(a * c, c)
        e = e + a * ek * c
        T = T + (a * Tk)[:, None] * c[None, :]
        o = ports[k].clone()
        b[k] ^= 1
        f = float(_objective(p, o))
        trace.append(f)
        kept += 1
        t = pos + 1
        if best and len(trace) >= sweeps:
            break
        if not best and t >= p.n:
            s, t, kept = s + 1, 0, 0
            if s >= sweeps:
                break
    return b, trace


def _final(p, b):
    W, e, T, o = _solved(p, b)
    return {"diag": W.diagonal().clone(), "e": e, "T": T, "o": o}


def _padded(values, cap):
    out = torch.zeros(cap, dtype=torch.float64, device="cuda")
    k = min(cap, len(values))
    out[:k] = torch.tensor(values[:k], dtype=torch.float64)
    return out


def _exact_tiles(ps, b, tiles, tau, sweeps):
    """Tile search on the mean objective, rank-m updates of every system's W in 64 bits."""
    st = [list(_solved(p, b)) for p in ps]
    b, trace = b.clone(), []
    K = torch.from_numpy(tiles).long().cuda()
    nt, m = K.shape
    eye = torch.eye(m, dtype=torch.complex128, device="cuda")
    F = float(sum(_objective(p, x[3]) for p, x in zip(ps, st)) / len(ps))
    s = t = kept = 0
    idx = torch.arange(nt, device="cuda")
    while True:
        Fn, per = 0.0, []
        for p, (W, e, T, o) in zip(ps, st):
            D = torch.where(b[K].bool(), -p.dv[K], p.dv[K])
            A = eye[None] - D[:, :, None] * W[K[:, :, None], K[:, None, :]]
            y = torch.linalg.solve(A, D * e[K])
            on = o[None, :] + torch.einsum("ptm,tm->tp", T[:, K], y)
            per.append((A, D, y, on))
            Fn = Fn + _objective(p, on)
        good = (Fn / len(ps) - F > tau * max(abs(F), 1e-30)) & (idx >= t)
        k = int(good.to(torch.uint8).argmax())
        if not bool(good[k]):
            if kept == 0:
                break
            s, t, kept = s + 1, 0, 0
            if s >= sweeps:
                break
            continue
        for x, (A, D, y, on) in zip(st, per):
            U = x[0][:, K[k]].clone()
            Z = torch.linalg.solve(A[k], torch.diag(D[k]))
            TK = x[2][:, K[k]].clone()
            x[0] = x[0] + (U @ Z) @ U.T
            x[1] = x[1] + U @ y[k]
            x[2] = x[2] + (TK @ Z) @ U.T
            x[3] = on[k].clone()
        b[K[k]] ^= 1
        F = float(sum(_objective(p, x[3]) for p, x in zip(ps, st)) / len(ps))
        trace.append(F)
        kept, t = kept + 1, k + 1
        if t >= nt:
            s, t, kept = s + 1, 0, 0
            if s >= sweeps:
                break
    return b, trace


def _pec_state(p, b):
    """H, Q, diag W, e, j, T, R, o of metal set b, formed anew."""
    M = torch.nonzero(b).reshape(-1)
    z = lambda *s: torch.zeros(s, dtype=torch.complex128, device="cuda")  # noqa: E731
    dH, j, R = z(p.n), z(p.n), z(p.n_o, p.n)
    H = torch.linalg.inv(p.G[M][:, M])
    GM, GoM = p.G[:, M], p.God[:, M]
    dH[M] = H.diagonal()
    j[M] = -(H @ p.cd[M])
    R[:, M] = GoM @ H
    e = p.cd + GM @ j[M]
    e[M] = 0
    T = p.God - (GoM @ H) @ GM.T
    T[:, M] = 0
    dW = p.G.diagonal() - ((GM @ H) * GM).sum(1)
    dW[M] = 0
    return dH, dW, e, j, T, R, p.co + GoM @ j[M]


def _exact_pec(p, b, tau, sweeps):
    b, trace = b.clone(), []
    s = t = kept = 0
    idx = torch.arange(p.n, device="cuda")
    dH, dW, e, j, T, R, o = _pec_state(p, b)
    f = float(_objective(p, o))
    while True:
        on = b.bool()
        g = torch.where(on, j / torch.where(on, dH, torch.ones_like(dH)), e / torch.where(on, torch.ones_like(dW), dW))
        ports = o[None, :] - g[:, None] * torch.where(on[None, :], R, T).T
        good = (_objective(p, ports) - f > tau * max(abs(f), 1e-30)) & (idx >= t)
        k = int(good.to(torch.uint8).argmax())
        if not bool(good[k]):
            if kept == 0:
                break
            s, t, kept = s + 1, 0, 0
            if s >= sweeps:
                break
            continue
        b[k] ^= 1
        dH, dW, e, j, T, R, o = _pec_state(p, b)
        f = float(_objective(p, o))
        trace.append(f)
        kept, t = kept + 1, k + 1
        if t >= p.n:
            s, t, kept = s + 1, 0, 0
            if s >= sweeps:
                break
    return b, trace, {"diag": dW, "e": e, "T": T, "o": o}


def exact(case, seed):
    torch.cuda.set_device(0)
    kind = case["kind"]
    if kind == "batch":  # the first runs of each size: all would take too long
        n, cap, runs = BATCH_SIDES[-1] ** 2, case["sweeps"] * BATCH_SIDES[-1] ** 2, case["runs"]
        return None if runs > 12 else _exact_runs(
            [(_problem(_region("metal", BATCH_SIDES[r % 3], BATCH_SIDES[r % 3])), seed * 1024 + r) for r in range(runs)],
            TAU["metal"], case["sweeps"], n, cap)
    if kind == "tiles":
        names = ("metal", "metal_l19", "metal_l21")[:case["systems"]]
        ps = [_problem(_region(d, case["w"], case["h"])) for d in names]
        tiles = workloads.square_tiles(case["w"], case["h"], 2)
        b, trace = _exact_tiles(ps, _start(ps[0].n, seed), tiles, TAU["metal"], case["sweeps"])
        fin = [_final(p, b) for p in ps]
        return {**{k: torch.stack([x[k] for x in fin]) for k in fin[0]},
                "trace_f": _padded(trace, case["sweeps"] * len(tiles)), "trace": None, "counters": None, "design": None}
    p = _problem(_region(case["device"], case["w"], case["h"]))
    if kind == "pec":
        b, trace, fin = _exact_pec(p, _start(p.n, seed), TAU["metal"], case["sweeps"])
        return {**fin, "trace_f": _padded(trace, case["sweeps"] * p.n), "trace": None, "counters": None, "design": None}
    if kind == "searches":
        return _exact_runs([(p, seed * 64 + r) for r in range(case["runs"])], _tau(case), case["sweeps"], p.n,
                           _cap(case, p.n))
    b = _start(p.n, seed)
    if kind == "search":
        best = case["mode"] == "best"
        order = None
        if case["shuffled"] and not best:
            order = torch.from_numpy(workloads.shuffled_order(p.n, case["sweeps"], seed)).long().cuda()
        b, trace = _exact_search(p, b, _tau(case), _steps(case), best, order)
        return {**_final(p, b), "trace_f": _padded(trace, _cap(case, p.n)), "trace": None, "counters": None,
                "design": None}
    if kind == "walk":
        for k in _walk_pixels(p.n, case["flips"], seed):
            b[int(k)] ^= 1
    W, e, T, o = _solved(p, b)
    diag = W.diagonal().clone()
    if kind == "factor":
        return {"diag": diag, "e": e, "T": T, "o": o, **({"W": W} if case["precision"] == "fp64" else {})}
    ports, _ = _flip_ports(p, b, diag, e, T, o)
    if kind == "walk":  # W below the diagonal is not kept current
        return {"diag": diag, "e": e, "T": T, "o": o, "W": None, "f": _objective(p, ports), "ports": ports,
                "design": None}
    s = (o - p.off) * p.scale
    dodrho = T * (e * p.dv)[None, :]
    return {"f": _objective(p, ports), "ports": ports, "dodrho": dodrho,
            "grad": 2.0 * ((p.w * s.conj() * p.scale)[:, None] * dodrho).real.sum(0)}


def _exact_runs(runs, tau, sweeps, n, cap):
    out = {**_state_buffers(n, runs[0][0].n_o, runs=len(runs)),
           "trace_f": torch.zeros((len(runs), cap), dtype=torch.float64, device="cuda")}
    for r, (p, seed) in enumerate(runs):
        b, trace = _exact_search(p, _start(p.n, seed), tau, sweeps, False, None)
        for k, x in _final(p, b).items():
            out[k][r].reshape(-1)[:x.numel()] = x.reshape(-1)
        out["trace_f"][r] = _padded(trace, cap)
    return {**out, "trace": None, "counters": None, "design": None}
