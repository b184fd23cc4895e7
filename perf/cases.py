"""The work that users of this framework have it do, as timed cases: one call sequence
each, through the public entry points (``dp``, ``torch_api``), with the inputs such a
program holds.

Kinds of cases:

* ``gradient``: model power and its gradients of one netlist, one activity (Algorithm 2, Eq. 7)
* ``step``: the whole hot path in one call - forward, simulation, beta, adjoint (Sec. III-B..E)
* ``simulate``: forward, bit-parallel simulation and every per-net result (Sec. III-C/D)
* ``autograd``: many activities at once through the autograd Function; ``tr_mode`` 2 is lag-one
* ``virus``: the gradient-ascent power-virus search with its P_virus (Algorithm 4, Eq. 3)
* ``sizing``: a sizing delta, the new adjoint and the best cells to resize (Eq. 8)
* ``serve``: a burst of mixed requests to several resident designs

Netlists come from the repository's generator, by the sizes in the case and a generator
seed that belongs to the case (a user's netlist stays while its activities change); the
activities, sizing deltas and requests come from ``prepare``'s seed.
"""
from __future__ import annotations

import functools
import math
import re

import numpy as np
import torch

from paper_2608_03778_gb300 import dp, netgen
from paper_2608_03778_gb300 import torch_api as ta

DEV = "cuda"


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest call: an engineering change on a block of 2,000 cells, re-analysed
        {"name": "gradient 2k", "kind": "gradient", "cells": 2000, "start": 96, "depth": 24, "tr_mode": 0},
        # a mid-size block: forward, power and all input and pin-cap gradients
        {"name": "gradient 120k", "kind": "gradient", "cells": 120000, "start": 9216, "depth": 48, "tr_mode": 0},
        # a full design of the size and depth of the paper's largest one, TR = 2PQ at every net
        {"name": "gradient 652k", "kind": "gradient", "cells": 652000, "start": 48052, "depth": 104, "tr_mode": 1},
        # the whole hot path on the paper's smallest shape, from and to host memory, a vector count
        # that is no multiple of 256
        {"name": "step 13k host", "kind": "step", "cells": 13000, "start": 958, "depth": 70, "tr_mode": 0,
         "grad_mode": 2, "words": 250, "host": True},
        # the headline workload: the whole hot path on two million cells, 4,096 vectors
        {"name": "step 2M", "kind": "step", "cells": 2000000, "start": 147456, "depth": 80, "tr_mode": 0,
         "grad_mode": 1, "words": 64, "host": False},
        # activity annotation: 16,384 vectors of a mid-size design, every per-net result read back
        {"name": "simulate 117k", "kind": "simulate", "cells": 117000, "start": 8623, "depth": 84, "tr_mode": 0,
         "words": 256},
        # the batched workload: 512 activities of the mid-size design, input gradients of the power sum
        {"name": "autograd 120k x 512", "kind": "autograd", "cells": 120000, "start": 9216, "depth": 48,
         "tr_mode": 1, "scenarios": 512, "pincap": False},
        # a few activities, an odd number of them, with the pin caps trained too
        {"name": "autograd 20k x 37", "kind": "autograd", "cells": 20000, "start": 1474, "depth": 38,
         "tr_mode": 0, "scenarios": 37, "pincap": True},
        # temporally correlated activities (lag-one), all gradients
        {"name": "lag one 50k x 128", "kind": "autograd", "cells": 50000, "start": 3685, "depth": 44, "tr_mode": 2,
         "scenarios": 128, "pincap": True},
        # a power-virus search from 256 starts
        {"name": "virus 50k x 256", "kind": "virus", "cells": 50000, "start": 3685, "depth": 44, "scenarios": 256,
         "steps": 40},
        # one turn of a sizing loop: 1 % of the cells resized, the 1,000 best candidates next
        {"name": "sizing 300k", "kind": "sizing", "cells": 300000, "start": 22110, "depth": 54, "tr_mode": 0,
         "grad_mode": 1, "top": 1000},
        # the serving configuration in small: three resident designs, a burst of mixed requests
        {"name": "serve 96 requests", "kind": "serve", "cells": 120000, "requests": 96, "batch": 32, "slots": 2},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["gradient", "gradient", "step", "step", "simulate", "autograd", "autograd", "autograd",
                       "virus", "sizing", "serve"])
    if kind == "serve":
        return {"kind": kind, "cells": _log(rng, 4000, 120000), "requests": rng.randint(1, 96),
                "batch": rng.choice([8, 16, 32, 64]), "slots": rng.randint(1, 2)}
    most = {"gradient": 800000, "step": 400000, "simulate": 120000, "autograd": 120000, "virus": 50000,
            "sizing": 300000}[kind]
    cells = _log(rng, 1500, most)
    depth = max(4, min(int(_log(rng, 12, 110)), cells // 20))
    c = {"kind": kind, "cells": cells, "start": max(24, int(cells * rng.uniform(0.04, 0.1))), "depth": depth}
    if kind in ("gradient", "step", "simulate", "sizing"):
        c["tr_mode"] = rng.randint(0, 1)
    if kind == "step":
        c["host"] = rng.random() < 0.5
    if kind in ("step", "sizing"):
        c["grad_mode"] = rng.randint(0, 2)
    if kind in ("step", "simulate"):
        c["words"] = _log(rng, 2, max(8, min(1024, 40000000 // cells)))
    if kind == "sizing":
        c["top"] = _log(rng, 1, 5000)
    if kind in ("autograd", "virus"):
        c["scenarios"] = _log(rng, 1, max(2, min(700, (60000000 if kind == "autograd" else 12000000) // cells)))
    if kind == "autograd":
        c["tr_mode"] = rng.randint(0, 2)
        c["pincap"] = rng.random() < 0.5
        if c["tr_mode"] == 2:
            c["scenarios"] = max(1, c["scenarios"] // 8)
    if kind == "virus":
        c["steps"] = rng.randint(5, 40)
    return c


# ------------------------------------------------------------- the user's data
def _spec(cells, start, depth):
    n_pi = max(1, start // 9)
    return netgen.NetlistSpec(cells, n_pi, start - n_pi, depth, 32 if cells >= 500000 else 16, 1 + cells % 89)


def _serve_cells(c):
    return [max(1500, c["cells"] // 24), max(1500, c["cells"] // 6), c["cells"]]


def _serve_spec(cells):
    return _spec(cells, max(24, int(cells * 0.0737)), int(min(80, max(16, round(24 + 14 * math.log10(cells / 2000))))))


@functools.lru_cache(maxsize=4)
def _text(spec):
    return netgen.netlist_text(spec)


@functools.lru_cache(maxsize=1)
def _library():
    return netgen.library_text()


_compiled = {}   # the last compiled netlist: a program compiles once and keeps the result


def _compile(spec):
    if spec not in _compiled:
        for old in list(_compiled):
            dp.dp_compiled_free(_compiled.pop(old))
        _compiled[spec] = dp.dp_compile(netgen.netlist_text(spec), _library())
    return _compiled[spec]


class Resident:
    """A design on the GPU with its context, as a program keeps it."""

    def __init__(self, spec):
        self.ctx = dp.dp_create(0, torch.cuda.current_stream().cuda_stream)
        self.d = dp.dp_design_upload(self.ctx, _compile(spec))
        i = dp.dp_design_info(self.d)
        self.n_start, self.n_cells, self.n_nets, self.n_edges = i.n_start, i.n_cells, i.n_nets, i.n_edges

    def __del__(self):
        if getattr(self, "d", None):
            dp.dp_design_free(self.d)
            dp.dp_destroy(self.ctx)
            self.d = None


class Server:
    def __init__(self, cfg):
        self.srv = dp.dp_server_create(cfg)

    def __del__(self):
        if getattr(self, "srv", None):
            dp.dp_server_destroy(self.srv)
            self.srv = None


def _activity(n, s, seed):
    """SP ~ U[0.1, 0.9] and TR ~ U[0, 2 min(SP, 1 - SP)], binary32, [n, s]."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    sp = 0.1 + 0.8 * torch.rand(n, s, generator=g, device=DEV)
    tr = torch.rand(n, s, generator=g, device=DEV) * (1.999 * torch.minimum(sp, 1 - sp))
    return sp, tr


def _pinned(t):
    return t.cpu().pin_memory()


def _host_out(*shape, dtype=torch.float32):
    return torch.zeros(*shape, dtype=dtype).pin_memory()


def _resizes(n_cells, count, seed):
    """`count` different cells and their new pin caps (X2 or X4 drive)."""
    r = np.random.default_rng(seed)
    cells = np.sort(r.choice(n_cells, count, replace=False)).astype(np.int32)
    return cells, r.choice(np.array([1.6, 3.2], np.float32), count)


def _serve_jobs(c):
    """(design, new activity or not, gradients or not) of every request of the case's mix."""
    r = np.random.default_rng(c["cells"])
    return [(int(r.integers(3)), bool(r.integers(2)), bool(r.integers(2))) for _ in range(c["requests"])]


def _config(c):
    return dp.config(tr_mode=c.get("tr_mode", 0), grad_mode=c.get("grad_mode", 0), sim_words=c.get("words", 64))


def prepare(case, seed):
    c = dict(case)
    st = {"case": c}
    kind = c["kind"]
    if kind == "serve":
        return _prepare_serve(c, seed)
    spec = _spec(c["cells"], c["start"], c["depth"])
    if kind in ("autograd", "virus"):
        st["design"] = ta.Design(_text(spec), _library())
        sp, tr = _activity(c["start"], c["scenarios"], seed)
        st["sp"], st["tr"] = sp, tr
        if kind == "autograd":
            st["sp"].requires_grad_()
            st["tr"].requires_grad_()
            if c["pincap"]:
                g = torch.Generator(device=DEV).manual_seed(seed + 1)
                st["pincap"] = (0.8 + 2.4 * torch.rand(c["cells"], generator=g, device=DEV)).requires_grad_()
        return st
    r = st["res"] = Resident(spec)
    st["cfg"] = _config(c)
    sp, tr = _activity(r.n_start, 1, seed)
    sp, tr = sp[:, 0].contiguous(), tr[:, 0].contiguous()
    host = bool(c.get("host"))
    st["sp"], st["tr"] = (_pinned(sp), _pinned(tr)) if host else (sp, tr)
    st["on"] = 0 if host else 1
    new = _host_out if host else functools.partial(torch.zeros, device=DEV)
    if kind in ("gradient", "step"):
        st["out"] = {"grad_sp": new(r.n_start), "grad_tr": new(r.n_start), "grad_pincap": new(r.n_cells),
                     "grad_cload": new(r.n_nets)}
        st["watts"] = np.zeros(2) if kind == "step" else torch.zeros(1, dtype=torch.float64, device=DEV)
    if kind == "simulate":
        n = r.n_nets
        st["out"] = {k: torch.zeros(n, device=DEV) for k in ("sp", "tr", "beta", "tr_hyb")}
        st["out"] |= {k: torch.zeros(n, dtype=torch.int32, device=DEV) for k in ("toggles", "ones")}
        st["watts"] = torch.zeros(2, dtype=torch.float64, device=DEV)
    if kind == "sizing":
        dp.dp_set_inputs(r.ctx, r.d, sp, tr, 1, 1)
        dp.dp_propagate(r.ctx, r.d, st["cfg"])
        dp.dp_simulate(r.ctx, r.d, st["cfg"])
        st["cells"], st["caps"] = _resizes(r.n_cells, max(1, r.n_cells // 100), seed)
        k = min(c["top"], r.n_cells)
        st["out"] = {"scores": torch.zeros(r.n_cells, device=DEV), "grad_pincap": torch.zeros(r.n_cells, device=DEV),
                     "grad_sp": torch.zeros(r.n_start, device=DEV),
                     "top_cells": torch.zeros(k, dtype=torch.int32, device=DEV),
                     "top_scores": torch.zeros(k, device=DEV)}
    return st


def _prepare_serve(c, seed):
    server = Server(dp.server_config(max_batch=c["batch"], slots_per_design=c["slots"]))
    sizes = []
    for i, cells in enumerate(_serve_cells(c)):
        spec = _serve_spec(cells)
        sp, tr = _activity(spec.n_start, 1, seed + 1000 + i)
        dp.dp_server_add_design(server.srv, _text(spec), _library(), sp.cpu().numpy()[:, 0].copy(),
                                tr.cpu().numpy()[:, 0].copy())
        sizes.append((spec.n_start, cells))
    jobs = _serve_jobs(c)
    power = _host_out(len(jobs), dtype=torch.float64)
    grads = [sum(g for k, _, g in jobs if k == i) for i in range(3)]
    out = [{"grad_sp": _host_out(grads[i], sizes[i][0]), "grad_tr": _host_out(grads[i], sizes[i][0]),
            "grad_pincap": _host_out(grads[i], sizes[i][1])} for i in range(3)]
    reqs, keep, row = [], [], [0, 0, 0]
    for j, (k, fresh, grad) in enumerate(jobs):
        ns, nc = sizes[k]
        kw = {}
        if fresh:
            sp, tr = _activity(ns, 1, seed + 2000 + j)
            kw["sp"], kw["tr"] = _pinned(sp[:, 0].contiguous()), _pinned(tr[:, 0].contiguous())
        else:
            cells, caps = _resizes(nc, max(1, nc // 100), seed + 3000 + j)
            kw["cells"], kw["pincap"] = _pinned(torch.from_numpy(cells)), _pinned(torch.from_numpy(caps))
        if grad:
            kw |= {"want_grad": 1} | {n: out[k][n][row[k]] for n in out[k]}
            row[k] += 1
        keep.append(kw)
        reqs.append(dp.request(k, power[j:j + 1], **kw))
    return {"case": c, "server": server, "reqs": reqs, "keep": keep, "out": {"power": power, "designs": out}}


# -------------------------------------------------------------------- one pass
def run(state):
    kind = state["case"]["kind"]
    if kind == "autograd":
        sp, tr, pin = state["sp"], state["tr"], state.get("pincap")
        p = ta.power(state["design"], sp, tr, pin, tr_mode=state["case"]["tr_mode"])
        leaves = [sp, tr] + ([pin] if pin is not None else [])
        return [p.detach()] + list(torch.autograd.grad(p.sum(), leaves))
    if kind == "virus":
        v = ta.power_virus(state["design"], state["sp"], state["tr"], state["case"]["steps"], 2e-3)
        return {"sp": v.sp, "v0": v.v0, "p_virus": v.p_virus, "proxy_start": v.proxy_start, "proxy_end": v.proxy_end}
    if kind == "serve":
        srv = state["server"].srv
        tickets = [dp.dp_server_submit(srv, r) for r in state["reqs"]]
        for t in tickets:
            dp.dp_server_wait(srv, t)
        return state["out"]
    r, cfg, on = state["res"], state["cfg"], state["on"]
    ctx, d, out = r.ctx, r.d, state["out"]
    if kind == "sizing":
        dp.dp_set_pincap(ctx, d, state["cells"], state["caps"])
        dp.dp_backward(ctx, d, cfg, out["grad_sp"], None, out["grad_pincap"], None, 1)
        dp.dp_sizing_scores(ctx, d, cfg, 0, out["scores"], len(out["top_cells"]), out["top_cells"],
                            out["top_scores"], 1)
        return out
    dp.dp_set_inputs(ctx, d, state["sp"], state["tr"], 1, on)
    if kind == "step":
        dp.dp_step(ctx, d, cfg, out["grad_sp"], out["grad_tr"], out["grad_pincap"], out["grad_cload"],
                   state["watts"], on)
    elif kind == "gradient":
        dp.dp_propagate(ctx, d, cfg)
        dp.dp_get_power(ctx, d, state["watts"], 0, 1)
        dp.dp_backward(ctx, d, cfg, out["grad_sp"], out["grad_tr"], out["grad_pincap"], out["grad_cload"], 1)
    else:
        dp.dp_propagate(ctx, d, cfg)
        dp.dp_simulate(ctx, d, cfg)
        for h in (0, 1):
            dp.dp_get_power(ctx, d, state["watts"][h:h + 1], h, 1)
        dp.dp_get_nets(ctx, d, out["sp"], out["tr"], out["beta"], out["tr_hyb"], out["toggles"], out["ones"], 1)
    return [state["watts"], out]


# ---------------------------------------------------------- what it has to move
def work(case):
    """Compulsory bytes, every structure, input and output array once (compact CSR, int32 indices,
    binary32 values), and the operations of the cells' polynomials.  The generator's cells have 29/13
    inputs on average."""
    c = case
    if c["kind"] == "serve":
        got = {"bytes": 0.0, "flops": 0.0}
        for k, fresh, grad in _serve_jobs(c):
            nc = _serve_cells(c)[k]
            ns = max(24, int(nc * 0.0737))
            got["bytes"] += (8 * ns if fresh else 8 * max(1, nc // 100)) + (8 * ns + 4 * nc if grad else 0)
            got["flops"] += (40.0 if fresh else 6.0) * nc + (40.0 * nc if grad else 0.0)
        for nc in _serve_cells(c):
            got["bytes"] += 26 * nc
        return got
    nc, ns = c["cells"], c["start"]
    nn, ne = nc + ns, nc * 29 // 13
    fanin, fanout = 4 * (nc + 1) + 4 * ne + nc, 4 * (nn + 1) + 4 * ne
    s, t = c.get("scenarios", 1), c.get("words", 0)
    grads = 8 * ns * s + 4 * nc + 4 * nn
    kind = c["kind"]
    if kind == "gradient":
        return {"bytes": 2 * fanin + fanout + 8 * ns + 4 * nn + grads, "flops": 80 * nc}
    if kind == "step":
        return {"bytes": 2 * fanin + fanout + 8 * ns + 4 * nn + grads, "flops": (80 + 8 * t) * nc + 40 * t * ns}
    if kind == "simulate":
        return {"bytes": fanin + 8 * ns + 4 * nn + 24 * nn, "flops": (40 + 8 * t) * nc + 40 * t * ns}
    if kind == "sizing":
        return {"bytes": fanin + fanout + 12 * nn + 4 * ns + 8 * nc + 8 * (nc // 100), "flops": 40 * nc}
    lag = 6 if c.get("tr_mode") == 2 else 1
    one = {"bytes": 2 * fanin + fanout + 4 * nn + 8 * ns * s + 8 * ns * s + 8 * s + (8 * nc if c.get("pincap") else 0),
           "flops": 80 * nc * s * lag}
    if kind == "virus":
        return {"bytes": one["bytes"] * c["steps"], "flops": one["flops"] * c["steps"]}
    return one


# ------------------------------------------- the same in 64 bits, without the package
class Plain:
    """A netlist read from its text into torch arrays: nets in declaration order, cells in line
    order, startpoints in the order of their lines."""

    def __init__(self, text, library):
        tables, pins, caps = {}, {}, {}
        for line in library.splitlines():
            w = line.split(None, 4)
            if w[:1] == ["cell"]:
                names = [p for p in dict.fromkeys(re.findall(r"[A-Z]\w*", w[4]))]
                names.sort()
                expr = w[4].replace("!", "~")
                tables[w[1]] = [eval(expr, {}, {n: (m >> (2 - i)) & 1 for i, n in enumerate(names)}) & 1  # noqa: S307
                                for m in range(8)]   # input 0 in the highest of three bits
                pins[w[1]], caps[w[1]] = names, float(np.float32(w[3]))
            elif w[:1] == ["seq"]:
                dff_cap = float(np.float32(w[4]))
        net, wire, start, dff_d, cells = {}, [], [], [], []
        refs = {r: i for i, r in enumerate(tables)}
        for line in text.splitlines():
            w = line.split()
            if w[0] == "net":
                net[w[1]] = len(wire)
                wire.append(w[2])
            elif w[0] == "cell":
                cells.append(w)
            elif w[0] == "input":
                start.append(net[w[1]])
            elif w[0] == "dff":
                dff_d.append(net[w[3][2:]])
                start.append(net[w[4][2:]])
        wire = np.array(wire).astype(np.float32).astype(np.float64)
        # a cell line names its inputs in the library's order (of their names), then its output
        kinds = [refs[w[2]] for w in cells]
        outs = [net[w[-1].partition("=")[2]] for w in cells]
        fans = [([net[x.partition("=")[2]] for x in w[3:-1]] + [-1, -1])[:3] for w in cells]
        assert all([x.partition("=")[0] for x in w[3:-1]] == pins[w[2]] for w in cells[:5000])
        self.nn, self.nc = len(wire), len(outs)
        out, fan, kind = np.array(outs), np.array(fans), np.array(kinds)
        fan = np.where(fan < 0, self.nn, fan)   # a net that is always 0 in the place of no input
        level = np.zeros(self.nn + 1, np.int64)
        while True:
            up = 1 + level[fan].max(1)
            if np.array_equal(up, level[out]):
                break
            level[out] = up
        base = wire.copy()
        np.add.at(base, np.array(dff_d, np.int64), dff_cap)
        dev = functools.partial(torch.as_tensor, device=DEV)
        self.out, self.fan, self.start = dev(out), dev(fan), dev(np.array(start))
        self.table = dev(np.array(list(tables.values()), np.float64)[kind])
        self.base, self.pincap = dev(base), dev(np.array(list(caps.values()))[kind])
        order = np.argsort(level[out], kind="stable")
        cuts = np.flatnonzero(np.diff(level[out][order])) + 1
        self.levels = [dev(x) for x in np.split(order, cuts)]

    def cload(self, pincap):
        """[nn, ...] loads for pin caps [nc, ...]"""
        c = torch.zeros((self.nn + 1,) + pincap.shape[1:], dtype=torch.float64, device=DEV)
        for j in range(3):
            c.index_add_(0, self.fan[:, j], pincap)
        return c[:-1] + self.base.reshape((-1,) + (1,) * (pincap.dim() - 1))

    def to_cells(self, per_net):
        """The sum over a cell's inputs of a per-net value: what a pin cap is multiplied by."""
        z = torch.cat([per_net, torch.zeros_like(per_net[:1])])
        return z[self.fan].sum(1)


def _fold(table, weights):
    """sum over input states of table[n, states] times the weights [n, b, s] of each input"""
    v = table[:, :, None]
    for w in reversed(weights):
        b = w.shape[1]
        v = (v.reshape(v.shape[0], -1, b, v.shape[2]) * w[:, None]).sum(2)
    return v[:, 0]


def _cell_p(table, x, q):
    return _fold(table, [torch.stack([q[:, j], x[:, j]], 1) for j in range(3)])


def _cell_t(table, x, t):
    m = torch.arange(64, device=DEV)
    a = sum(((m >> (2 * (2 - i) + 1)) & 1) << (2 - i) for i in range(3))
    b = sum(((m >> (2 * (2 - i))) & 1) << (2 - i) for i in range(3))
    differ = (table[:, a] != table[:, b]).double()
    return _fold(differ, [torch.stack([1 - x[:, j] - t[:, j] / 2, t[:, j] / 2, t[:, j] / 2, x[:, j] - t[:, j] / 2], 1)
                          for j in range(3)])


def _exact_forward(n, sp, tr, tr_mode):
    """P, 1 - P and TR of every net, [nn, S].  1 - P is folded beside P (deep nets are within 1e-15 of
    0 or 1), and both are divided by their sum, so that its rounding does not grow along the paths."""
    s = sp.shape[1]
    p = torch.zeros(n.nn + 1, s, dtype=torch.float64, device=DEV)
    t, q = torch.zeros_like(p), torch.ones_like(p)
    p[n.start], q[n.start], t[n.start] = sp, 1 - sp, tr
    for ids in n.levels:
        o, f = n.out[ids], n.fan[ids]
        x, y = p[f], q[f]
        a, b = _cell_p(n.table[ids], x, y), _cell_p(1 - n.table[ids], x, y)
        p[o], q[o] = a / (a + b), b / (a + b)
        if tr_mode == 2:
            t[o] = _cell_t(n.table[ids], x, t[f])
    if tr_mode != 2:
        t = 2 * p * q
        if tr_mode == 0:
            t[n.start] = tr
    return p[:-1], q[:-1], t[:-1]


def _exact_adjoint(n, p, t, local_p, local_t, scale, tr_mode):
    """Adjoints of every net's P (and T in the lag-one mode); `scale` multiplies each net's whole
    adjoint before it goes on to the fanins (Eq. 6)."""
    z = torch.zeros_like(p[:1])
    p, t = torch.cat([p, z]), torch.cat([t, z])
    gp, gt = torch.cat([local_p, z]), torch.cat([local_t, z])
    for ids in reversed(n.levels):
        o, f = n.out[ids], n.fan[ids]
        if scale is not None:
            gp[o] *= scale[o]
        with torch.enable_grad():
            x = p[f].requires_grad_()
            y = t[f].requires_grad_()
            v = (_cell_p(n.table[ids], x, 1 - x) * gp[o]).sum()
            if tr_mode == 2:
                v = v + (_cell_t(n.table[ids], x, y) * gt[o]).sum()
            dx, dy = torch.autograd.grad(v, (x, y), allow_unused=True)
        for j in range(3):
            gp.index_add_(0, f[:, j], dx[:, j])
            if dy is not None:
                gt.index_add_(0, f[:, j], dy[:, j])
    if scale is not None:
        gp[n.start] *= scale[n.start]
    return gp[:-1], gt[:-1]


def _exact_model(n, sp, tr, tr_mode, cl, k):
    """P, TR, d TR / d P, power [S] and the gradients of the startpoints' SP and TR"""
    p, q, t = _exact_forward(n, sp, tr, tr_mode)
    slope = 2 * (q - p)
    if tr_mode == 0:
        slope[n.start] = 0
    local = torch.zeros_like(p) if tr_mode == 2 else k * cl * slope
    direct = k * cl * torch.ones_like(p)
    gp, gt = _exact_adjoint(n, p, t, local, direct if tr_mode == 2 else torch.zeros_like(p), None, tr_mode)
    if tr_mode == 0:
        gt = direct
    return p, t, slope, k * (t * cl).sum(0), gp[n.start], gt[n.start] if tr_mode != 1 else torch.zeros_like(sp)


def _popcount(x):
    x = x - ((x >> 1) & 0x5555555555555555)
    x = (x & 0x3333333333333333) + ((x >> 2) & 0x3333333333333333)
    x = (x + (x >> 4)) & 0x0F0F0F0F0F0F0F0F
    return ((x * 0x0101010101010101) >> 56) & 0x7F


def _chains(sp, tr, words, seed=42):
    """[n_start, words] 64-lane Markov chains from Philox4x32-10 draws of 16 bits"""
    ns, m32 = sp.shape[0], 0xFFFFFFFF
    dev = functools.partial(torch.arange, device=DEV)
    half = (words + 1) // 2
    c = [dev(ns)[:, None, None].expand(ns, half, 16), dev(half)[None, :, None].expand(ns, half, 16),
         dev(16)[None, None, :].expand(ns, half, 16), torch.zeros(ns, half, 16, dtype=torch.int64, device=DEV)]
    k0, k1 = seed & m32, seed >> 32
    for _ in range(10):
        a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((b >> 32) & m32) ^ c[1] ^ k0, b & m32, ((a >> 32) & m32) ^ c[3] ^ k1, a & m32]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    u = torch.stack(c, 2).reshape(ns, half, 64)   # lane 16 r + q
    thr = lambda v: torch.floor(v.clamp(0, 1) * 65536).long()  # noqa: E731
    t0, t10, t01 = thr(sp), thr(tr / (2 * sp)), thr(tr / (2 * (1 - sp)))
    lane = dev(64)
    got, state = [], None
    for i in range(words):
        d = (u[:, i // 2] >> (16 * (i & 1))) & 0xFFFF
        state = d < t0 if i == 0 else state ^ (d < torch.where(state, t10, t01))
        got.append((state.long() << lane).sum(1))
    return torch.stack(got, 1)


def _exact_hybrid(n, sp, tr, t, words):
    """toggles, ones, beta (Eq. 4, Eq. 5) of every net"""
    w = torch.zeros(n.nn + 1, words, dtype=torch.int64, device=DEV)
    w[n.start] = _chains(sp, tr, words)
    for ids in n.levels:
        x = w[n.fan[ids]]
        v = torch.zeros_like(x[:, 0])
        for m in range(8):
            s = -(n.table[ids][:, m].long())[:, None]
            for j in range(3):
                s = s & (x[:, j] if (m >> (2 - j)) & 1 else ~x[:, j])
            v |= s
        w[n.out[ids]] = v
    w = w[:-1]
    ones = _popcount(w).sum(1)
    toggles = _popcount(w[:, 1:] ^ w[:, :-1]).sum(1)
    t = t[:, 0]
    acc = toggles.double() / (64 * (words - 1))
    beta = torch.where(t > 0, (acc / t).clamp(float(np.float32(0.1)), 10), torch.where(toggles > 0, 10.0, 1.0))
    return toggles, ones, beta


def exact(case, seed):
    c = case
    k = 0.5 * 0.8 * 0.8 * 1e9 * 1e-15
    kind, mode = c["kind"], c.get("tr_mode", 0)
    if kind == "virus" or c["cells"] > 700000 or c["cells"] * c.get("words", 0) > 45000000:
        return None   # a search ends at a vector of bits; the others take too long in Python
    with torch.no_grad():
        if kind == "serve":
            return _exact_serve(c, seed, k)
        n = Plain(netgen.netlist_text(_spec(c["cells"], c["start"], c["depth"])), _library())
        if kind == "autograd":
            sp, tr = (x.double() for x in _activity(c["start"], c["scenarios"], seed))
            pincap = n.pincap
            if c["pincap"]:
                g = torch.Generator(device=DEV).manual_seed(seed + 1)
                pincap = (0.8 + 2.4 * torch.rand(c["cells"], generator=g, device=DEV)).double()
            _, t, _, watts, gsp, gtr = _exact_model(n, sp, tr, mode, n.cload(pincap)[:, None], k)
            return [watts, gsp, gtr] + ([k * n.to_cells(t.sum(1))] if c["pincap"] else [])
        sp, tr = (x.double() for x in _activity(c["start"], 1, seed))
        pincap = n.pincap.clone()
        if kind == "sizing":
            cells, caps = _resizes(n.nc, max(1, n.nc // 100), seed)
            pincap[torch.from_numpy(cells).long().to(DEV)] = torch.from_numpy(caps).double().to(DEV)
        cl = n.cload(pincap)[:, None]
        p, t, slope, watts, gsp, gtr = _exact_model(n, sp, tr, mode, cl, k)
        if kind == "gradient":
            return [watts, {"grad_sp": gsp[:, 0], "grad_tr": gtr[:, 0], "grad_pincap": k * n.to_cells(t)[:, 0],
                            "grad_cload": k * t[:, 0]}]
        toggles, ones, beta = _exact_hybrid(n, sp, tr, t, c.get("words", 64))
        th = t * beta[:, None]
        both = torch.stack([watts[0], k * (th * cl).sum()])
        if kind == "simulate":
            return [both, {"sp": p[:, 0], "tr": t[:, 0], "beta": beta, "tr_hyb": th[:, 0], "toggles": toggles,
                           "ones": ones}]
        alpha, gnet = t, None
        if c["grad_mode"]:
            alpha = th
            local = k * cl * slope
            if c["grad_mode"] == 2:
                local = local * beta[:, None]
            gnet, _ = _exact_adjoint(n, p, t, local, torch.zeros_like(p),
                                     beta[:, None] if c["grad_mode"] == 1 else None, mode)
            gsp = gnet[n.start]
            gtr = k * (beta[:, None] * cl)[n.start] if mode == 0 else torch.zeros_like(sp)
        gpin = k * n.to_cells(alpha)[:, 0]
        if kind == "step":
            return [both, {"grad_sp": gsp[:, 0], "grad_tr": gtr[:, 0], "grad_pincap": gpin,
                           "grad_cload": k * alpha[:, 0]}]
        if gnet is None:
            gnet, _ = _exact_adjoint(n, p, t, k * cl * slope, torch.zeros_like(p), None, mode)
        scores = (gnet.abs() * k * alpha * cl)[n.out, 0]
        return {"scores": scores, "grad_pincap": gpin, "grad_sp": gsp[:, 0], "top_cells": None,
                "top_scores": torch.sort(scores, descending=True)[0][:min(c["top"], n.nc)]}


def _exact_serve(c, seed, k):
    jobs = _serve_jobs(c)
    power = torch.zeros(len(jobs), dtype=torch.float64)
    designs = []
    for i, cells in enumerate(_serve_cells(c)):
        spec = _serve_spec(cells)
        n = Plain(netgen.netlist_text(spec), _library())
        ref = _activity(spec.n_start, 1, seed + 1000 + i)
        mine = [j for j, job in enumerate(jobs) if job[0] == i]
        got = {"grad_sp": [], "grad_tr": [], "grad_pincap": []}
        for at in range(0, len(mine), 16):
            part = mine[at:at + 16]
            act = [_activity(spec.n_start, 1, seed + 2000 + j) if jobs[j][1] else ref for j in part]
            pincap = n.pincap[:, None].repeat(1, len(part))
            for col, j in enumerate(part):
                if not jobs[j][1]:
                    ids, caps = _resizes(n.nc, max(1, n.nc // 100), seed + 3000 + j)
                    pincap[torch.from_numpy(ids).long().to(DEV), col] = torch.from_numpy(caps).double().to(DEV)
            sp, tr = (torch.cat([a[x] for a in act], 1).double() for x in (0, 1))
            _, t, _, watts, gsp, gtr = _exact_model(n, sp, tr, 0, n.cload(pincap), k)
            power[part] = watts.cpu()
            cols = [col for col, j in enumerate(part) if jobs[j][2]]
            for name, v in (("grad_sp", gsp), ("grad_tr", gtr), ("grad_pincap", k * n.to_cells(t))):
                got[name].append(v[:, cols].T)
        ns, nc = spec.n_start, cells
        designs.append({name: torch.cat(v) if v else torch.zeros(0, nc if name == "grad_pincap" else ns,
                                                                 dtype=torch.float64)
                        for name, v in got.items()})
    return {"power": power, "designs": designs}
