"""Performance cases: the work that users of this framework have it do.

Two groups, all through public entry points:

* whole solves of a graphical model -- PR + MAR (``Model.mar`` /
  ``Model.mar_dev``), learning (``autograd.log_partition`` and its gradient),
  MAP, MMAP and exact sampling -- on the model families of ``synth``;
* single pairwise contractions (``tn.contract_dev``), the layer that every
  solve is made of: GEMM-shaped nodes in each precision, skinny nodes (one
  group too small for a GEMM) and max-plus nodes with argmax capture.

A program keeps its model's structure and contraction tree (the plan) and
comes with new couplings, evidence or operands: the seed gives those, the case
the structure.  Solves in FP32, TF32 or BF16 hold their tensors in 32 bits, and
a program that asks for them keeps their results in 32 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2405_14060_gb300 import synth, tn
from paper_2405_14060_gb300.autograd import log_partition


def listed():
    return [
        # the smallest solve: one 10 x 10 grid, double precision, host arrays in and out
        dict(name="mar_grid10_fp64", kind="mar", graph="grid", size=10, batch=1, prec="fp64",
             observed=0.0, host=True),
        # one large grid, all marginals, tensors on the device
        dict(name="mar_grid24_tf32", kind="mar", graph="grid", size=24, batch=1, prec="tf32",
             observed=0.0, host=False),
        # many evidence sets of one random 3-regular graph in one call (the benchmark's model;
        # a batch whose tensors leave room for other work on the card)
        dict(name="mar_rrg200_b32_bf16", kind="mar", graph="rrg", size=200, batch=32, prec="bf16",
             observed=0.1, host=False),
        # a training step: log Z of a batch of data and its gradient in every log table
        dict(name="learn_grid12_b16_fp64", kind="learn", graph="grid", size=12, batch=16,
             prec="fp64", observed=0.2),
        # most likely assignment of a 300-variable Bayesian network with sensors read
        dict(name="map_bn300_fp32", kind="map", graph="bn", size=300, prec="fp32", observed=0.2),
        # the same network with 30% of the free variables queried and the rest summed
        dict(name="mmap_bn300_fp32", kind="mmap", graph="bn", size=300, prec="fp32", observed=0.2),
        # exact samples of a medium grid, default precision
        dict(name="sample_grid16_100k", kind="sample", graph="grid", size=16, prec="fp64",
             samples=100000),
        # contraction of two large tensors with interleaved label groups, tensor cores
        contraction("gemm_bf16_4096", "mkMK,KnkN->mnMN",
                    "bf16", m=64, M=64, k=64, K=64, n=64, N=64),
        # ragged groups with a shared (batch) label
        contraction("gemm_tf32_ragged", "gmk,gkn->gmn", "tf32", g=3, m=1000, k=1155, n=777),
        # the same kind of node in full single precision, both operands transposed
        contraction("gemm_fp32_2048", "km,nk->mn", "fp32", m=2048, k=1024, n=1536),
        # a long tensor times a small one: 2^20 rows, neither summed nor new group of GEMM size
        contraction("skinny_fp32", "mgk,kgn->ngm", "fp32", m=262144, g=4, k=24, n=36),
        # max-plus node with argmax capture (the forward pass of MAP)
        contraction("maxplus_fp32", "mgk,gkn->gmn", "fp32", semiring=1, g=4, m=1024, k=48, n=96),
    ]


def contraction(name, spec, prec, semiring=0, **sizes):
    return dict(name=name, kind="contract", spec=spec, prec=prec, semiring=semiring, **sizes)


GEMM_SPECS = ["mk,kn->mn", "km,nk->mn", "mk,nk->nm", "gmk,gkn->gmn", "kgm,gnk->gnm",
              "mkMK,KnkN->mnMN", "kmKM,nNkK->nmMN"]
SKINNY_SPECS = ["mk,kn->mn", "mk,kn->nm", "km,kn->nm", "mgk,kgn->ngm", "gmk,gkn->gmn",
                "kmg,gkn->mng"]
MAX_SPECS = ["mk,kn->mn", "mgk,gkn->gmn", "km,nk->nm", "kgm,gn->mng"]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["mar", "mar", "learn", "map", "mmap", "sample", "gemm", "gemm", "skinny",
                       "max"])
    if kind == "mar":
        if rng.random() < 0.6:
            prec = rng.choice(["fp64", "fp32", "tf32", "bf16"])
            size = rng.randint(5, 16 if prec == "fp64" else 22)
            return dict(kind="mar", graph="grid", size=size, prec=prec, observed=rng.choice([0.0, 0.1]),
                        batch=1 if size > 14 else _log_int(rng, 1, 48), host=rng.random() < 0.5)
        return dict(kind="mar", graph="rrg", size=2 * rng.randint(15, 60), batch=_log_int(rng, 1, 64),
                    prec=rng.choice(["fp64", "fp32", "tf32", "bf16"]), observed=rng.uniform(0.0, 0.3),
                    host=rng.random() < 0.5)
    if kind == "learn":
        return dict(kind="learn", graph="grid", size=rng.randint(4, 13), batch=_log_int(rng, 1, 32),
                    prec=rng.choice(["fp64", "fp32"]), observed=rng.uniform(0.0, 0.5))
    if kind == "map":
        if rng.random() < 0.5:
            return dict(kind="map", graph="bn", size=_log_int(rng, 40, 500),
                        prec=rng.choice(["fp64", "fp32"]), observed=rng.uniform(0.0, 0.3))
        return dict(kind="map", graph="grid", size=rng.randint(6, 20),
                    prec=rng.choice(["fp64", "fp32"]), observed=0.0)
    if kind == "mmap":
        return dict(kind="mmap", graph="bn", size=_log_int(rng, 60, 400),
                    prec=rng.choice(["fp64", "fp32"]), observed=rng.uniform(0.1, 0.3))
    if kind == "sample":
        return dict(kind="sample", graph="grid", size=rng.randint(6, 16), prec="fp64",
                    samples=_log_int(rng, 1000, 200000))
    if kind == "gemm":
        spec = rng.choice(GEMM_SPECS)
        prec = rng.choice(["bf16", "tf32", "fp32", "fp64"])
        top = 1024 if prec == "fp64" else 2048 if prec == "fp32" else 4096
        out = dict(kind="contract", spec=spec, prec=prec, semiring=0)
        for low, up in (("m", "M"), ("n", "N"), ("k", "K")):
            size = _log_int(rng, 64, top)
            if up in spec:          # two labels of the group, about equal
                a = max(8, int(math.sqrt(size)))
                out[low], out[up] = a, -(-size // a)
            else:
                out[low] = size
        if "g" in spec:
            out["g"] = rng.randint(2, 4)
        return out
    if kind == "skinny":
        spec = rng.choice(SKINNY_SPECS)
        out = dict(kind="contract", spec=spec, prec=rng.choice(["fp32", "tf32", "fp64"]), semiring=0,
                   m=_log_int(rng, 1000, 1000000), k=rng.randint(2, 63), n=rng.randint(2, 63))
        if "g" in spec:
            out["g"] = rng.randint(2, 6)
            out["m"] = max(200, out["m"] // out["g"])
        return out
    spec = rng.choice(MAX_SPECS)
    out = dict(kind="contract", spec=spec, prec=rng.choice(["fp32", "fp64"]), semiring=1,
               m=_log_int(rng, 100, 4000), k=rng.randint(2, 64), n=rng.randint(2, 128))
    if "g" in spec:
        out["g"] = rng.randint(2, 4)
    return out


# ------------------------------------------------------------------ inputs

_plans = {}   # structure -> (model of that structure, tree): a user's program keeps its plan


def _structure(case):
    key = (case["graph"], case["size"])
    if key not in _plans:
        n = case["size"]
        if case["graph"] == "grid":
            m = synth.grid_ising(n, 1)
        elif case["graph"] == "rrg":
            m = synth.rrg3_ising(n, synth.BASE_SEED + 4)
        else:
            m = synth.bayes_net(n, synth.BASE_SEED + 3)
        M = tn.Model.from_synth(m)
        if case["graph"] == "grid":
            tree = M.reassociate(*M.optimize_order(0))
        elif case["graph"] == "rrg":
            tree = M.optimize_order(3, 12, 2) if n >= 160 else M.optimize_order(1, 8, 1)
        else:
            tree = M.optimize_order(0)
        M.set_order(*tree)
        _plans[key] = (m, tree, M.tree_stats(1, "fp32"))
    return _plans[key]


def _tables(case, rng):
    """New couplings, fields or CPT rows on the case's structure."""
    m = _structure(case)[0]
    out = []
    for s, t in zip(m.scopes, m.tables):
        if case["graph"] == "bn":
            c = int(m.card[s[-1]])
            out.append(rng.dirichlet(np.ones(c), size=len(t) // c).reshape(-1))
        elif len(s) == 2:
            spin = np.array([-1.0, 1.0])
            out.append(np.exp(rng.normal() * np.outer(spin, spin)).reshape(-1))
        else:
            out.append(np.exp(rng.normal(0.0, 0.5) * np.array([-1.0, 1.0])))
    return out


def _evidence(case, rng, batch):
    """Values of the observed variables, another set of them per row; MMAP: the
    same sensors (and query) in every call, with new readings."""
    m = _structure(case)[0]
    ev = np.full((batch, m.nvars), -1, np.int32)
    fixed = np.random.default_rng(case["size"])
    k = int(round(case.get("observed", 0.0) * m.nvars))
    for b in range(batch):
        who = (fixed if case["kind"] == "mmap" else rng).choice(m.nvars, size=k, replace=False)
        ev[b, who] = rng.integers(0, m.card[who])
    return ev


def _query(case):
    m = _structure(case)[0]
    fixed = np.random.default_rng(case["size"])
    who = fixed.choice(m.nvars, size=int(round(case["observed"] * m.nvars)), replace=False)
    free = np.setdiff1d(np.arange(m.nvars), who)
    return np.sort(fixed.choice(free, size=max(1, int(round(0.3 * len(free)))),
                                replace=False)).astype(np.int32)


def _solve_inputs(case, seed):
    rng = np.random.default_rng(seed)
    return _tables(case, rng), _evidence(case, rng, case.get("batch", 1))


def _labels(case):
    (a, b), c = case["spec"].split("->")[0].split(","), case["spec"].split("->")[1]
    letters = sorted(set(a + b))
    return letters, a, b, c


def _operands(case, seed):
    letters, a, b, _ = _labels(case)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dt = torch.float64 if case["prec"] == "fp64" else torch.float32
    ops = [torch.rand([case[l] for l in s], generator=gen, device="cuda", dtype=dt) for s in (a, b)]
    if case["semiring"]:       # logarithms of the tables
        ops = [x.clamp_min_(1e-6).log_() for x in ops]
    return ops


# ----------------------------------------------------------------- running

def prepare(case, seed):
    if case["kind"] == "contract":
        letters, a, b, c = _labels(case)
        A, B = _operands(case, seed)
        C = torch.zeros([case[l] for l in c], dtype=A.dtype, device="cuda")
        st = dict(case=case, sizes=[case[l] for l in letters], A=A, B=B, C=C,
                  la=[letters.index(l) for l in a], lb=[letters.index(l) for l in b],
                  lc=[letters.index(l) for l in c])
        if case["semiring"]:
            st["argmax"] = torch.zeros(C.shape, dtype=torch.int32, device="cuda")
        return st
    m, tree, _ = _structure(case)
    tables, evid = _solve_inputs(case, seed)
    M = tn.Model.from_arrays(m.card, m.scopes, tables)
    M.set_order(*tree)
    st = dict(case=case, M=M, evid=evid, seed=seed)
    if case["kind"] == "mar" and not case["host"]:
        st["stream"] = torch.cuda.Stream()
        st["evid"] = torch.from_numpy(evid).cuda()
        st["logz"] = torch.zeros(len(evid), dtype=torch.float64, device="cuda")
        st["marg"] = torch.zeros(len(evid), int(m.card.sum()), dtype=torch.float64, device="cuda")
    elif case["kind"] == "learn":
        st["stream"] = torch.cuda.Stream()
        st["evid"] = torch.from_numpy(evid).cuda()
        st["log_tables"] = torch.from_numpy(np.log(np.concatenate(tables))).cuda().requires_grad_()
    elif case["kind"] == "mmap":
        st["query"] = _query(case)
    return st


def run(state):
    case = state["case"]
    kind, prec = case["kind"], case["prec"]
    f32 = prec != "fp64"
    if kind == "contract":
        tn.contract_dev(state["sizes"], state["la"], state["A"], state["lb"], state["B"],
                        state["lc"], state["C"], semiring=case["semiring"],
                        argmax=state.get("argmax"), prec=prec)
        return [state["C"], state["argmax"]] if case["semiring"] else state["C"]
    M = state["M"]
    if kind == "mar":
        if case["host"]:
            logz, marg = M.mar(state["evid"], prec=prec)
            return [x.astype(np.float32) for x in (logz, marg)] if f32 else [logz, marg]
        with torch.cuda.stream(state["stream"]):
            M.mar_dev(state["evid"], state["logz"], state["marg"], prec=prec,
                      stream=state["stream"].cuda_stream)
            out = [state["logz"], state["marg"]]
            return [x.float() for x in out] if f32 else out
    if kind == "learn":
        with torch.cuda.stream(state["stream"]):
            logz, marg = log_partition(M, state["log_tables"], state["evid"], prec=prec)
            grad, = torch.autograd.grad(logz.sum(), state["log_tables"])
            out = [logz.detach(), marg, grad]
            return [x.float() for x in out] if f32 else out
    if kind == "sample":
        return M.sample(case["samples"], seed=state["seed"], prec=prec)
    if kind == "map":
        x, logp = M.map(state["evid"], prec=prec)
    else:
        x, logp = M.mmap(state["query"], state["evid"], prec=prec)
    return [x, np.float32(logp) if f32 else logp]


def work(case):
    """Of a contraction: its operands and result once.  Of a solve: the nodes of
    the given tree (each operand and result once; a training step or MAR adds
    the two adjoint contractions of every node), and its samples."""
    if case["kind"] == "contract":
        letters, a, b, c = _labels(case)
        es = 8 if case["prec"] == "fp64" else 4
        prod = lambda s: math.prod(case[l] for l in s)  # noqa: E731
        return {"bytes": es * (prod(a) + prod(b) + prod(c)) + (4 * prod(c) if case["semiring"] else 0),
                "flops": 2 * prod(letters)}
    m, _, stats = _structure(case)
    es = 2 if case["prec"] == "fp64" else 1
    times = (3 if case["kind"] in ("mar", "learn") else 1) * case.get("batch", 1)
    return {"bytes": float(stats["bytes"]) * es * times + case.get("samples", 0) * m.nvars,
            "flops": float(stats["flops"]) * times}


# ------------------------------------------------------- 64-bit references

def exact(case, seed):
    if case["kind"] == "contract":
        return _exact_contract(case, seed)
    if case["kind"] == "sample":
        return None
    tables, evid = _solve_inputs(case, seed)
    m = _structure(case)[0]
    if case["kind"] in ("map", "mmap"):
        query = _query(case) if case["kind"] == "mmap" else np.arange(m.nvars)
        return [None, float(_eliminate(m, tables, evid[0], query)[0])]
    if case["graph"] == "grid":
        logs = torch.from_numpy(np.log(np.concatenate(tables))).cuda().requires_grad_()
        rows = [_grid(case["size"], logs, e) for e in evid]
    elif case["size"] <= 120:
        rows = [_eliminate(m, tables, e) for e in evid]
    else:
        return None          # the elimination of larger random graphs takes minutes
    out = [torch.stack([r[0] for r in rows]), torch.stack([r[1] for r in rows])]
    return out + [sum(r[2] for r in rows)] if case["kind"] == "learn" else out


def _exact_contract(case, seed):
    letters, a, b, c = _labels(case)
    A, B = (x.double() for x in _operands(case, seed))
    if not case["semiring"]:
        return torch.einsum(case["spec"], A, B)
    view = lambda x, s, keep: x.permute([s.index(l) for l in keep if l in s]).reshape(  # noqa: E731
        [case[l] if l in s else 1 for l in keep])
    best = None
    for k in range(case["k"]):          # one summed value at a time
        pick = lambda x, s: x.select(s.index("k"), k) if "k" in s else x  # noqa: E731
        v = view(pick(A, a), a.replace("k", ""), c) + view(pick(B, b), b.replace("k", ""), c)
        best = v if best is None else torch.maximum(best, v)
    return [best, None]


def _grid(L, logs, evid):
    """log Z, marginals and d log Z / d log tables of an L x L binary grid: the
    sites one at a time into the vector of the last L spins, 64 bits."""
    n = L * L
    u = torch.ones(n, 2, dtype=torch.float64, device=logs.device)
    for v in np.nonzero(evid >= 0)[0]:
        u[v, 1 - int(evid[v])] = 0.0
    u.requires_grad_()
    nedge = 2 * L * (L - 1)
    pair, unary = logs[:4 * nedge].exp().view(nedge, 2, 2), logs[4 * nedge:].exp().view(n, 2)
    edge, e = {}, 0
    for i in range(n):
        if i % L + 1 < L:
            edge["right", i] = e
            e += 1
        if i + L < n:
            edge["down", i] = e
            e += 1

    def row(r, v, log, pair, unary, u):
        for c in range(L):
            i = r * L + c
            w = unary[i] * u[i]
            if r == 0:
                v = v.view(-1, 1) * w
            else:
                v = torch.einsum("abc,bd->adc", v.view(2 ** c, 2, -1),
                                 pair[edge["down", i - L]] * w)
            if c:
                v = v.reshape(2 ** (c - 1), 2, 2, -1) * pair[edge["right", i - 1]][None, :, :, None]
            big = v.detach().max()
            v, log = (v / big).reshape(-1), log + big.log()
        return v, log

    v = torch.ones(1, dtype=torch.float64, device=logs.device)
    log = torch.zeros((), dtype=torch.float64, device=logs.device)
    for r in range(L):
        v, log = checkpoint(row, r, v, log, pair, unary, u, use_reentrant=False)
    logz = v.sum().log() + log
    gu, gl = torch.autograd.grad(logz, [u, logs])
    return logz.detach(), (u.detach() * gu).reshape(-1), gl


def _eliminate(m, tables, evid, query=None):
    """Bucket elimination in logarithms, 64 bits: log Z and the marginals, or,
    with a query, the largest weight of its variables after the others are summed."""
    dev = "cuda"
    free = [v for v in range(m.nvars) if evid[v] < 0]
    ones = {v: torch.zeros(int(m.card[v]), dtype=torch.float64, device=dev,
                           requires_grad=query is None) for v in free}
    ts = [([v], ones[v]) for v in free]
    const = torch.zeros((), dtype=torch.float64, device=dev)
    for s, t in zip(m.scopes, tables):
        x = torch.from_numpy(np.log(np.asarray(t))).to(dev).reshape([int(m.card[v]) for v in s])
        for d in reversed(range(len(s))):
            if evid[s[d]] >= 0:
                x = x.select(d, int(evid[s[d]]))
        ts.append(([int(v) for v in s if evid[v] < 0], x))
    asked = set() if query is None else {int(v) for v in query}
    for group in ([v for v in free if v not in asked], [v for v in free if v in asked]):
        left = set(group)
        while left:
            # the variable whose product holds the fewest entries
            near = {v: set() for v in left}
            for s, _ in ts:
                for v in s:
                    if v in near:
                        near[v].update(s)
            v = min(left, key=lambda x: (math.prod(int(m.card[y]) for y in near[x]), x))
            left.remove(v)
            union = sorted(near[v])
            total = 0.0
            for s, t in [x for x in ts if v in x[0]]:
                order = sorted(range(len(s)), key=lambda i: s[i])
                total = total + t.permute(order).reshape(
                    [int(m.card[y]) if y in s else 1 for y in union])
            d = union.index(v)
            total = total.amax(d) if v in asked else total.logsumexp(d)
            ts = [x for x in ts if v not in x[0]] + [([y for y in union if y != v], total)]
    logz = const + sum(t for _, t in ts)
    if query is not None:
        return logz.cpu(), None
    grads = dict(zip(free, torch.autograd.grad(logz, [ones[v] for v in free])))
    marg = [grads[v] if v in grads else
            torch.eye(int(m.card[v]), dtype=torch.float64, device=dev)[int(evid[v])]
            for v in range(m.nvars)]
    return logz.detach(), torch.cat(marg)
