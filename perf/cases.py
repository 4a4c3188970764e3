"""The work that users of this decoder have it do, as cases that can be timed
and checked through the package's public entry points.

A case is a dict of plain values.  Kinds:

  decode   ``Graph.decode`` of one batch of syndromes that lies on the GPU
  multi    ``decode_multi``: batches of several codes and error rates in one call
  host     ``decode_host``: syndromes and results in page-locked host memory
  serve    ``serving.Server``: a queue of requests of two codes, host to host
  train    one step of weighted-BP training: ``wbp.weighted_bp``, its loss and
           the gradient of the weights
  sample   ``Graph.sample``: seeded errors, syndromes and observables

The codes are the ones the repository studies: bivariate-bicycle codes, the
hypergraph product code of 2500 bits, the phenomenological and circuit-level
detector models and rotated surface codes, with the error rates, iteration
limits and request sizes of its benchmark and tests.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import bpdc_inputs as bi
import paper_2510_08695_gb300 as pkg
from bpdc_inputs import circuit
from paper_2510_08695_gb300 import serving, wbp

RATES_BB = [0.01, 0.02, 0.03, 0.04, 0.05, 0.06, 0.07, 0.08, 0.09, 0.10]
RATES_PHEN = [0.002, 0.004, 0.006, 0.008, 0.010]
RATES_SURFACE = [0.01, 0.03, 0.05, 0.06, 0.08]
RATES_CIRCUIT = [0.0005, 0.001, 0.002]

# mean BP iterations of a shot (both runs), a property of the code, the rate
# and the iteration limit; only the estimate of the arithmetic in work() uses it
MEAN_ITERATIONS = {
    "bb72": (RATES_BB, [0.71, 2.11, 4.82, 9.28, 15.6, 23.2, 31.4, 39.9, 47.8, 54.7]),
    "bb108": (RATES_BB, [0.83, 1.90, 4.12, 8.66, 16.5, 27.3, 40.0, 53.3, 65.4, 75.6]),
    "bb144": (RATES_BB, [0.98, 2.12, 4.27, 8.66, 16.4, 28.0, 42.2, 56.9, 70.2, 80.7]),
    "hgp2500": (RATES_BB, [4.89, 14.2, 28.6, 48.6, 71.2, 89.7, 98.5, 99.9, 100.0, 100.0]),
    "phen_bb144": (RATES_PHEN, [1.43, 3.81, 10.7, 22.2, 40.8]),
    "phen_bb72": (RATES_PHEN, [0.86, 1.31, 1.84, 2.70, 3.99]),
    "surface3": (RATES_SURFACE, [0.45, 1.27, 1.98, 2.29, 2.84]),
    "surface5": (RATES_SURFACE, [2.26, 6.42, 10.1, 11.7, 14.5]),
    "surface7": (RATES_SURFACE, [6.30, 18.0, 27.4, 31.4, 38.3]),
    "surface9": (RATES_SURFACE, [13.7, 37.9, 56.0, 63.0, 74.4]),
    "circuit_bb72": (RATES_CIRCUIT, [55.5, 118.0, 239.0]),
    "circuit_bb144": (RATES_CIRCUIT, [213.0, 396.0, 700.0]),
}
# arithmetic of one edge in one iteration: min-sum takes a sign, two minima, a
# choice, a scaling and three additions; product-sum two evaluations of
# log tanh with their sums; the adjoint of product-sum as much again twice
OPS_MIN_SUM, OPS_PRODUCT_SUM, OPS_ADJOINT = 8, 40, 120


@functools.lru_cache(maxsize=None)
def problem(code: str, p: float):
    """The decoding problem of a code at error rate p."""
    if code.startswith("circuit_"):
        name = code[len("circuit_"):]
        return circuit.circuit_level_problem(name, 6 if name == "bb72" else 12, p)
    if code.startswith("phen_"):
        name = code[len("phen_"):]
        return bi.phenomenological_bb_problem(name, 6 if name == "bb72" else 12, p)
    if code.startswith("surface"):
        return bi.surface_problem(int(code[len("surface"):]), p)
    if code == "hgp2500":
        return bi.hgp_problem(p)
    return bi.bb_problem(code, p)


def options(code: str, soft: bool = False):
    """Decoder options the repository uses for a family of codes."""
    if code.startswith("surface"):   # product-sum, second run on the posterior, T = n
        d = int(code[len("surface"):])
        return pkg.Options(variant=1, max_iter=d * d, dc_prior=1)
    if code.startswith("circuit_") or code == "phen_bb144":
        return pkg.Options(max_iter=1000)
    if code == "phen_bb72":
        return pkg.Options(max_iter=100)
    return pkg.Options(max_iter=50, dc_enable=0 if soft else 1)


def listed():
    return [
        # a real-time request of a small code: launch and latency
        dict(name="request_bb72", kind="decode", code="bb72", p=0.05, shots=64, soft=False, persistent=True),
        # a short request of the large circuit-level model: few shots, many
        # iterations, most of the GPU without work
        dict(name="request_circuit_bb144", kind="decode", code="circuit_bb144", p=0.001, shots=40, soft=False,
             persistent=True),
        # logical-error-rate points of Monte Carlo studies, one code at a time
        dict(name="batch_bb144", kind="decode", code="bb144", p=0.04, shots=1000000, soft=False, persistent=True),
        dict(name="batch_hgp2500", kind="decode", code="hgp2500", p=0.06, shots=30001, soft=False, persistent=True),
        dict(name="batch_phen_bb144", kind="decode", code="phen_bb144", p=0.006, shots=100001, soft=False,
             persistent=True),
        # product-sum decoding of a surface code, the second rule of the library
        dict(name="batch_surface7", kind="decode", code="surface7", p=0.05, shots=100003, soft=False,
             persistent=True),
        # posterior LLRs of plain BP, for a post-processor of the user's own
        dict(name="soft_bb108", kind="decode", code="bb108", p=0.03, shots=50021, soft=True, persistent=True),
        # the benchmark's workload, smaller: uneven codes and rates in one call
        dict(name="mixed_codes", kind="multi", codes="bb144,bb72,hgp2500", rates="0.01,0.04,0.07,0.1", shots=20011),
        # a decoder fed by the host
        dict(name="host_bb72", kind="host", code="bb72", p=0.05, shots=500009),
        # the decode server under a queue of uneven requests
        dict(name="serve_mixed", kind="serve", codes="circuit_bb144,bb72", rates="0.001,0.05", requests=16,
             most=1024),
        # one step of weight training (20 unrolled iterations: the gradient of many
        # more grows without bound on shots that do not converge)
        dict(name="train_bb144", kind="train", code="bb144", p=0.06, T=20, batch=4096, ckpt=5),
        # inputs of a Monte Carlo study
        dict(name="sample_bb144", kind="sample", code="bb144", p=0.05, shots=1000000, errors=True),
    ]


def _spread(rng, lo: int, hi: int) -> int:
    """A whole number in [lo, hi], even over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# most shots of a drawn batch (each below the largest listed case)
MOST = {"bb72": 1000000, "bb108": 1000000, "bb144": 1000000, "hgp2500": 30000, "phen_bb144": 100000,
        "phen_bb72": 100000, "surface3": 100000, "surface5": 100000, "surface7": 100000, "surface9": 100000,
        "circuit_bb72": 1024, "circuit_bb144": 1024}


def draw(rng):
    kind = rng.choice(["decode", "decode", "decode", "decode", "soft", "multi", "host", "serve", "train", "sample"])
    if kind == "decode":
        code = rng.choice(sorted(MOST))
        return dict(kind="decode", code=code, p=rng.choice(MEAN_ITERATIONS[code][0]), shots=_spread(rng, 1, MOST[code]),
                    soft=False, persistent=rng.random() < 0.8)
    if kind == "soft":
        code = rng.choice(["bb72", "bb108", "bb144"])
        return dict(kind="decode", code=code, p=rng.choice([0.02, 0.03, 0.04]), shots=_spread(rng, 100, 60000),
                    soft=True, persistent=True)
    if kind == "multi":
        codes = rng.sample(["bb144", "bb108", "bb72", "hgp2500", "phen_bb72"], rng.randint(2, 3))
        rates = rng.sample([0.01, 0.02, 0.04, 0.06, 0.08, 0.1], rng.randint(1, 4))
        return dict(kind="multi", codes=",".join(codes), rates=",".join("%g" % p for p in rates),
                    shots=_spread(rng, 500, 20000))
    if kind == "host":
        code = rng.choice(["bb72", "bb108", "bb144"])
        return dict(kind="host", code=code, p=rng.choice(RATES_BB[:6]), shots=_spread(rng, 1000, 500000))
    if kind == "serve":
        first = rng.choice(["circuit_bb144", "circuit_bb72", "bb144"])
        rates = "%g,%g" % (0.05 if first == "bb144" else 0.001, rng.choice([0.03, 0.05, 0.08]))
        return dict(kind="serve", codes=first + ",bb72", rates=rates, requests=rng.randint(2, 16),
                    most=_spread(rng, 16, 1024))
    if kind == "train":
        return dict(kind="train", code=rng.choice(["bb72", "bb108", "bb144"]), p=rng.choice([0.04, 0.05, 0.06]),
                    T=rng.randint(5, 20), batch=_spread(rng, 32, 4096), ckpt=rng.choice([3, 5]))
    code = rng.choice(sorted(MOST))
    return dict(kind="sample", code=code, p=rng.choice(MEAN_ITERATIONS[code][0]),
                shots=_spread(rng, 100, 1000000 if code.startswith("bb") else 100000), errors=rng.random() < 0.5)


def _graph(code, p, soft=False):
    return pkg.Graph.from_problem(problem(code, p), options(code, soft))


def _pairs(case):
    codes, rates = case["codes"].split(","), [float(x) for x in case["rates"].split(",")]
    return codes, rates


def _multi_points(case):
    codes, rates = _pairs(case)
    # the phenomenological model's rates are a tenth of the code-capacity ones
    return [(c, p / 10 if c.startswith("phen") else p) for c in codes for p in rates]


def _request_sizes(case):
    """Sizes of the requests, uneven in [1, most], the codes in turn."""
    r = np.random.RandomState(case["requests"] * 4099 + case["most"])
    return [int(x) for x in r.randint(1, case["most"] + 1, size=case["requests"])]


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case, offset=seed % 1000 * 1000003)
    if kind == "decode":
        s["graph"] = _graph(case["code"], case["p"], case["soft"])
        s["syn"], s["obs"], _ = s["graph"].sample(case["shots"], seed, s["offset"])
    elif kind == "multi":
        s["items"] = []
        for i, (code, p) in enumerate(_multi_points(case)):
            g = _graph(code, p)
            n = case["shots"] + 7 * i   # uneven batches
            syn, obs, _ = g.sample(n, seed + i, s["offset"])
            s["items"].append(dict(graph=g, syndromes=syn, obs_true=obs, shot_offset=s["offset"],
                                   out=g.alloc_outputs(n)))
    elif kind == "host":
        g = _graph(case["code"], case["p"])
        syn, obs, _ = g.sample(case["shots"], seed, s["offset"])
        s["items"] = [dict(graph=g, syndromes=syn.cpu().pin_memory(), obs_true=obs.cpu().pin_memory(),
                           shot_offset=s["offset"], out=g.alloc_host_outputs(case["shots"]))]
    elif kind == "serve":
        codes, rates = _pairs(case)
        graphs = [_graph(c, p) for c, p in zip(codes, rates)]
        s["server"] = serving.Server(graphs, slots=8, max_shots=1024)
        s["requests"] = []
        for i, n in enumerate(_request_sizes(case)):
            gid = i % len(graphs)
            syn = graphs[gid].sample(n, seed + i, s["offset"])[0].cpu().pin_memory()
            s["requests"].append((gid, syn, s["offset"]))
    elif kind == "train":
        g = pkg.Graph.from_problem(problem(case["code"], case["p"]), pkg.Options(variant=1, max_iter=case["T"]))
        syn, _, err = g.sample(case["batch"], seed, s["offset"], errors=True)
        s.update(graph=g, syn=syn, errors=wbp.unpack_words(err, g.N), weights=_weights(case, seed, g.E))
        s["weights"].requires_grad_(True)
    else:
        s.update(graph=_graph(case["code"], case["p"]), seed=seed)
    return s


def _weights(case, seed, E):
    """Weights some steps into a training run: near 1."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return 1.0 + 0.05 * torch.randn((2, case["T"], E), generator=gen, device="cuda")


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "decode":
        g = state["graph"]
        if case["soft"]:
            return g.decode(state["syn"], state["offset"], posterior=True, persistent=case["persistent"])
        if case["shots"] <= 1024:   # a request
            return g.decode(state["syn"], state["offset"], persistent=case["persistent"])
        counters = torch.zeros(4, dtype=torch.int64, device="cuda")
        out = g.decode(state["syn"], state["offset"], obs_true=state["obs"], counters=counters,
                       persistent=case["persistent"])
        return dict(out, counters=counters)
    if kind == "multi":
        counters = torch.zeros((len(state["items"]), 4), dtype=torch.int64, device="cuda")
        pkg.decode_multi([dict(it, counters=counters[i]) for i, it in enumerate(state["items"])])
        return dict(counters=counters, outs=[it["out"] for it in state["items"]])
    if kind == "host":
        pkg.decode_host(state["items"])
        return state["items"][0]["out"]
    if kind == "serve":
        server = state["server"]
        server.completed.clear()
        reqs = [serving.Request(gid, syn, off, 0.0, i) for i, (gid, syn, off) in enumerate(state["requests"])]
        for r in reqs:
            server.submit(r)
        while len(server.completed) < len(reqs):
            server.step()
        return [r.result for r in reqs]
    if kind == "train":
        w = state["weights"]
        w.grad = None
        post = wbp.weighted_bp(w, state["graph"], state["syn"], 20.0, case["ckpt"])
        loss = wbp.bce_loss(post, state["errors"])
        loss.backward()
        return dict(loss=loss.detach(), posteriors=post.detach(), grad=w.grad)
    syn, obs, err = state["graph"].sample(case["shots"], state["seed"], state["offset"], errors=case["errors"])
    return dict(syndromes=syn, observables=obs, errors=err)


def _decode_work(code, p, shots, soft=False):
    P = problem(code, p)
    words = sum((n + 31) // 32 for n in (P.M, P.N, P.K))
    ops = OPS_PRODUCT_SUM if code.startswith("surface") else OPS_MIN_SUM
    rates, mean = MEAN_ITERATIONS[code]
    iters = float(np.interp(p, rates, mean))
    return shots * (4 * words + 5 + (4 * P.N if soft else 0)), shots * iters * P.E * ops


def work(case):
    kind = case["kind"]
    if kind in ("decode", "host"):
        parts = [_decode_work(case["code"], case["p"], case["shots"], case.get("soft", False))]
    elif kind == "multi":
        parts = [_decode_work(c, p, case["shots"] + 7 * i) for i, (c, p) in enumerate(_multi_points(case))]
    elif kind == "serve":
        codes, rates = _pairs(case)
        parts = [_decode_work(codes[i % 2], rates[i % 2], n) for i, n in enumerate(_request_sizes(case))]
    elif kind == "train":
        P, T, B = problem(case["code"], case["p"]), case["T"], case["batch"]
        # posteriors out, errors and syndromes in, weights in and their gradient out
        parts = [(4 * (B * T * P.N + B * P.N + B * ((P.M + 31) // 32) + 4 * T * P.E),
                  B * T * P.E * (OPS_PRODUCT_SUM + OPS_ADJOINT))]
    else:
        P = problem(case["code"], case["p"])
        words = sum((n + 31) // 32 for n in ((P.M, P.N, P.K) if case["errors"] else (P.M, P.K)))
        parts = [(4 * case["shots"] * words, case["shots"] * P.N * 20)]   # one 64-bit hash per column
    return dict(bytes=sum(b for b, _ in parts), flops=sum(f for _, f in parts))


# ---- the same numbers in 64 bits, by plain torch --------------------------------

def _tanner(P):
    """Edges in row order: their check and column, and the edges of every check
    and of every column (padded with nnz)."""
    H = P.H.tocsr()
    row = np.repeat(np.arange(P.M), np.diff(H.indptr))
    col = H.indices.astype(np.int64)

    def members(of, n):
        groups = [np.nonzero(of == i)[0] for i in range(n)]
        pad = np.full((n, max(1, max(len(x) for x in groups))), len(of), dtype=np.int64)
        for i, x in enumerate(groups):
            pad[i, :len(x)] = x
        return torch.from_numpy(pad).cuda()

    return (torch.from_numpy(row).cuda(), torch.from_numpy(col).cuda(), members(row, P.M), members(col, P.N))


def _bits(words, n):
    """Bit words [B, ceil(n/32)] to booleans [B, n]."""
    w = words.to(torch.int64) & 0xFFFFFFFF
    return ((w[:, :, None] >> torch.arange(32, device=w.device)) & 1).reshape(w.shape[0], -1)[:, :n].bool()


def _exact_soft(case, state):
    """Posterior LLRs of normalized min-sum BP (scale 5/8, at most 50
    iterations, stopping when the decision reproduces the syndrome)."""
    P = problem(case["code"], case["p"])
    row, col, of_row, of_col = _tanner(P)
    syn = _bits(state["syn"], P.M)
    B, E = syn.shape[0], row.numel()
    lam = torch.from_numpy(np.log((1 - P.priors) / P.priors)).cuda()
    post = lam.expand(B, P.N).clone()
    q = lam[col].expand(B, E).clone()
    todo = syn.any(1).nonzero()[:, 0]
    for _ in range(50):
        if todo.numel() == 0:
            break
        qa = torch.cat([q[todo].abs(), torch.full((todo.numel(), 1), math.inf, dtype=q.dtype, device="cuda")], 1)
        neg = torch.cat([q[todo] < 0, torch.zeros((todo.numel(), 1), dtype=torch.bool, device="cuda")], 1)
        two, arg = torch.topk(qa[:, of_row], 2, dim=2, largest=False)
        least = two[:, row, 0]
        where = of_row[torch.arange(P.M, device="cuda")[None], arg[:, :, 0]][:, row]
        other = torch.where(where == torch.arange(E, device="cuda")[None], two[:, row, 1], least)
        flip = (neg[:, of_row].sum(2) % 2 == 1) ^ syn[todo]
        r = 0.625 * torch.where(flip[:, row] ^ neg[:, :E], -other, other)
        r0 = torch.cat([r, torch.zeros((todo.numel(), 1), dtype=r.dtype, device="cuda")], 1)
        L = lam + r0[:, of_col].sum(2)
        post[todo] = L
        q[todo] = L[:, col] - r
        e = torch.cat([L <= 0, torch.zeros((todo.numel(), 1), dtype=torch.bool, device="cuda")], 1)
        colp = torch.cat([col, torch.tensor([P.N], device="cuda")])
        todo = todo[((e[:, colp[of_row]].sum(2) % 2 == 1) != syn[todo]).any(1)]
    return post


def _exact_train(case, state):
    """Unrolled weighted product-sum BP and the gradient of the mean binary
    cross-entropy of its posteriors."""
    P = problem(case["code"], case["p"])
    row, col, of_row, of_col = _tanner(P)
    E, T = row.numel(), case["T"]
    lam = torch.from_numpy(np.log((1 - P.priors) / P.priors)).cuda()
    w = state["weights"].detach().double().requires_grad_(True)
    s = torch.where(_bits(state["syn"], P.M), -1.0, 1.0).double()
    B = s.shape[0]
    # the other edges of every edge's check and column
    def others(table, of):
        t = table[of]
        return torch.where(t == torch.arange(E, device="cuda")[:, None], E, t)
    chk, var = others(of_row, row), others(of_col, col)
    zero, one = torch.zeros((B, 1), dtype=torch.float64, device="cuda"), torch.ones((B, 1), dtype=torch.float64, device="cuda")
    phi = lambda x: -torch.log(torch.tanh(x / 2))  # noqa: E731
    r = torch.zeros((B, E), dtype=torch.float64, device="cuda")
    post = []
    for t in range(T):
        q = (w[1, t] * (lam[col] + torch.cat([r, zero], 1)[:, var].sum(2))).clamp(-20.0, 20.0)
        f = phi(q.abs().clamp_min(1e-6))
        sign = torch.cat([torch.where(q < 0, -one, one), one], 1)[:, chk].prod(2) * s[:, row]
        r = w[0, t] * sign * phi(torch.cat([f, zero], 1)[:, chk].sum(2))
        post.append(lam + torch.cat([r, zero], 1)[:, of_col].sum(2))
    post = torch.stack(post, 1)
    e = state["errors"].double()[:, None, :]
    loss = (e * torch.nn.functional.softplus(post) + (1 - e) * torch.nn.functional.softplus(-post)).mean()
    loss.backward()
    return dict(loss=loss.detach(), posteriors=post.detach(), grad=w.grad)


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, prepare(case, seed))
    if case["kind"] == "decode" and case["soft"]:
        post = _exact_soft(case, prepare(case, seed))
        return dict(corrections=None, status=None, logical_flips=None, iterations=None, posterior_llr=post)
    return None   # every other output is a whole number
