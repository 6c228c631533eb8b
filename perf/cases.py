"""The work users of this framework have it do, as measurable cases.

A server owner loads an item set and evaluates encrypted requests against it
(`Context.eval`, `Context.eval_batch`, `Engine`); a client encrypts its items
(`Context.query`) and decrypts the response (`Context.decrypt`); both sides'
programs also use the ring operations by themselves (`Context.ntt`,
`Context.ct_mult`).  Contexts, loaded sets, engines and response buffers are
kept between calls, as such programs keep them; requests are what arrives.

Sizes are the configurations of `paper_2310_14565_gb300/workload.py`, of
`bench.py` and of the tests: rings of 4096, 8192 and 16384, three to eight
ciphertext primes of 36 to 55 bits, Hamming weights 2, 4 and 8, sets of 2^10
to 2^20 items.  Every output is whole numbers (ciphertext residues, slots)
except the noise budget of a decryption.
"""
import math

import numpy as np
import torch

import paper_2310_14565_gb300 as pepsi
from paper_2310_14565_gb300.workload import make_sets

T = 65537
HASH_KEY = 0x5EED
P3 = "36,36,37"
P4 = "55,55,54,54"
P4X = "51,51,51,51"
P8 = "55,55,55,55,55,55,54,54"
RINGS = {4096: (P3,), 8192: (P4, P4X), 16384: (P8,)}
# (Hamming weight, effective item bits): the code length follows (Eq. 1)
CODES = {4096: ((2, 16), (4, 16)), 8192: ((2, 16), (4, 32), (8, 40), (8, 19)), 16384: ((4, 32), (8, 40))}
MODES = {"indicator": pepsi.MODE_INDICATOR, "cardinality": pepsi.MODE_CARDINALITY, "labels": pepsi.MODE_LABELS,
         "sum": pepsi.MODE_SUM}


def _eval(**kw):
    """An evaluation case: the defaults of a context unless said otherwise."""
    case = dict(op="eval", N=8192, primes=P4, h=4, lam=32, ell=0, mu=0, m=1024, n=1 << 16, bits=64, rescale="layer",
                resp=0, mode="indicator", table_bytes=8, resident=True, host=False, requests=1, share=0, chunk=0)
    case.update(kw)
    return case


def listed():
    return [
        # a client reads its response: one ciphertext at one prime, from host memory (the smallest call)
        dict(name="decrypt", op="decrypt", N=8192, primes=P4, resp=1),
        # the NTT of one whole request, the ring operation the benchmark quotes against memory bandwidth
        dict(name="ntt_request", op="ntt", N=8192, primes=P4, count=1200, inverse=False),
        # ciphertext products with relinearisation at the benchmark's batch
        dict(name="ct_mult_256", op="ct_mult", N=8192, primes=P4, count=256, relin=True),
        # a client encrypts 1024 items for the paper-shaped code
        dict(name="query_1024", op="query", N=8192, primes=P4, h=4, lam=32, ell=600, m=1024, bits=64),
        # the toy configuration: a small set, where launches and latency count
        _eval(name="eval_toy", N=4096, primes=P3, h=2, lam=16, ell=363, mu=16, m=64, n=1024, bits=32),
        # a set of 2^16 items with a context's default rounding (per layer) and full response, a masked cardinality
        _eval(name="eval_2^16_h2", h=2, lam=16, ell=363, mu=74, n=1 << 16, mode="cardinality"),
        # labelled PSI: values per item, one rounding per evaluation, an odd set size
        _eval(name="eval_labels", h=4, lam=32, ell=600, n=50001, m=777, rescale="all", resp=1, mode="labels"),
        # the paper's own headline parameters (h = 8, 51-bit primes, 32-bit items), request and response in pinned
        # host memory
        _eval(name="eval_host_h8", primes=P4X, h=8, lam=19, ell=24, mu=526, n=1 << 20, bits=32, rescale="all", resp=1,
              host=True),
        # the large ring with plaintexts regenerated at evaluation, as for tables that do not fit in memory
        _eval(name="eval_regenerated", N=16384, primes=P8, h=8, lam=40, ell=128, mu=100, n=1 << 18, rescale="all",
              resp=1, resident=False),
        # four requests on one set in one call, sharing the plaintext reads
        _eval(name="batch_4", h=4, lam=32, ell=600, n=1 << 18, rescale="all", resp=1, requests=4, share=4, chunk=256),
        # a server of two resident sets on two rings, six requests in flight
        dict(name="engine_mixed", op="engine", n0=1 << 16, n1=1 << 16, requests=6),
        # the paper-shaped evaluation: 1024 client items against 2^20, one rounding, a one-prime response
        _eval(name="eval_paper", h=4, lam=32, ell=600, mu=526, n=1 << 20, rescale="all", resp=1, chunk=256),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["eval", "eval", "eval", "eval", "batch", "regenerated", "engine", "query", "ntt", "ntt", "ct_mult",
                     "decrypt"])
    N = rng.choice(sorted(RINGS))
    primes = rng.choice(RINGS[N])
    h, lam = rng.choice(CODES[N])
    if op == "decrypt":
        return dict(op="decrypt", N=N, primes=primes, resp=rng.randint(1, primes.count(",") + 1))
    if op == "ntt":
        return dict(op="ntt", N=N, primes=primes, count=_log_uniform(rng, 1, 1500), inverse=rng.random() < 0.5)
    if op == "ct_mult":
        return dict(op="ct_mult", N=N, primes=primes, count=_log_uniform(rng, 1, 256), relin=rng.random() < 0.7)
    if op == "query":
        return dict(op="query", N=N, primes=primes, h=h, lam=lam, ell=0, m=_log_uniform(rng, 16, N // 2), bits=64)
    if op == "engine":
        return dict(op="engine", n0=_log_uniform(rng, 1 << 10, 1 << 17), n1=_log_uniform(rng, 1 << 10, 1 << 16),
                    requests=rng.randint(2, 9))
    case = _eval(N=N, primes=primes, h=h, lam=lam, m=_log_uniform(rng, 16, 4096), n=_log_uniform(rng, 1 << 10, 1 << 18),
                 rescale=rng.choice(["layer", "all", "all", "16"]), resp=rng.choice([0, 1]))
    if N == 16384:
        case["n"] = min(case["n"], 1 << 17)
    if N == 4096:
        case["m"] = min(case["m"], N // 2)
    if op == "batch":
        case["requests"] = rng.randint(2, 6)
        case["share"] = rng.choice([0, 3, 4])
        case["mode"] = rng.choice(["indicator", "cardinality"])
    elif op == "regenerated":
        case["resident"] = False
        case["n"] = min(case["n"], 1 << 16)
    else:
        case["mode"] = rng.choice(["indicator", "indicator", "cardinality", "labels", "sum"])
        case["host"] = rng.random() < 0.3
        case["table_bytes"] = rng.choice([8, 8, 7])
        case["chunk"] = rng.choice([0, 0, 256])
    return case


# ------------------------------------------------------------------ state
def _bits(case):
    return [int(b) for b in case["primes"].split(",")]


def _context(case, seed, **kw):
    return pepsi.Context(N=case["N"], t=T, prime_bits=_bits(case), hash_key=HASH_KEY, key_seed=seed, **kw)


def _residues(ctx, count, gen):
    """count polynomials [count][k][N] of uniform residues, on the GPU."""
    out = torch.empty((count, ctx.k, ctx.N), dtype=torch.int64, device="cuda")
    for i, q in enumerate(ctx.q):
        out[:, i] = torch.randint(0, q, (count, ctx.N), generator=gen, device="cuda", dtype=torch.int64)
    return out


def _request(ctx, items, seed):
    cts = torch.empty((ctx.ell, 2, ctx.k, ctx.N), dtype=torch.int64, device="cuda")
    ctx.query(items, seed, out=cts)
    return cts


def _server(case, seed, lanes=0):
    """Context, set id and requests of an evaluation case."""
    group = {"layer": 0, "all": pepsi.RESCALE_ALL, "16": 16}[case["rescale"]]
    valued = case["mode"] in ("labels", "sum")
    ctx = _context(case, seed, h=case["h"], ell=case["ell"], lambda_bar=case["lam"], mu=case["mu"],
                   resident_bytes=_resident(case), rescale_group=group, server_values=int(valued),
                   response_primes=case["resp"], plaintext_bytes=case["table_bytes"])
    if case["chunk"] or case["share"]:
        ctx.set_schedule(chunk=case["chunk"] or None, batch_requests=case["share"] or None,
                         batch_groups=1 if case["share"] else None)
    m, n = case["m"], case["n"]
    reqs = []
    for r in range(case["requests"]):
        sets = make_sets(m, n, min(m, n) // 10, bits=case["bits"], seed_items=seed, seed_plant=seed + 1 + r)
        if r == 0:
            if valued:
                vals = np.random.default_rng(seed).integers(0, T, size=n).astype(np.uint32)
                sid = ctx.server_load_values(sets.server, vals)
            else:
                sid = ctx.server_load(sets.server)
        reqs.append(_request(ctx, sets.client, seed + 2 + r))
    return ctx, sid, reqs


def _resident(case):
    """The resident-plaintext budget: none, or the whole table (its size is known to the program that loads it)."""
    return (1 << 64) - 1 if not case["resident"] else 100 << 30


def _response(ctx):
    return torch.zeros((2, ctx.response_primes, ctx.N), dtype=torch.int64, device="cuda")


def prepare(case, seed):
    op = case["op"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    s = {"op": op, "case": case, "seed": seed}
    if op == "ntt":
        s["ctx"] = _context(case, seed)
        s["polys"] = _residues(s["ctx"], case["count"], gen)
    elif op == "ct_mult":
        s["ctx"] = ctx = _context(case, seed)
        n = case["count"]
        s["a"] = _residues(ctx, 2 * n, gen)
        s["b"] = _residues(ctx, 2 * n, gen)
        s["out"] = torch.zeros((n, 2 if case["relin"] else 3, ctx.k, ctx.N), dtype=torch.int64, device="cuda")
    elif op == "query":
        s["ctx"] = ctx = _context(case, seed, h=case["h"], ell=case["ell"], lambda_bar=case["lam"])
        s["items"] = make_sets(case["m"], 16, 0, bits=case["bits"], seed_items=seed, seed_plant=seed + 1).client
        s["out"] = torch.zeros((ctx.ell, 2, ctx.k, ctx.N), dtype=torch.int64, device="cuda")
    elif op == "decrypt":
        c = _eval(N=case["N"], primes=case["primes"], h=2, lam=16, m=256, n=1024, resp=case["resp"])
        s["ctx"], sid, reqs = _server(c, seed)
        s["ct"] = s["ctx"].eval(sid, reqs[0])  # the response as the client receives it, in host memory
    elif op == "engine":
        a = _eval(h=2, lam=16, n=case["n0"], rescale="all", resp=1, requests=case["requests"] - case["requests"] // 2)
        b = _eval(N=16384, primes=P8, h=8, lam=40, n=case["n1"], rescale="all", resp=1,
                  requests=case["requests"] // 2)
        s["lanes"] = [_server(a, seed), _server(b, seed + 100)]
        s["engine"] = pepsi.Engine([(ctx, sid, 4) for ctx, sid, _ in s["lanes"]])
        s["outs"] = [[_response(ctx) for _ in reqs] for ctx, _, reqs in s["lanes"]]
    else:
        s["ctx"], s["sid"], s["reqs"] = _server(case, seed)
        s["outs"] = [_response(s["ctx"]) for _ in s["reqs"]]
        if case["host"]:
            s["reqs"] = [r.cpu().pin_memory() for r in s["reqs"]]
            s["outs"] = [o.cpu().pin_memory() for o in s["outs"]]
    torch.cuda.synchronize()
    return s


def run(s):
    op, case = s["op"], s["case"]
    if op == "ntt":
        s["ctx"].ntt(s["polys"], case["count"], inverse=case["inverse"])  # in place: each pass transforms the last one's
        return s["polys"]
    if op == "ct_mult":
        s["ctx"].ct_mult(s["a"], s["b"], case["count"], s["out"], relin=case["relin"])
        return s["out"]
    if op == "query":
        _, where = s["ctx"].query(s["items"], s["seed"], out=s["out"])
        return s["out"], where
    if op == "decrypt":
        return s["ctx"].decrypt(s["ct"])
    if op == "engine":
        eng, tickets = s["engine"], []
        for lane, (_, _, reqs) in enumerate(s["lanes"]):
            for r, (cts, out) in enumerate(zip(reqs, s["outs"][lane])):
                mode = MODES["cardinality"] if r & 1 else MODES["indicator"]
                tickets.append(eng.submit(lane, cts, out=out, mode=mode, mask_seed=r)[0])
        eng.run()
        for t in tickets:
            eng.wait(t)
        return s["outs"]
    mode = MODES[case["mode"]]
    if case["requests"] > 1:
        n = case["requests"]
        return s["ctx"].eval_batch([s["sid"]] * n, s["reqs"], modes=[mode] * n, mask_seeds=list(range(n)),
                                   outs=s["outs"])
    return s["ctx"].eval(s["sid"], s["reqs"][0], mode=mode, mask_seed=7, out=s["outs"][0])


# ------------------------------------------------------------------- work
def _code_length(case):
    """Eq. 1: the smallest code length with C(ell, h) >= 2^lam, unless given."""
    ell = case["ell"] or case["h"]
    while not case["ell"] and math.comb(ell, case["h"]) < 1 << case["lam"]:
        ell += 1
    return ell


def _layers(case):
    """Layers of the server table: given, or the loads of the fullest of N bins under 3 n throws (mean + tail)."""
    mean = 3.0 * case["n"] / case["N"]
    return case["mu"] or int(mean + 8 * math.sqrt(mean) + 8)


def _base(bits, N):
    """Residues of the second base an exact product needs beside the ciphertext primes (61-bit words)."""
    return math.ceil((math.log2(T * N) + sum(bits) + 3) / 61)


def _ntt_flops(N, rows):
    return 5.0 * rows * (N // 2) * math.log2(N)  # per butterfly: a modular product and two sums


def _mult_rows(k, kb, relin):
    return 2 * k + 2 * kb + 3 * (k + kb) + (k * (k + 2) + 2 * k if relin else 0)


def _eval_work(case, shared=1):
    bits, N = _bits(case), case["N"]
    k, kb, ell, mu = len(bits), _base(bits, case["N"]), _code_length(case), _layers(case)
    q_bytes = sum(bits) / 8.0
    table = mu * ell * N * q_bytes if case["resident"] else mu * N * case["h"] * 2.0
    per = ell * 2 * N * q_bytes + 2 * (case["resp"] or k) * N * 8.0
    flops = mu * ell * k * N * 4.0 * case["requests"]
    products = {1: 0, 2: 1, 4: 2, 8: 3}[case["h"]]
    flops += case["requests"] * mu * products * _ntt_flops(N, _mult_rows(k, kb, True))
    if not case["resident"]:
        flops += mu * ell * _ntt_flops(N, k + 1)
    return {"bytes": table + case["requests"] * per, "flops": flops}


def work(case):
    op = case["op"]
    if op == "engine":
        a = _eval(h=2, lam=16, n=case["n0"], resp=1, requests=case["requests"] - case["requests"] // 2)
        b = _eval(N=16384, primes=P8, h=8, lam=40, n=case["n1"], resp=1, requests=case["requests"] // 2)
        wa, wb = _eval_work(a), _eval_work(b)
        return {key: wa[key] + wb[key] for key in wa}
    if op == "eval":
        return _eval_work(case)
    bits, N = _bits(case), case["N"]
    k, kb = len(bits), _base(bits, case["N"])
    if op == "ntt":
        return {"bytes": 16.0 * case["count"] * k * N, "flops": _ntt_flops(N, case["count"] * k)}
    if op == "ct_mult":
        rows = _mult_rows(k, kb, case["relin"])
        return {"bytes": case["count"] * k * N * 8.0 * (4 + (2 if case["relin"] else 3)),
                "flops": case["count"] * _ntt_flops(N, rows)}
    if op == "query":
        ell = _code_length(case)
        return {"bytes": ell * 2 * k * N * 8.0, "flops": _ntt_flops(N, ell * (2 * k + 1))}
    return {"bytes": 2 * case["resp"] * N * 8.0 + 4.0 * N, "flops": _ntt_flops(N, 2 * case["resp"] + 1)}


def exact(case, seed):
    """Outputs are residues, slots and table positions: whole numbers, equal or wrong.  The one computed number, a
    decryption's noise budget, is a property of the ciphertext's hidden noise that only the library's keys give."""
    return None
