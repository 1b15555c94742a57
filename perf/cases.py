"""Performance cases: the encrypted 1:N match and its parts, as a server runs them.

A case names a ring, a modulus chain, the form of the algorithm (which of the hoisted forms are on,
the BSGS schedule, the storage tier of the templates), a database size and a number of queries.
`prepare` makes what a server has in hand: a context with the evaluation keys resident, a loaded
database, and the clients' query ciphertexts in host memory. `run` takes one pass: the match of the
queries and the export of the result ciphertexts, the words that go back to the clients. Contexts
and their keys depend on the parameters alone and are kept between preparations, as a server keeps
them; templates and queries come from the seed. Every output is a ciphertext of whole numbers
(residues), so results are compared word for word.
"""
import math
from collections import OrderedDict

import numpy as np
import torch

from paper_2604_00546_gb300 import fr

MODES = {"scores": fr.FR_MODE_SCORES, "identify": fr.FR_MODE_IDENTIFY, "membership": fr.FR_MODE_MEMBERSHIP}
KEY_SEED = 0xC0FFEE11
MAX_CONTEXTS = 6


def _match(name, log_n, K, ell, n1, mode, *, n_q=9, q_bits=50, n_p=3, p_bits=60, dnum=3, degree=59, hoist=0, radix=0,
           schedule=0, tier=1, level_mode=1, batch=1, comparator=0):
    c = {"kind": "match", "log_n": log_n, "K": K, "ell": ell, "n1": n1, "mode": mode, "n_q": n_q, "q_bits": q_bits,
         "n_p": n_p, "p_bits": p_bits, "dnum": dnum, "degree": degree, "hoist": hoist, "radix": radix,
         "schedule": schedule, "tier": tier, "level_mode": level_mode, "batch": batch, "comparator": comparator}
    return dict(c, name=name) if name else c


def _block(kind, name, log_n, level, *, n_q=9, q_bits=50, n_p=3, p_bits=60, dnum=3, degree=59, comparator=0):
    c = {"kind": kind, "log_n": log_n, "level": level, "n_q": n_q, "q_bits": q_bits, "n_p": n_p, "p_bits": p_bits,
         "dnum": dnum, "degree": degree, "comparator": comparator}
    return dict(c, name=name) if name else c


# the headline chain: Q = 60 + 24 x 50 bits, P = 4 x 60 bits, 6 digits
CHAIN = dict(n_q=25, q_bits=50, n_p=4, p_bits=60, dnum=6)


def listed():
    return [
        # a gallery of 64 faces on the smallest ring in use: launches and host calls are what counts
        _match("tiny_scores", 12, 64, 64, 8, "scores", n_q=3, q_bits=40, n_p=3, dnum=1, degree=0, level_mode=0),
        # a site's 5000 people on a mid-size ring, two template groups, the second one ragged
        _match("mid_membership", 13, 5000, 64, 8, "membership", q_bits=45, dnum=3, level_mode=0),
        # one rotation on caller-owned device buffers (a server that must not allocate)
        _block("rotate", "rotate_n16", 16, 8),
        # the threshold alone, hybrid comparator (a counting membership), on an uploaded ciphertext
        _block("threshold", "hybrid_threshold_n16", 16, 11, n_q=13, n_p=4, dnum=5, comparator=1),
        # the paper's own form (every rotation with its own ModDown, radix-2 slot sum)
        _match("membership_plain_n16", 16, 1 << 15, 512, 32, "membership"),
        # the headline: one membership query against 2^15 templates, every hoisted form on
        _match("membership_n16", 16, 1 << 15, 512, 32, "membership", hoist=1, radix=8, **CHAIN),
        # the same without dropping the query to a working level: key switching over 25 + 4 limbs
        _match("full_chain_n16", 16, 1 << 15, 512, 32, "membership", hoist=1, radix=8, level_mode=0, **CHAIN),
        # eight clients' queries in one pass
        _match("batch8_n16", 16, 1 << 15, 512, 32, "membership", hoist=1, radix=8, batch=8, **CHAIN),
        # identification against a database too large to keep encoded: diagonals encoded per query
        _match("identify_encode_n16", 16, 100000, 512, 32, "identify", hoist=1, radix=8, tier=2, **CHAIN),
        # identification on a smaller ring, three ragged groups, diagonals kept as integer coefficients
        _match("identify_coeffs_n15", 15, 40001, 256, 16, "identify", hoist=0, tier=3),
        # the rotated-query table schedule (Algorithm 1), five ragged groups sharing one table
        _match("table_scores_n14", 14, 40000, 128, 16, "scores", n_q=4, schedule=1, degree=0),
        # the paper's encrypted database: ciphertext x ciphertext products, lazily relinearised
        _match("encrypted_db_n15", 15, 16000, 128, 16, "membership", tier=4),
    ]


def _dnum(n_q):
    """Digits of at most 3 limbs, so that the 180 bits of P cover a digit."""
    return -(-n_q // 3)


def draw(rng):
    kind = rng.choice(["match"] * 6 + ["rotate", "threshold"])
    log_n = rng.choice([12, 13, 14, 15, 16])
    q_bits = rng.choice([40, 45, 50, 50])
    if kind == "rotate":
        n_q = rng.randint(3, 9)
        return _block(kind, None, log_n, rng.randint(1, n_q - 1), n_q=n_q, q_bits=q_bits, dnum=_dnum(n_q))
    if kind == "threshold":
        comparator = rng.choice([0, 1])
        degree = rng.choice([27, 59])
        depth = (5 if degree == 27 else 6) + 4 * comparator
        level = depth + rng.randint(0, 2)
        return _block(kind, None, log_n, level, n_q=level + 1, q_bits=q_bits, n_p=rng.choice([3, 4]),
                      dnum=_dnum(level + 1), degree=degree, comparator=comparator)
    ell = rng.choice([e for e in (64, 128, 256, 512) if log_n >= 14 or e <= 128])
    n1 = rng.choice([n for n in (4, 8, 12, 16, 32) if n * n <= 2 * ell])
    mode = rng.choice(["scores", "identify", "membership"])
    degree = 0 if mode == "scores" else rng.choice([27, 59, 59])
    depth = {0: 0, 27: 5, 59: 6}[degree]
    n_q = 3 + depth + rng.choice([0, 0, 1, 2])
    n = 1 << (log_n - 1)
    form = rng.choice(["plain", "hoisted", "hoisted", "table", "encrypted"])
    tier = 4 if form == "encrypted" else rng.choice([1, 1, 1, 2, 3])
    groups = 1 if form == "encrypted" else rng.choice([1, 1, 2, 3])
    K = int(round(math.exp(rng.uniform(math.log(n // 16), math.log(n * groups)))))
    batch = rng.choice([1, 1, 2, 3, 5]) if form != "table" and groups == 1 and tier == 1 else 1
    if form in ("table", "encrypted"):
        ell, n1 = min(ell, 128), min(n1, 16)
    return _match(None, log_n, K, ell, n1, mode, n_q=n_q, q_bits=q_bits, dnum=_dnum(n_q), degree=degree,
                  hoist=1 if form == "hoisted" else 0, radix=rng.choice([4, 8]) if form == "hoisted" else 0,
                  schedule=1 if form == "table" else 0, tier=tier, level_mode=1, batch=batch)


_contexts = OrderedDict()


def _context(case):
    """(context with its evaluation keys resident, the client's keys) of the case's parameters."""
    match = case["kind"] == "match"
    key = tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "K", "tier", "batch")))
    if key in _contexts:
        _contexts.move_to_end(key)
        return _contexts[key]
    while len(_contexts) >= MAX_CONTEXTS:
        _contexts.popitem(last=False)[1][0].close()
    hoist = case.get("hoist", 0)
    ctx = fr.Context(device=torch.cuda.current_device(), log_n=case["log_n"],
                     q_bits=[60] + [case["q_bits"]] * (case["n_q"] - 1), p_bits=[case["p_bits"]] * case["n_p"],
                     dnum=case["dnum"], scale_bits=case["q_bits"], ell=case["ell"] if match else 64,
                     n1=case["n1"] if match else 8, cheb_degree=case["degree"], threshold=0.5,
                     schedule=case.get("schedule", 0), level_mode=case.get("level_mode", 0),
                     sum_radix=case.get("radix", 0), hoist_giants=hoist, hoist_babies=hoist, hoist_sum=hoist,
                     comparator=case["comparator"])
    if match:
        rotations = ctx.required_rotations(MODES[case["mode"]])
    else:
        rotations = [5] if case["kind"] == "rotate" else []
    ctx.load_keys(ctx.keygen(rotations, KEY_SEED))
    _contexts[key] = ctx, ctx.keygen([], KEY_SEED)
    return _contexts[key]


def _faces(case, seed):
    """(templates float32 [K, ell], queries float64 [batch, ell]), L2-normalised rows; every query
    is a noisy view of an enrolled face."""
    K, ell = case["K"], case["ell"]
    g = torch.Generator(device="cuda").manual_seed(seed * 7919 + 17)
    T = torch.randn(K, ell, device="cuda", generator=g)
    T /= T.norm(dim=1, keepdim=True)
    at = torch.randint(0, K, (case["batch"],), device="cuda", generator=g)
    q = T[at].double() + 0.6 / math.sqrt(ell) * torch.randn(case["batch"], ell, device="cuda", generator=g).double()
    q /= q.norm(dim=1, keepdim=True)
    return T.cpu().numpy(), q.cpu().numpy()


def prepare(case, seed):
    ctx, keys = _context(case)
    if case["kind"] == "rotate":
        limbs, N = case["level"] + 1, 1 << case["log_n"]
        g = torch.Generator(device="cuda").manual_seed(seed * 7919 + 17)
        ct = torch.empty(2, limbs, N, dtype=torch.int64, device="cuda")
        for i, q in enumerate(ctx.primes()[:limbs]):
            ct[:, i] = torch.randint(0, q, (2, N), device="cuda", generator=g)
        out = torch.empty_like(ct)
        torch.cuda.synchronize()
        return {"case": case, "ctx": ctx, "ct": ct, "out": out}
    if case["kind"] == "threshold":
        z = np.random.default_rng(seed).uniform(-1.0, 1.0, ctx.n)
        return {"case": case, "ctx": ctx, "ct": ctx.encrypt_slots(keys, z, seed).upload()}
    T, q = _faces(case, seed)
    if case["tier"] == 4:
        db = ctx.load_db_encrypted(ctx.encrypt_db(keys, T, seed=seed), len(T))
    else:
        db = ctx.load_db(T, tier=case["tier"])
    queries = [ctx.encrypt(keys, v, seed * 64 + b) for b, v in enumerate(q)]
    return {"case": case, "ctx": ctx, "db": db, "queries": queries}


def run(state):
    case, ctx = state["case"], state["ctx"]
    if case["kind"] == "rotate":
        ctx.rotate_noalloc(state["ct"].data_ptr(), case["level"], 5, state["out"].data_ptr())
        return state["out"]
    if case["kind"] == "threshold":
        return ctx.chebyshev(state["ct"]).export().view(np.int64)
    mode = MODES[case["mode"]]
    if case["batch"] == 1:
        outs = ctx.match(state["db"], state["queries"][0], mode)
    else:
        outs = [o for per in ctx.match_batch(state["db"], state["queries"], mode) for o in per]
    return [o.export().view(np.int64) for o in outs]


def exact(case, seed):
    """No output of any case is a rounded number: all are residues, compared word for word."""
    return None


def work(case):
    """Bytes one pass cannot do without: the keys it switches with, the database in the form it is
    kept, the queries in and the results out, each once."""
    N = 1 << case["log_n"]
    limb = 8 * N
    if case["kind"] != "match":
        level = case["level"]
        key = _digits(case, level) * 2 * (level + 1 + case["n_p"]) * limb
        depth = 0
        if case["kind"] == "threshold":
            depth = {27: 5, 59: 6}[case["degree"]] + 4 * case["comparator"]
        return {"bytes": key + 2 * (level + 1) * limb + 2 * (level + 1 - depth) * limb, "flops": 0}
    depth = {0: 0, 27: 5, 59: 6}[case["degree"]]
    top = case["n_q"] - 1
    L = min(top, 2 + depth) if case["level_mode"] else top
    G = -(-case["K"] // (N // 2))
    ell, n1 = case["ell"], case["n1"]
    n2 = -(-ell // n1)
    limbs = L + 1 + (case["n_p"] if case["hoist"] and not case["schedule"] else 0)
    rotations = (n1 - 1) + (n2 - 1)
    if case["mode"] == "membership":
        r, s = max(2, case["radix"]), 1
        while s < N // 2:
            rotations += min(r, N // 2 // s) - 1
            s *= r
    keys = (rotations + (1 if depth else 0)) * _digits(case, L) * 2 * (L + 1 + case["n_p"]) * limb
    db = {1: G * ell * limbs * limb, 2: 4 * case["K"] * ell, 3: G * ell * limb, 4: G * ell * 2 * (L + 1) * limb}
    lo = L - 1 - depth
    outs = case["batch"] * (1 if case["mode"] == "membership" else G)
    return {"bytes": keys + db[case["tier"]] + case["batch"] * 2 * (L + 1) * limb + outs * 2 * (lo + 1) * limb,
            "flops": 0}


def _digits(case, level):
    """Key-switching digits that hold a limb of 0..level: n_q limbs in dnum digits, the remainder
    spread one limb at a time over the last ones."""
    n_d = min(case["dnum"], case["n_q"])
    base, extra = divmod(case["n_q"], n_d)
    lo, used = 0, 0
    for d in range(n_d):
        used += lo <= level
        lo += base + (1 if d >= n_d - extra else 0)
    return used
