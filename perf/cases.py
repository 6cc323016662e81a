"""The performance cases: what users of the library have it do, through its
public Python entry points, over the range of sizes it serves.

A case is a dict of plain values; ``listed()`` gives the fixed ones,
``draw(rng)`` one more of the same ranges, ``prepare(case, seed)`` what a
program holds before the call, ``run(state)`` one call, ``work(case)`` the
bytes and operations one call cannot do without, and ``exact(case, seed)`` the
64-bit reference of a computed (floating-point) output.

Exact counts have no input but (variant, n) and the moduli, so the seed picks
the moduli (the caller's option ``primes``), and the residues are returned
beside the count.
"""
import random

import numpy as np

import paper_1507_00315_gb300 as sk

HIDDEN = 256
VARIANT = {"skolem": 0, "langford": 1, "hooked": 2}
SYMMETRY = {"negation": sk.SYMMETRY_NEGATION, "reversal": sk.SYMMETRY_REVERSAL,
            "reversal_even": sk.SYMMETRY_REVERSAL_EVEN}


def listed():
    return [
        # the smallest counts: a script that tabulates S(n), L(n) for small n
        # calls them one by one, and waits for each (launch latency)
        {"name": "count_s8", "kind": "count", "variant": "skolem", "n": 8, "symmetry": "negation"},
        # a mid-size count of the third variant (2^35 terms)
        {"name": "count_h18", "kind": "count", "variant": "hooked", "n": 18, "symmetry": "negation"},
        # the headline workload's largest job: S(20), 2^39 terms
        {"name": "count_s20", "kind": "count", "variant": "skolem", "n": 20, "symmetry": "negation"},
        # what a user in a hurry asks for: every symmetry of the paper
        {"name": "count_l19_sym", "kind": "count", "variant": "langford", "n": 19,
         "symmetry": "reversal_even"},
        # the independent cross-check by inclusion-exclusion (2^32 terms)
        {"name": "ie_s16", "kind": "ie", "variant": "skolem", "n": 16},
        # the uneven sweep: three variants, n = 4..16, one call
        {"name": "batch_4_16", "kind": "batch", "n_lo": 4, "n_hi": 16, "variants": 3},
        # one part of a sharded S(24): a range of wide work items, residues of each
        {"name": "items_s24", "kind": "items", "variant": "skolem", "n": 24, "m": 18,
         "count": 16384},
        # an approximate count with the defaults: ladder tuned by pilots, then
        # 4096 ladders of 32 rungs
        {"name": "estimate_s20", "kind": "estimate", "variant": "skolem", "n": 20, "rungs": 32,
         "ladders": 4096, "budget": 20000},
        # the long ladders of the large orders: 64 rungs, final configurations
        # kept (training data)
        {"name": "run_l32_64", "kind": "pt_run", "variant": "langford", "n": 32, "rungs": 64,
         "ladders": 4096, "iters": 3000},
        # tempering with the network's proposals, 32 x 4096 chains
        {"name": "learned_s20", "kind": "learned", "variant": "skolem", "n": 20, "rungs": 32,
         "ladders": 4096, "iters": 100},
        # training the network: 16 minibatches of 4096 states
        {"name": "train_s20", "kind": "train", "variant": "skolem", "n": 20, "batch": 4096,
         "steps": 16},
        # the network's logits of a ragged batch of host states
        {"name": "forward_l24", "kind": "forward", "variant": "langford", "n": 24, "batch": 5000},
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["count", "count", "sym", "ie", "batch", "items", "estimate", "pt_run",
                       "learned", "train", "forward"])
    two = rng.choice(["skolem", "langford"])
    three = rng.choice(["skolem", "langford", "hooked"])
    if kind == "count":
        return {"kind": "count", "variant": three, "n": rng.randint(4, 19), "symmetry": "negation"}
    if kind == "sym":
        return {"kind": "count", "variant": two, "n": rng.randint(6, 20),
                "symmetry": rng.choice(["reversal", "reversal_even"])}
    if kind == "ie":
        return {"kind": "ie", "variant": three, "n": rng.randint(4, 18)}
    if kind == "batch":
        hi = rng.randint(7, 17)
        return {"kind": "batch", "n_lo": rng.randint(3, hi - 2), "n_hi": hi,
                "variants": rng.randint(1, 3)}
    if kind == "items":
        n = rng.randint(14, 28)
        m = rng.randint(8, 14)              # every order takes these widths
        return {"kind": "items", "variant": three, "n": n, "m": m,
                "count": _log(rng, 100, min(32768, 1 << (2 * n - 2 - m)))}
    if kind == "estimate":
        return {"kind": "estimate", "variant": two, "n": rng.randint(8, 33),
                "rungs": rng.randint(8, 32), "ladders": _log(rng, 64, 4096),
                "budget": _log(rng, 500, 20000)}
    if kind == "pt_run":
        return {"kind": "pt_run", "variant": two, "n": rng.randint(16, 64),
                "rungs": rng.randint(20, 64), "ladders": _log(rng, 64, 4096),
                "iters": _log(rng, 200, 3000)}
    if kind == "learned":
        return {"kind": "learned", "variant": two, "n": rng.randint(8, 33),
                "rungs": rng.randint(8, 32), "ladders": _log(rng, 32, 4096),
                "iters": _log(rng, 10, 100)}
    if kind == "train":
        return {"kind": "train", "variant": two, "n": rng.randint(8, 33),
                "batch": 128 * _log(rng, 2, 64), "steps": rng.randint(2, 16)}
    return {"kind": "forward", "variant": two, "n": rng.randint(8, 33),
            "batch": _log(rng, 1, 8192)}


# ---------------------------------------------------------------- inputs

def _is_prime(p):
    if p % 2 == 0:
        return p == 2
    d, r = p - 1, 0
    while d % 2 == 0:
        d //= 2
        r += 1
    for a in (2, 3, 5, 7, 11, 13, 17, 19, 23, 29, 31, 37):
        x = pow(a, d, p)
        if x in (1, p - 1):
            continue
        for _ in range(r - 1):
            x = x * x % p
            if x == p - 1:
                break
        else:
            return False
    return True


def _moduli(seed):
    """Three distinct primes in the library's window (2^62 - 2^31, 2^62)."""
    rng = random.Random(seed)
    out = []
    while len(out) < 3:
        p = (1 << 62) - 2 * rng.randrange(1, 1 << 30) + 1
        while not _is_prime(p):
            p -= 2
        if p > (1 << 62) - (1 << 31) and p not in out:
            out.append(p)
    return out


def _distance(case):
    return [k + (1 if case["variant"] == "langford" else 0) for k in range(1, case["n"] + 1)]


def _slots(rng, case, count):
    """Start slots of random states: half uniform, half annealed a little (each
    pair's best of four draws against a common occupancy), as chains hold."""
    n, dist = case["n"], _distance(case)
    out = np.zeros((count, n), dtype=np.uint8)
    occ = np.zeros((count, 2 * n), dtype=np.int32)
    rows = np.arange(count)
    picky = rng.random(count) < 0.5
    for k in range(n - 1, -1, -1):
        width = 2 * n - dist[k]
        best, load = None, None
        for _ in range(4):
            s = rng.integers(0, width, count)
            c = occ[rows, s] + occ[rows, s + dist[k]]
            if best is None:
                best, load = s, c
            else:
                take = picky & (c < load)
                best, load = np.where(take, s, best), np.where(take, c, load)
        out[:, k] = best
        np.add.at(occ, (rows, best), 1)
        np.add.at(occ, (rows, best + dist[k]), 1)
    return out


def _network(rng, case):
    """Parameters of a proposal network as training leaves it: the first layer
    sees each bin empty or crowded, the logits favour moves into empty bins;
    every weight has some noise.  Values are exact in bf16 (they are kept so)."""
    n, dist = case["n"], _distance(case)
    w1 = 0.02 * rng.standard_normal((2 * n, HIDDEN))
    b1 = 0.02 * rng.standard_normal(HIDDEN)
    w2 = 0.01 * rng.standard_normal((HIDDEN, HIDDEN))
    b2 = 0.02 * rng.standard_normal(HIDDEN)
    nm = sum(2 * n - d for d in dist)
    w3 = 0.02 * rng.standard_normal((HIDDEN, nm))
    b3 = 0.02 * rng.standard_normal(nm)
    for b in range(2 * n):
        w1[b, b] -= 1.0                      # unit b: 1 on an empty bin
        b1[b] += 1.0
        w2[b, b] += 1.0
    m = 0
    for k in range(n):
        for s in range(2 * n - dist[k]):
            w3[s, m] += 2.0
            w3[s + dist[k], m] += 2.0
            m += 1
    flat = np.concatenate([a.ravel() for a in (w1, b1, w2, b2, w3, b3)]).astype(np.float32)
    return (flat.view(np.uint32) & np.uint32(0xFFFF0000)).view(np.float32)


def _ladder(rungs, top):
    x = np.linspace(0.0, 1.0, rungs)
    return top * (np.exp(3.0 * x) - 1.0) / (np.exp(3.0) - 1.0)


def prepare(case, seed):
    kind, rng = case["kind"], np.random.default_rng(seed)
    st = {"case": case, "seed": int(seed)}
    if kind in ("count", "ie", "batch", "items"):
        st["primes"] = _moduli(seed)
    if kind == "batch":
        jobs = [(v, n) for v in range(case["variants"])
                for n in range(case["n_lo"], case["n_hi"] + 1)]
        random.Random(seed).shuffle(jobs)            # a user's list, in any order
        st["jobs"] = jobs
    if kind == "items":
        items = 1 << (2 * case["n"] - 1 - case["m"])
        st["q_lo"] = random.Random(seed).randrange(items - case["count"] + 1)
    if kind in ("pt_run", "learned"):
        st["beta"] = _ladder(case["rungs"], 12.0)
    if kind in ("learned", "train", "forward"):
        rows = case["ladders"] * case["rungs"] if kind == "learned" else case["batch"]
        model = sk.Mlp(VARIANT[case["variant"]], case["n"], (rows + 127) // 128 * 128, seed=seed)
        model.set_params(_network(rng, case))
        st["model"] = model
    if kind == "train":
        st["states"] = _slots(rng, case, case["batch"] * case["steps"])
    if kind == "forward":
        st["states"] = _slots(rng, case, case["batch"])
    return st


# ---------------------------------------------------------------- the call

def _residues(rep):
    """A sum's residues and the moduli they belong to."""
    return {k: np.array(rep[k][:3], dtype=np.int64) for k in ("residues", "primes")}


def run(st):
    case, kind, seed = st["case"], st["case"]["kind"], st["seed"]
    if kind == "count":
        c, rep = sk.count_ex(case["variant"], case["n"], primes=st["primes"],
                             symmetry=SYMMETRY[case["symmetry"]])
        return {"count": c, **_residues(rep)}
    if kind == "ie":
        c, rep = sk.count_inclusion_exclusion(case["variant"], case["n"], primes=st["primes"])
        return {"count": c, **_residues(rep)}
    if kind == "batch":
        counts, statuses, _ = sk.count_batch(st["jobs"], primes=st["primes"])
        return {"counts": np.array(counts, dtype=np.int64),
                "statuses": np.array(statuses, dtype=np.int64)}
    if kind == "items":
        r = sk.item_residues(case["variant"], case["n"], case["m"], st["q_lo"], case["count"],
                             st["primes"])
        return np.array(r, dtype=np.int64)
    if kind == "estimate":
        est, rep = sk.pt_estimate(case["variant"], case["n"], case["budget"], rungs=case["rungs"],
                                  ladders=case["ladders"], seed=seed)
        return {"estimate": est, "rel_stderr": rep["rel_stderr"],
                **{k: np.array(rep[k], dtype=np.float64)
                   for k in ("beta", "ratio", "acc_move", "acc_swap")}}
    if kind == "pt_run":
        r = sk.pt_run(case["variant"], case["n"], st["beta"], case["ladders"], case["iters"],
                      case["iters"] // 10, seed, want_final=True)
        return {"hist": r["hist"].astype(np.int64), "acc_move": r["acc_move"].astype(np.int64),
                "acc_swap": r["acc_swap"].astype(np.int64), "final_slots": r["final_slots"]}
    if kind == "learned":
        r = sk.pt_run(case["variant"], case["n"], st["beta"], case["ladders"], case["iters"],
                      case["iters"] // 10, seed, model=st["model"])
        return {k: r[k].astype(np.int64) for k in ("hist", "acc_move", "acc_swap")}
    if kind == "train":
        loss, _ = st["model"].train(st["states"], epochs=1, batch=case["batch"], lr=1e-3,
                                    beta_star=2.0, seed=seed)
        return {"loss": loss, "params": st["model"].get_params()}
    return st["model"].forward(st["states"])


# ---------------------------------------------------------------- floors

def _layers(case):
    n = case["n"]
    nm = sum(2 * n - d for d in _distance(case))
    return 2 * n * HIDDEN + HIDDEN * HIDDEN + HIDDEN * nm, nm


def work(case):
    """Bytes and operations of one call: host inputs and outputs once; one
    operation per assignment of an exact sum (its signed addition); the random
    block (10 rounds of 2 wide products and 4 logic operations) of a tempering
    move; 2 M N K of the network's products."""
    kind, n = case["kind"], case["n"] if "n" in case else 0
    if kind == "count":
        cut = {"negation": 1, "reversal": 2, "reversal_even": 4}[case["symmetry"]]
        return {"bytes": 64, "flops": 2.0 ** (2 * n - 1) / cut}
    if kind == "ie":
        return {"bytes": 64, "flops": 2.0 ** (2 * n)}
    if kind == "batch":
        terms = sum(2.0 ** (2 * k - 1) for k in range(case["n_lo"], case["n_hi"] + 1))
        jobs = case["variants"] * (case["n_hi"] - case["n_lo"] + 1)
        return {"bytes": 32 * jobs, "flops": case["variants"] * terms}
    if kind == "items":
        return {"bytes": 24 * case["count"], "flops": case["count"] * 2.0 ** case["m"]}
    if kind in ("estimate", "pt_run"):
        moves = float(case["rungs"]) * case["ladders"] * case.get("budget", case.get("iters"))
        out = 8 * case["rungs"] * (2 * n + 3)
        if kind == "pt_run":
            out += case["rungs"] * case["ladders"] * n
        return {"bytes": out, "flops": 60 * moves}
    mac, nm = _layers(case)
    if kind == "learned":
        rows = float(case["rungs"]) * case["ladders"]
        # each iteration's logits written once and read once (bf16)
        return {"bytes": case["iters"] * rows * nm * 4, "flops": 2 * mac * rows * case["iters"]}
    if kind == "train":
        rows = float(case["batch"]) * case["steps"]
        return {"bytes": rows * n + case["steps"] * 28 * mac, "flops": 6 * mac * rows}
    return {"bytes": case["batch"] * (n + 4 * nm) + 4 * mac, "flops": 2 * mac * case["batch"]}


def exact(case, seed):
    """The network's logits in 64 bits.  Counts, residues and histograms are
    whole numbers, and a tempering run or a training run has no closed form."""
    if case["kind"] != "forward":
        return None
    rng = np.random.default_rng(seed)
    p = _network(rng, case).astype(np.float64)
    slots = _slots(rng, case, case["batch"])
    n, dist = case["n"], _distance(case)
    nm = sum(2 * n - d for d in dist)
    rows = np.arange(case["batch"])
    x = np.zeros((case["batch"], 2 * n))
    for k in range(n):
        np.add.at(x, (rows, slots[:, k].astype(int)), 1.0)
        np.add.at(x, (rows, slots[:, k].astype(int) + dist[k]), 1.0)
    at = 0

    def take(*shape):
        nonlocal at
        size = int(np.prod(shape))
        a = p[at:at + size].reshape(shape)
        at += size
        return a

    w1, b1 = take(2 * n, HIDDEN), take(HIDDEN)
    w2, b2 = take(HIDDEN, HIDDEN), take(HIDDEN)
    w3, b3 = take(HIDDEN, nm), take(nm)
    h = np.maximum(x @ w1 + b1, 0.0)
    h = np.maximum(h @ w2 + b2, 0.0)
    return h @ w3 + b3
