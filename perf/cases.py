"""The work a user of this library has it do, as cases that can be timed and compared.

Every case goes through the package's public calls (``join_inner``, ``join_batch``,
``sort``, ``sort_multi``, ``gather_pairs``) on device-resident columns, with row
positions as ids, as the benchmark and the serving loop use them:

* joins: foreign-key pairs (R unique, S drawn Zipf over R's keys; dense or spread
  over 64 bits), uniform keys in twice |R| values, and log-normal clusters on 40 bits
  with duplicates on both sides; with and without a memory budget;
* many small joins in one batch;
* ORDER BY one column (dense or full-range keys) and several columns;
* gathering payload columns through a join's pairs.

Joins write into a buffer of |S| pairs that the program keeps (at most |S| pairs come
out in these workloads).  ``sort`` and ``sort_multi`` work in place; a pass sorts a copy, so that the base
relation stays as it is and every pass sorts unsorted rows.
"""
import math

import numpy as np
import torch

from paper_2602_21237_gb300 import api, datagen

MIB = 1 << 20
DEV = "cuda"


def listed():
    return [
        # the smallest served request: a lookup of 3x10^4 facts in a 10^4-row dimension
        {"name": "join_small", "op": "join", "keys": "fk", "n_r": 10_000, "n_s": 30_000,
         "zipf": 1.0, "bits": 64, "budget": 0},
        # the paper's size: 10^6 x 10^6 with 32-bit keys
        {"name": "join_1e6_int32", "op": "join", "keys": "uniform", "n_r": 1_000_000,
         "n_s": 1_000_000, "zipf": 0.0, "bits": 32, "budget": 0},
        # an ordinary fact-to-dimension join
        {"name": "join_1e7", "op": "join", "keys": "fk", "n_r": 10_000_000,
         "n_s": 40_000_000, "zipf": 0.8, "bits": 64, "budget": 0},
        # the headline join under its memory budget
        {"name": "join_1e8_budget", "op": "join", "keys": "fk", "n_r": 100_000_000,
         "n_s": 400_000_000, "zipf": 0.8, "bits": 64, "budget": 256 * MIB},
        # the same relations, strongly skewed, without a budget
        {"name": "join_1e8_skewed", "op": "join", "keys": "fk", "n_r": 100_000_000,
         "n_s": 400_000_000, "zipf": 1.2, "bits": 64, "budget": 0},
        # clustered keys on 40 bits, duplicates on both sides, ragged sizes
        {"name": "join_clustered", "op": "join", "keys": "lognormal", "n_r": (1 << 26) + 7,
         "n_s": (1 << 26) - 13, "zipf": 0.0, "bits": 64, "budget": 0},
        # many independent joins of 10^3 to 10^6 rows at once
        {"name": "join_batch", "op": "batch", "jobs": 1024, "lo": 1_000, "hi": 1_000_000,
         "bits": 32},
        # ORDER BY on the paper's 10^6 rows, 32-bit keys
        {"name": "sort_1e6_int32", "op": "sort", "keys": "uniform", "n": 1_000_000, "bits": 32},
        # ORDER BY a dense 64-bit key column of 10^8 rows
        {"name": "sort_1e8", "op": "sort", "keys": "dense", "n": 100_000_000, "bits": 64},
        # ORDER BY a hashed (full-range) 64-bit column, ragged size
        {"name": "sort_hashed", "op": "sort", "keys": "scattered", "n": 30_000_001, "bits": 64},
        # ORDER BY three columns (20 + 30 + 10 bits)
        {"name": "sort_three_keys", "op": "sort_multi", "n": 10_000_000, "b0": 20, "b1": 30,
         "b2": 10, "bits": 64},
        # two payload columns of each side through a foreign-key join's pairs
        {"name": "gather_payload", "op": "gather", "n_r": 10_000_000, "n_s": 40_000_000,
         "zipf": 0.8, "bits": 64},
    ]


def _size(rng, lo, hi):
    """Log-uniform in [lo, hi], odd as often as even."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["join", "join", "join", "join", "sort", "sort", "sort_multi", "gather",
                     "batch"])
    bits = rng.choice([32, 64])
    if op == "join":
        keys = rng.choice(["fk", "fk", "uniform", "scattered", "lognormal"])
        if keys in ("scattered", "lognormal"):  # 64-bit values
            bits = 64
        top_r, top_s = {"fk": (100_000_000, 400_000_000), "uniform": (60_000_000, 60_000_000),
                        "scattered": (20_000_000, 80_000_000),
                        "lognormal": (1 << 26, 1 << 26)}[keys]
        n_r, n_s = _size(rng, 1_000, top_r), _size(rng, 1_000, top_s)
        zipf = round(rng.uniform(0.0, 1.2), 2) if keys in ("fk", "scattered") else 0.0
        budget = 256 * MIB if keys == "fk" and rng.random() < 0.5 else 0
        return {"op": op, "keys": keys, "n_r": n_r, "n_s": n_s, "zipf": zipf, "bits": bits,
                "budget": budget}
    if op == "batch":
        return {"op": op, "jobs": _size(rng, 16, 1024), "lo": 1_000,
                "hi": _size(rng, 10_000, 1_000_000), "bits": bits}
    if op == "sort":
        keys = rng.choice(["dense", "uniform"] if bits == 32 else ["dense", "uniform", "scattered"])
        return {"op": op, "keys": keys, "n": _size(rng, 1_000, 100_000_000), "bits": bits}
    if op == "sort_multi":
        b = [rng.randint(4, 10), rng.randint(4, 12), rng.randint(4, 9)] if bits == 32 else \
            [rng.randint(8, 30), rng.randint(8, 30), rng.randint(4, 24)]
        return {"op": op, "n": _size(rng, 10_000, 20_000_000), "b0": b[0], "b1": b[1],
                "b2": b[2], "bits": bits}
    return {"op": op, "n_r": _size(rng, 1_000, 20_000_000), "n_s": _size(rng, 1_000, 40_000_000),
            "zipf": round(rng.uniform(0.0, 1.2), 2), "bits": bits}


def _dtype(case):
    return torch.int32 if case["bits"] == 32 else torch.int64


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _zipf_ranks(n, m, s, g):
    """n ranks in [0, m), P(rank) ~ (rank + 1)^-s: the inverse CDF of the bounded power law
    (element by element, so that a seed always gives the same ranks)."""
    if s == 0.0:
        return torch.randint(0, m, (n,), generator=g, device=DEV)
    ranks = torch.empty(n, dtype=torch.int64, device=DEV)
    for a in range(0, n, 1 << 26):
        u = torch.rand(min(n - a, 1 << 26), generator=g, device=DEV, dtype=torch.float64)
        x = torch.pow(m + 1.0, u) if s == 1.0 else \
            torch.pow(((m + 1.0) ** (1.0 - s) - 1.0) * u + 1.0, 1.0 / (1.0 - s))
        ranks[a:a + u.numel()] = (x - 1.0).to(torch.int64).clamp_(0, m - 1)
    return ranks


def _fk_pair(case, seed, dt):
    """R's keys unique in random order, S's keys drawn from them; ids are row positions."""
    g, n_r, n_s = _gen(seed), case["n_r"], case["n_s"]
    kr = torch.randperm(n_r, generator=g, device=DEV)
    if case.get("keys") == "scattered":
        kr = datagen.scatter64(kr)
    of_rank = torch.randperm(n_r, generator=g, device=DEV)
    ks = kr[of_rank[_zipf_ranks(n_s, n_r, case["zipf"], g)]]
    return (kr.to(dt), torch.arange(n_r, device=DEV, dtype=dt), ks.to(dt),
            torch.arange(n_s, device=DEV, dtype=dt))


def prepare(case, seed):
    dt, op = _dtype(case), case["op"]
    if op == "batch":
        off_r, off_s, *cols = datagen.batch_jobs(case["jobs"], case["lo"], case["hi"], seed, DEV,
                                                 dt)
        # about half a pair per S row comes out: room for three times the mean of that
        room = int(1.5 * case["jobs"] * _mean_rows(case)) + case["hi"]
        return {"op": op, "off_r": off_r, "off_s": off_s, "cols": cols,
                "out": torch.zeros((room, 2), dtype=dt, device=DEV)}
    if op == "join":
        if case["keys"] == "uniform":
            cols = datagen.uniform_pair(case["n_r"], case["n_s"], 0, 2 * case["n_r"], seed, dt,
                                        DEV)
        elif case["keys"] == "lognormal":
            cols = (*datagen.lognormal_mix(case["n_r"], seed, DEV),
                    *datagen.lognormal_mix(case["n_s"], seed + 500_009, DEV))
        else:
            cols = _fk_pair(case, seed, dt)
        return {"op": op, "cols": cols, "budget": case["budget"],
                "out": torch.zeros((case["n_s"], 2), dtype=dt, device=DEV)}
    if op == "gather":
        cols = _fk_pair(case, seed, dt)
        g = _gen(seed + 1)
        wide = torch.float64 if dt == torch.int64 else torch.float32
        return {"op": op, "pairs": api.join_inner(*cols),
                "r_cols": [torch.randint(-1000, 1000, (case["n_r"],), generator=g, device=DEV,
                                         dtype=dt),
                           torch.rand(case["n_r"], generator=g, device=DEV, dtype=wide)],
                "s_cols": [torch.randint(0, 1 << 20, (case["n_s"],), generator=g, device=DEV,
                                         dtype=dt),
                           torch.rand(case["n_s"], generator=g, device=DEV, dtype=torch.float32)]}
    g, n = _gen(seed), case["n"]
    ids = torch.arange(n, device=DEV, dtype=dt)
    if op == "sort_multi":
        cols = [torch.randint(0, 1 << case[b], (n,), generator=g, device=DEV, dtype=dt)
                for b in ("b0", "b1", "b2")]
        return {"op": op, "cols": cols, "ids": ids}
    if case["keys"] == "uniform":  # any non-negative 32-bit value, duplicates among them
        keys = torch.randint(0, (1 << 31) - 1, (n,), generator=g, device=DEV, dtype=dt)
    else:
        keys = torch.randperm(n, generator=g, device=DEV, dtype=torch.int64)
        keys = datagen.scatter64(keys + seed) if case["keys"] == "scattered" else keys.to(dt)
    return {"op": op, "keys": keys, "ids": ids}


def run(state):
    op = state["op"]
    if op == "join":
        pairs = api.join_inner(*state["cols"], mem_budget_bytes=state["budget"],
                               out=state["out"])
        return {"out": state["out"], "count": pairs.shape[0]}
    if op == "batch":
        pairs, out_off = api.join_batch(state["off_r"], state["off_s"], *state["cols"],
                                        out=state["out"])
        return {"out": state["out"], "count": pairs.shape[0], "out_off": out_off}
    if op == "sort":
        return api.sort(state["keys"].clone(), state["ids"].clone())
    if op == "sort_multi":
        return api.sort_multi([c.clone() for c in state["cols"]], state["ids"].clone())
    return api.gather_pairs(state["pairs"], state["r_cols"], state["s_cols"])


def _mean_rows(case):
    """Mean of a log-uniform size in [lo, hi]."""
    return (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])


def _lognormal_pairs(n_r, n_s):
    """Expected |J| of two log-normal mixtures: n_r n_s times the integral of the squared
    key density (8 clusters and 5% uniform on 40 bits), on a grid of log2(key)."""
    u = np.linspace(16.0, 40.0, 24_001)
    x = np.exp2(u)
    f = np.full_like(x, 0.05 / 2.0 ** 40)
    for c in range(8):
        m, s = math.log(2.0 ** (24 + 2 * c)), 0.3 + 0.05 * c
        f += 0.95 / 8 * np.exp(-0.5 * ((np.log(x) - m) / s) ** 2) / (x * s * math.sqrt(2 * math.pi))
    return n_r * n_s * float(np.sum(f * f * x) * math.log(2.0) * (u[1] - u[0]))


def work(case):
    """Each input column read once, each output column written once (no arithmetic)."""
    w, op = case["bits"] // 8, case["op"]
    if op == "join":
        n_r, n_s = case["n_r"], case["n_s"]
        pairs = {"uniform": n_s / 2, "lognormal": _lognormal_pairs(n_r, n_s)}.get(case["keys"], n_s)
        return {"bytes": 2 * w * (n_r + n_s + pairs), "flops": 0}
    if op == "batch":
        return {"bytes": 2 * w * case["jobs"] * _mean_rows(case) * 2.5, "flops": 0}
    if op == "sort":
        return {"bytes": 4 * w * case["n"], "flops": 0}
    if op == "sort_multi":
        return {"bytes": 8 * w * case["n"], "flops": 0}
    per_r, per_s = (16 if w == 8 else 8), w + 4
    return {"bytes": case["n_s"] * (2 * w + per_r + 2 * per_s) +
            min(case["n_r"], case["n_s"]) * per_r, "flops": 0}


def exact(case, seed):
    """Joins and sorts give whole numbers, which are the same or wrong; gathered payload
    columns are copies, which plain indexing gives."""
    if case["op"] != "gather":
        return None
    s = prepare(case, seed)
    rows = s["pairs"].to(torch.int64)
    return tuple([c[rows[:, side]].double() if c.is_floating_point() else None for c in cols]
                 for side, cols in enumerate((s["r_cols"], s["s_cols"])))
