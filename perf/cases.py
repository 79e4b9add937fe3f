"""The work users have this engine do, as cases that can be timed: query
batches, sampled and exhaustive sweeps into a histogram, and batches of many
triangulations, each through the package's public entry points.

A case is a dict of plain values: "kind" and "d" (or a range of degrees), the
number of sign vectors and the options of the call.  Triangulations are the
seeded regular ones of tcurve_inputs; the sign vectors, the sweep's first mask
and (but for batches, which a program plans once) the triangulation come from
the seed.
"""
import functools

import numpy as np
import torch

import paper_2604_09221_gb300 as ts
import tcurve_inputs as ti

FLAGS = {"plain": 0, "flip": ts.TS_ENUM_FLIP, "reduced": ts.TS_ENUM_REDUCED,
         "orbits": ts.TS_ENUM_ORBITS}
LARGEST = 1 << 30  # masks of the largest sweep


def listed():
    return [
        # every sign vector of a quartic in one call: the smallest exhaustive
        # query, where launches and host work count
        {"name": "query_d4_all", "kind": "query", "d": 4, "n": 1 << 15, "wait": False},
        # a served query of a few sign vectors whose caller waits for the codes
        {"name": "query_d7_1000", "kind": "query", "d": 7, "n": 1000, "wait": True},
        # a long list of septic sign vectors (witness search), an odd number
        {"name": "query_d7_4m", "kind": "query", "d": 7, "n": (1 << 22) + 13, "wait": False},
        # a middling list at the last degree with one-word sign vectors
        {"name": "query_d9_70k", "kind": "query", "d": 9, "n": 70001, "wait": False},
        # two sign words, two code words: a middling list of a larger degree
        {"name": "query_d12_262k", "kind": "query", "d": 12, "n": (1 << 18) - 3, "wait": False},
        # sampled histograms (scheme statistics of one triangulation)
        {"name": "sample_d10_2m", "kind": "sample", "d": 10, "n": (1 << 21) + 777},
        {"name": "sample_d16_262k", "kind": "sample", "d": 16, "n": (1 << 18) + 5},
        # a chunk of an exhaustive sweep, not aligned to anything
        {"name": "sweep_d7_1g", "kind": "sweep", "d": 7, "n": LARGEST, "flag": "plain"},
        # chunks of sweeps modulo symmetry, as checkpointed sweeps run them
        {"name": "sweep_d8_reduced", "kind": "sweep", "d": 8, "n": (1 << 27) + 12345,
         "flag": "reduced"},
        {"name": "sweep_d9_flip", "kind": "sweep", "d": 9, "n": 1 << 26, "flag": "flip"},
        # a mixed-degree batch in one launch, log-uniform job sizes
        {"name": "batch_mixed_fused", "kind": "batch", "d": 5, "d_to": 10, "per_degree": 2,
         "log2_from": 10, "log2_to": 21, "sizes": 31, "fused": True, "given": False},
        # the caller's own sign vectors for many sextic triangulations at once
        {"name": "batch_d6_given", "kind": "batch", "d": 6, "d_to": 6, "per_degree": 60,
         "log2_from": 14, "log2_to": 16, "sizes": 6, "fused": True, "given": True},
    ]


def draw(rng):
    def size(a, b):
        return int(2 ** rng.uniform(a, b)) | rng.randrange(2)

    kind = rng.choice(["query", "query", "sample", "sweep", "sweep", "batch"])
    if kind == "query":
        return {"kind": kind, "d": rng.randint(4, 16), "n": size(8, 21),
                "wait": rng.random() < 0.5}
    if kind == "sample":
        return {"kind": kind, "d": rng.randint(5, 16), "n": size(10, 21)}
    if kind == "sweep":
        d = rng.randint(6, 9)
        return {"kind": kind, "d": d, "n": size(18, 23 if d == 6 else 28),
                "flag": rng.choice(sorted(FLAGS))}
    d = rng.randint(5, 10)
    given = rng.random() < 0.4
    return {"kind": kind, "d": d, "d_to": rng.randint(d, 10), "per_degree": rng.randint(1, 3),
            "log2_from": 8, "log2_to": rng.randint(12, 19), "sizes": rng.randrange(1000),
            "fused": given or rng.random() < 0.7, "given": given}


@functools.lru_cache(maxsize=None)
def _edges(d, tri_id):
    return ti.regular_triangulation(d, seed=d, tri_id=tri_id)


def _words(d, n, seed):
    """n random sign vectors of degree d (W words each) on the GPU."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    w = torch.randint(-(1 << 63), (1 << 63) - 1, (n, ti.sign_words(d)), generator=g,
                      dtype=torch.int64, device="cuda")
    top = ti.num_points(d) - 64 * (ti.sign_words(d) - 1)
    if top < 64:
        w[:, -1] &= (1 << top) - 1
    return w


def _sizes(case):
    """(degree, count) of every job of a batch case."""
    r = np.random.default_rng(case["sizes"])
    return [(d, int(2 ** r.uniform(case["log2_from"], case["log2_to"])))
            for d in range(case["d"], case["d_to"] + 1) for _ in range(case["per_degree"])]


def _free_bits(d, flag):
    return ti.num_points(d) - {"plain": 0, "flip": 1, "reduced": 3, "orbits": 3}[flag]


def _hist_capacity(d):
    return 4096 if d <= 9 else 1 << 16


def prepare(case, seed):
    kind, d = case["kind"], case["d"]
    if kind == "batch":
        jobs = _sizes(case)
        tris = [ts.Triangulation(dj, _edges(dj, j)) for j, (dj, _) in enumerate(jobs)]
        counts = [n for _, n in jobs]
        bases = [(ti.splitmix64_int(seed * 1000 + j) >> 2) for j in range(len(jobs))]
        outs = None
        if case["given"]:  # the codes of all jobs in one buffer
            words = [n * t.code_words for t, n in zip(tris, counts)]
            codes = torch.zeros(sum(words), dtype=torch.int64, device="cuda")
            outs = list(codes.split(words))
        batch = ts.Batch(tris, counts, bases, code_outputs=outs, hist_capacity=1 << 14)
        batch.set_fused(case["fused"])
        if case["given"]:
            for j, (dj, n) in enumerate(jobs):
                batch.set_signs(j, _words(dj, n, seed * 1000 + j))
            return {"kind": kind, "batch": batch, "codes": codes}
        return {"kind": kind, "batch": batch, "codes": None}
    tri = ts.Triangulation(d, _edges(d, seed % 2))
    if kind == "query":
        if d <= 9 and case["n"] >= 1 << 16:
            tri.prepare()
        if case["n"] == 1 << ti.num_points(d):  # all of them, in an order of the seed's
            flip = ti.splitmix64_int(seed) & (case["n"] - 1)
            signs = (torch.arange(case["n"], dtype=torch.int64, device="cuda") ^ flip).reshape(-1, 1)
        else:
            signs = _words(d, case["n"], seed)
        return {"kind": kind, "tri": tri, "signs": signs, "wait": case["wait"]}
    if d <= 9:
        tri.prepare()
    hist = ts.Histogram(_hist_capacity(d), tri.code_words)
    r = ti.splitmix64_int(seed)
    if kind == "sample":
        return {"kind": kind, "tri": tri, "hist": hist, "lo": r >> 2, "n": case["n"],
                "flags": ts.TS_ENUM_SPLITMIX}
    lo = r % ((1 << _free_bits(d, case["flag"])) - case["n"])
    return {"kind": kind, "tri": tri, "hist": hist, "lo": lo, "n": case["n"],
            "flags": FLAGS[case["flag"]]}


def _read(hist, rows):
    """A histogram as a table of fixed length: its sorted codes and their counts, then zeros."""
    codes, counts, failed = hist
    table = np.zeros((rows, 1 + codes.size // max(len(counts), 1)), dtype=np.int64)
    table[:len(counts), 0] = counts.view(np.int64)
    table[:len(counts), 1:] = codes.view(np.int64).reshape(len(counts), -1)
    return {"table": table, "codes": len(counts), "failed": int(failed)}


def run(state):
    if state["kind"] == "query":
        return state["tri"].real_schemes(state["signs"], sync=state["wait"])
    if state["kind"] == "batch":
        batch = state["batch"]
        batch.run()
        if state["codes"] is not None:
            return state["codes"]
        return [_read(batch.read(j), 1 << 14) for j in range(batch.njobs)]
    hist = state["hist"]
    hist.clear()
    ts.enumerate_schemes(state["tri"], state["lo"], state["lo"] + state["n"], hist, state["flags"])
    return _read(hist.read(), hist.capacity)


def work(case):
    """Sign words read once and codes written once (a sweep or sample draws its
    sign vectors and writes a histogram of at most a few thousand codes), and
    the method's integer operations: per instance 3 per sign word, 3.5 per
    edge of the reflected triangulation (6 d^2 + 2 d edges: a crossing test,
    about 1.5 union steps, one find), 6 per antipodal pair and about 4 per
    oval of Harnack's bound."""
    def code_words(d):
        m = (d - 1) * (d - 2) // 2 + 1
        return (2 * (m if d % 2 == 0 else m - 1) + 1 + 63) // 64

    def ops(d):
        return (3 * ti.sign_words(d) + 3.5 * (6 * d * d + 2 * d) + 6 * d
                + 4 * ((d - 1) * (d - 2) // 2 + 1))

    jobs = _sizes(case) if case["kind"] == "batch" else [(case["d"], case["n"])]
    flops = sum(n * ops(d) for d, n in jobs)
    if case["kind"] == "query" or case.get("given"):
        moved = sum(8 * n * (ti.sign_words(d) + code_words(d)) for d, n in jobs)
    else:
        moved = sum(8 * 64 * (1 + code_words(d)) for d, _ in jobs)
    return {"bytes": moved, "flops": flops}


def exact(case, seed):
    """Every output is a whole number (a scheme's code, a count), which has to
    be equal: there is nothing to round."""
    return None
