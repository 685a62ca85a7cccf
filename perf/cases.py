"""The calls whose speed counts, as a user's program makes them.

Twelve listed cases and a generator of more over the same ranges: 2-way tables
of a few hundred to fifty thousand SNPs over a thousand to a million
individuals, whole, thresholded, batched and in two steps, on the tensor-core
and the popcount path, 3-way tables, and markers with several allele states.
Panels are synthetic with the distributions of `synth/` (Hardy-Weinberg
genotypes, folded Beta(1/2, 1/2) allele frequencies floored at 0.01, 1%
missing; uniform genotypes with 2% missing for the small panel), drawn on the
GPU from the seed.
"""

import math
import random

import torch

import paper_1705_08213_gb300 as ccc

GAMMA = 2.0 / 3.0
HIT_CAP = 8192  # records of the thresholded output's buffer
CHUNK = 1 << 27  # entries generated or decoded at a time


def listed():
    return [
        # A candidate-gene set: one launch-bound call, the smallest panel of the benchmark.
        {"name": "pairs_small", "kind": "pairs", "n_v": 256, "n_f": 1024, "norm": "persnp", "uniform": True},
        # A chromosome window of a small cohort, no size a multiple of anything; joint normalisation.
        {"name": "pairs_odd", "kind": "pairs", "n_v": 3001, "n_f": 2503, "norm": "joint", "uniform": False},
        # Many SNPs over an ordinary cohort: as many bytes of results as of tensor work.
        {"name": "pairs_wide", "kind": "pairs", "n_v": 20000, "n_f": 4096, "norm": "persnp", "uniform": False},
        # The benchmark's headline panel.
        {"name": "pairs_scale", "kind": "pairs", "n_v": 20000, "n_f": 16384, "norm": "persnp", "uniform": False},
        # A biobank: few SNPs, a million individuals.
        {"name": "pairs_long", "kind": "pairs", "n_v": 512, "n_f": 1000000, "norm": "persnp", "uniform": False},
        # Counts, tallies and values by separate calls, as a program does that sums
        # the tallies of several cohorts before it takes the values.
        {"name": "pairs_two_step", "kind": "two_step", "n_v": 10000, "n_f": 2048, "norm": "persnp", "uniform": False},
        # Thresholded output: only near-duplicate pairs are kept.
        {"name": "pairs_filter", "kind": "filter", "n_v": 50000, "n_f": 4096, "norm": "persnp", "uniform": False},
        # A multi-study run: panels of uneven sizes in one call.
        {"name": "pairs_batched", "kind": "batched", "panels": 16, "n_v": 8000, "n_f": 50000, "shapes": 2, "norm": "persnp"},
        # The bitwise path of the paper.
        {"name": "pairs_popc", "kind": "popc", "n_v": 4096, "n_f": 16384, "norm": "persnp", "uniform": False},
        # All triples of the benchmark's 3-way panel.
        {"name": "triples", "kind": "triples", "n_v": 1536, "n_f": 8192, "norm": "persnp", "uniform": False},
        # All triples of a short candidate list; joint normalisation.
        {"name": "triples_odd", "kind": "triples", "n_v": 301, "n_f": 2001, "norm": "joint", "uniform": False},
        # Nucleotide markers (four states), the benchmark's panel.
        {"name": "markers", "kind": "markers", "n_v": 10000, "n_f": 16384, "s": 4, "norm": "persnp"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pairs", "pairs", "pairs", "long", "two_step", "filter", "batched", "popc", "triples",
                       "triples", "markers", "markers"])
    norm = rng.choice(["persnp", "persnp", "joint"])
    if kind == "pairs":
        return {"kind": kind, "n_v": _log(rng, 256, 20000), "n_f": _log(rng, 1000, 16384), "norm": norm,
                "uniform": rng.random() < 0.2}
    if kind == "long":
        return {"kind": "pairs", "n_v": _log(rng, 100, 512), "n_f": _log(rng, 100000, 1000000), "norm": norm,
                "uniform": False}
    if kind == "two_step":
        return {"kind": kind, "n_v": _log(rng, 500, 10000), "n_f": _log(rng, 1000, 8192), "norm": norm,
                "uniform": False}
    if kind == "filter":
        return {"kind": kind, "n_v": _log(rng, 5000, 50000), "n_f": _log(rng, 4096, 8192), "norm": "persnp",
                "uniform": False}
    if kind == "batched":
        return {"kind": kind, "panels": rng.randint(4, 16), "n_v": _log(rng, 1000, 8000),
                "n_f": _log(rng, 4000, 50000), "shapes": rng.randrange(1 << 20), "norm": norm}
    if kind == "popc":
        return {"kind": kind, "n_v": _log(rng, 256, 4096), "n_f": _log(rng, 1000, 16384), "norm": norm,
                "uniform": False}
    if kind == "triples":
        return {"kind": kind, "n_v": _log(rng, 150, 1200), "n_f": _log(rng, 1000, 8192), "norm": norm,
                "uniform": False}
    return {"kind": kind, "n_v": _log(rng, 500, 5000), "n_f": _log(rng, 1000, 16384), "s": rng.choice([2, 3, 4, 5, 6, 8]),
            "norm": norm}


# ---------------------------------------------------------------- inputs


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)


def _codes(n_v, n_f, seed, uniform):
    """2-bit entry codes as uint8 [n_v, n_f]: 0 = (0,0), 1 = (0,1), 3 = (1,1), 2 = missing."""
    g = _generator(seed)
    x = torch.sin(torch.rand(n_v, 1, generator=g, device="cuda") * (math.pi / 2)) ** 2
    p = torch.minimum(x, 1 - x).clamp_min(0.01)
    a, b = ((1 - p) ** 2, 1 - p ** 2) if not uniform else (torch.full_like(p, 1 / 3), torch.full_like(p, 2 / 3))
    missing = 0.02 if uniform else 0.01
    out = torch.empty(n_v, n_f, dtype=torch.uint8, device="cuda")
    rows = max(1, CHUNK // n_f)
    for r in range(0, n_v, rows):
        s = slice(r, min(n_v, r + rows))
        u = torch.rand(s.stop - s.start, n_f, generator=g, device="cuda")
        c = (u >= a[s]).to(torch.uint8)
        c += 2 * (u >= b[s]).to(torch.uint8)
        u.uniform_(generator=g)
        out[s] = c.masked_fill_(u < missing, 2)
    return out


def _plant(codes, seed, pairs):
    """Near-duplicates: the second row of `pairs` random disjoint pairs becomes the first with
    1% of its entries redrawn."""
    g = _generator(seed + 77)
    n_v, n_f = codes.shape
    rows = torch.randperm(n_v, generator=g, device="cuda")[:2 * pairs]
    src, dst = codes[rows[:pairs]], rows[pairs:]
    other = torch.gather(src, 1, torch.randint(0, n_f, src.shape, generator=g, device="cuda"))
    codes[dst] = torch.where(torch.rand(src.shape, generator=g, device="cuda") < 0.01, other, src)
    return codes


def _pack(codes):
    """The packed panel: int64 [n_v, ld], 32 entries per word, rows of whole 16 bytes."""
    n_v, n_f = codes.shape
    width = -(-n_f // 64) * 64
    out = torch.empty(n_v, width // 4, dtype=torch.uint8, device="cuda")
    rows = max(1, CHUNK // n_f)
    for r in range(0, n_v, rows):
        c = codes[r:r + rows]
        if width != n_f:
            c = torch.nn.functional.pad(c, (0, width - n_f))
        c = c.view(c.shape[0], width // 4, 4)
        out[r:r + rows] = c[..., 0] | (c[..., 1] << 2) | (c[..., 2] << 4) | (c[..., 3] << 6)
    return out.view(torch.int64)


def _states(n_v, n_f, s, seed):
    """Unordered allele-state pairs as bytes x | (y << 4), 0xFF = missing."""
    g = _generator(seed)
    w = (torch.sin(torch.rand(n_v, s, generator=g, device="cuda") * (math.pi / 2)) ** 2).clamp_min(0.01)
    cum = (w / w.sum(1, keepdim=True)).cumsum(1)
    out = torch.empty(n_v, n_f, dtype=torch.uint8, device="cuda")
    rows = max(1, CHUNK // n_f)
    for r in range(0, n_v, rows):
        e = slice(r, min(n_v, r + rows))
        both = []
        for _ in range(2):
            u = torch.rand(e.stop - e.start, n_f, generator=g, device="cuda")
            both.append(sum((u >= cum[e, a:a + 1]).to(torch.uint8) for a in range(s - 1)))
        byte = both[0] | (both[1] << 4)
        out[e] = byte.masked_fill_(torch.rand(byte.shape, generator=g, device="cuda") < 0.01, 0xFF)
    return out


def _shapes(case):
    r = random.Random(case["shapes"])
    return [(r.randint(min(500, case["n_v"]), case["n_v"]), r.randint(min(2000, case["n_f"]), case["n_f"]))
            for _ in range(case["panels"])]


def _panel_codes(case, seed):
    codes = _codes(case["n_v"], case["n_f"], seed, case["uniform"])
    return _plant(codes, seed, case["n_v"] // 100) if case["kind"] == "filter" else codes


def _norm(case):
    return ccc.CCC_NORM_JOINT if case["norm"] == "joint" else ccc.CCC_NORM_PERSNP


def _results(count, width):
    return (torch.empty(count, width, dtype=torch.int32, device="cuda"),
            torch.empty(count, width, dtype=torch.float32, device="cuda"))


def _workspace(size_of, **options):
    """Options with a workspace of the size the library asks for."""
    opts = ccc.ccc_opts_default(**options)
    workspace = torch.empty(size_of(opts), dtype=torch.uint8, device="cuda")
    return ccc.ccc_opts_default(workspace=workspace, **options), workspace


def prepare(case, seed):
    kind, norm = case["kind"], _norm(case)
    if kind == "batched":
        shapes = _shapes(case)
        genos = [_pack(_codes(v, f, seed * 64 + k, False)) for k, (v, f) in enumerate(shapes)]
        n_fs = [f for _, f in shapes]
        opts, ws = _workspace(lambda o: ccc.ccc2_batched_workspace_size(genos, n_fs, o), norm=norm)
        outs = [_results(ccc.ccc2_count(v), 4) for v, _ in shapes]
        return {"kind": kind, "genos": genos, "n_fs": n_fs, "opts": opts, "workspace": ws,
                "tallies": [t for t, _ in outs], "cccs": [c for _, c in outs]}
    n_v, n_f = case["n_v"], case["n_f"]
    state = {"kind": kind, "n_v": n_v, "n_f": n_f}
    if kind == "markers":
        s = state["s"] = case["s"]
        geno = _states(n_v, n_f, s, seed)
        if n_f % 16:
            geno = torch.nn.functional.pad(geno, (0, -n_f % 16), value=0xFF)
        state["geno"] = geno.contiguous()
        state["opts"], state["workspace"] = _workspace(
            lambda o: ccc.ccc_multi_workspace_size(state["geno"], n_f, s, o), norm=norm)
        state["tally"], state["ccc"] = _results(ccc.ccc2_count(n_v), s * s)
        return state
    geno = state["geno"] = _pack(_panel_codes(case, seed))
    op = ccc.CCC_OP_3WAY if kind == "triples" else ccc.CCC_OP_2WAY
    state["opts"], state["workspace"] = _workspace(
        lambda o: ccc.ccc_workspace_size(geno, n_f, o, op), norm=norm,
        path=ccc.CCC_PATH_POPC if kind == "popc" else ccc.CCC_PATH_TC)
    if kind == "filter":
        state["hits"] = torch.zeros(HIT_CAP, 10, dtype=torch.int32, device="cuda")
        state["n_hits"] = torch.zeros(1, dtype=torch.int64, device="cuda")
    elif kind == "triples":
        state["tally"], state["ccc"] = _results(ccc.ccc3_count(n_v, 0, n_v), 8)
    else:
        state["tally"], state["ccc"] = _results(ccc.ccc2_count(n_v), 4)
    if kind == "two_step":
        state["counts"] = torch.empty(n_v, 3, dtype=torch.int32, device="cuda")
    return state


# ---------------------------------------------------------------- one pass


THRESHOLD = 0.16  # above what independent SNPs reach, below near-duplicates of common ones


def run(state):
    kind, opts = state["kind"], state["opts"]
    if kind == "batched":
        ccc.ccc2_batched(state["genos"], state["n_fs"], state["tallies"], state["cccs"], opts)
        return {"tally": state["tallies"], "ccc": state["cccs"]}
    geno, n_f = state["geno"], state["n_f"]
    if kind == "filter":
        hits = state["hits"]
        ccc.ccc2_filter(geno, n_f, THRESHOLD, hits, HIT_CAP, state["n_hits"], opts)
        # The records come in no particular order: by pair, the unused (zero) ones first.
        hits = hits[(hits[:, 0].long() * state["n_v"] + hits[:, 1]).argsort()]
        return {"n_hits": state["n_hits"], "pair": hits[:, :2], "tally": hits[:, 2:6],
                "ccc": hits[:, 6:].view(torch.float32)}
    tally, value = state["tally"], state["ccc"]
    if kind == "triples":
        ccc.ccc3_tally_metric(geno, n_f, 0, state["n_v"], tally, value, opts)
    elif kind == "markers":
        ccc.ccc2_multi_tally_metric(geno, n_f, state["s"], tally, value, opts)
    elif kind == "two_step":
        ccc.ccc_allele_counts(geno, n_f, state["counts"])
        ccc.ccc2_tally(geno, n_f, tally, opts)
        ccc.ccc2_metric(tally, state["counts"], state["n_v"], opts, value)
        return {"counts": state["counts"], "tally": tally, "ccc": value}
    else:
        ccc.ccc2_tally_metric(geno, n_f, tally, value, opts)
    return {"tally": tally, "ccc": value}


def _pair_work(n_v, n_f, s, entry_bytes):
    """Panel read once, s * s tallies and values written once; s * s multiply-adds per comparison."""
    pairs = n_v * (n_v - 1) // 2
    return entry_bytes * n_v * n_f + 8 * s * s * pairs, 2 * s * s * pairs * n_f


def work(case):
    kind = case["kind"]
    if kind == "batched":
        parts = [_pair_work(v, f, 2, 0.25) for v, f in _shapes(case)]
        return {"bytes": sum(b for b, _ in parts), "flops": sum(f for _, f in parts)}
    n_v, n_f = case["n_v"], case["n_f"]
    if kind == "triples":
        triples = n_v * (n_v - 1) * (n_v - 2) // 6
        return {"bytes": 0.25 * n_v * n_f + 64 * triples, "flops": 16 * triples * n_f}
    s = case["s"] if kind == "markers" else 2
    nbytes, flops = _pair_work(n_v, n_f, s, 1 if kind == "markers" else 0.25)
    if kind == "filter":
        nbytes = 0.25 * n_v * n_f
    elif kind == "two_step":
        nbytes += 12 * n_v
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- the same in 64 bits
#
# Tallies come from single-precision matrix products of allele counts: every
# partial sum is a whole number below 2^24, so they are exact in any order.
# Everything after them is in 64 bits.


def _count_rows(codes):
    """[2 n_v, n_f] single-precision allele counts: row 2 i + a = copies of allele a."""
    table = torch.tensor([[2, 0], [1, 1], [0, 0], [0, 2]], dtype=torch.float32, device="cuda")
    out = torch.empty(codes.shape[0], 2, codes.shape[1], dtype=torch.float32, device="cuda")
    for a in range(2):
        rows = max(1, CHUNK // codes.shape[1])
        for r in range(0, codes.shape[0], rows):
            out[r:r + rows, a] = table[:, a][codes[r:r + rows].int()]
    return out.view(2 * codes.shape[0], codes.shape[1])


def _state_rows(byte, s):
    """The same for s states: row s i + a."""
    out = torch.empty(byte.shape[0], s, byte.shape[1], dtype=torch.float32, device="cuda")
    for a in range(s):
        out[:, a] = (byte & 15 == a).float() + (byte >> 4 == a).float()
    return out.view(s * byte.shape[0], byte.shape[1])


def _factors(rows, s):
    """1 - gamma f_i(a), [n_v, s]."""
    sums = torch.stack([rows[k::s].sum(1, dtype=torch.float64) for k in range(s)], 1)
    total = sums.sum(1, keepdim=True)
    return 1 - GAMMA * torch.where(total > 0, sums / total.clamp_min(1), 0.0)


def _values(t, joint, factors):
    """CCC values of tables t [..., s, s (, s)] (64 bits); factors: one [..., s] per axis."""
    axes = len(factors)
    over = tuple(range(t.dim() - axes, t.dim()))
    n = t.sum(over, keepdim=True)
    out = t / n.clamp_min(1)
    for k, f in enumerate(factors):
        if joint:
            w = 1 - GAMMA * t.sum([d for d in over if d != over[k]], keepdim=True) / n.clamp_min(1)
        else:
            w = f.reshape(f.shape[:-1] + (1,) * k + (f.shape[-1],) + (1,) * (axes - 1 - k))
        out = out * w
    return out


def _pair_blocks(rows, s):
    """(i, j, tables [pairs, s, s] in 64 bits) of row blocks of the upper triangle, in its order."""
    n_v = rows.shape[0] // s
    step = max(1, (1 << 25) // (s * s * n_v))
    for i0 in range(0, n_v - 1, step):
        i1 = min(n_v, i0 + step)
        t = rows[s * i0:s * i1] @ rows[s * i0:].T
        t = t.view(i1 - i0, s, n_v - i0, s).permute(0, 2, 1, 3)
        keep = torch.ones(i1 - i0, n_v - i0, dtype=torch.bool, device="cuda").triu_(1)
        i, j = keep.nonzero(as_tuple=True)
        yield i + i0, j + i0, t[i, j].double()


def _exact_pairs(rows, s, joint):
    n_v = rows.shape[0] // s
    w = _factors(rows, s)
    tally = torch.empty(n_v * (n_v - 1) // 2, s * s, dtype=torch.int32, device="cuda")
    value = torch.empty(tally.shape, dtype=torch.float64, device="cuda")
    at = 0
    for i, j, t in _pair_blocks(rows, s):
        tally[at:at + len(i)] = t.reshape(-1, s * s).int()
        value[at:at + len(i)] = _values(t, joint, (w[i], w[j])).reshape(-1, s * s)
        at += len(i)
    return {"tally": tally, "ccc": value}


def _exact_filter(rows, n_v):
    w = _factors(rows, 2)
    pair, tally, value, keys, total = [], [], [], [], 0
    for i, j, t in _pair_blocks(rows, 2):
        v = _values(t, False, (w[i], w[j])).reshape(-1, 4)
        k = (v.amax(1) > THRESHOLD).nonzero().flatten()
        total += len(k)
        pair.append(torch.stack([i[k], j[k]], 1).int())
        tally.append(t.reshape(-1, 4)[k].int())
        value.append(v[k])
        keys.append(i[k] * n_v + j[k])
    order = torch.cat(keys).argsort()
    free = HIT_CAP - total

    def laid(parts):
        kept = torch.cat(parts)[order]
        return torch.cat([kept.new_zeros(free, kept.shape[1]), kept])

    return {"n_hits": torch.tensor([total], device="cuda"), "pair": laid(pair), "tally": laid(tally), "ccc": laid(value)}


def _exact_triples(rows, n_v, joint):
    w = _factors(rows, 2)
    count = n_v * (n_v - 1) * (n_v - 2) // 6
    tally = torch.empty(count, 8, dtype=torch.int32, device="cuda")
    value = torch.empty(count, 8, dtype=torch.float64, device="cuda")
    at = 0
    for j in range(1, n_v - 1):
        left, right = rows[:2 * j], rows[2 * j + 2:]
        t = torch.stack([((left * rows[2 * j + b]) @ right.T).view(j, 2, n_v - 1 - j, 2) for b in range(2)], 2)
        t = t.permute(0, 3, 1, 2, 4).double()  # i, k, a, b, c
        v = _values(t, joint, (w[:j, None], w[j][None, None], w[None, j + 1:]))
        n = t.shape[0] * t.shape[1]
        tally[at:at + n] = t.reshape(n, 8).int()
        value[at:at + n] = v.reshape(n, 8)
        at += n
    return {"tally": tally, "ccc": value}


def exact(case, seed):
    kind, joint = case["kind"], case["norm"] == "joint"
    if kind == "batched":
        outs = [_exact_pairs(_count_rows(_codes(v, f, seed * 64 + k, False)), 2, joint)
                for k, (v, f) in enumerate(_shapes(case))]
        return {"tally": [o["tally"] for o in outs], "ccc": [o["ccc"] for o in outs]}
    if kind == "markers":
        return _exact_pairs(_state_rows(_states(case["n_v"], case["n_f"], case["s"], seed), case["s"]), case["s"], joint)
    rows = _count_rows(_panel_codes(case, seed))
    if kind == "triples":
        return _exact_triples(rows, case["n_v"], joint)
    if kind == "filter":
        return _exact_filter(rows, case["n_v"])
    out = _exact_pairs(rows, 2, joint)
    if kind == "two_step":
        sums = torch.stack([rows[a::2].sum(1, dtype=torch.float64) for a in range(2)], 1)
        out["counts"] = torch.cat([sums, sums.sum(1, keepdim=True) / 2], 1).int()
    return out
