"""Performance cases of the comparison library: the calls an application makes,
through the public entry points, over the sizes it makes them at.

Databases and queries are synthetic SNP profiles drawn on the GPU from a seed:
per-locus minor-allele frequency p = 0.05 + 0.45 u, one bit per locus set with
probability 1 - (1 - p)^2.  Queries are individuals (mode 0, mismatch count),
half of them exact copies of database rows, or mixtures of 1-5 people (mode 1,
unexplained alleles) with at least one contributor in the database.

Kinds of case:
  scores   Searcher.scores: the full matrix (small problems, reports)
  topk     Searcher.topk: the fused top-k over a resident database
  host     Searcher.search_host: contributor alleles in host memory in, top-k out
  noalloc  fastid_topk_noalloc: the plain form for callers that may not allocate
  hits     fastid_compare: every pair within a threshold, sorted
  plan     Plan.replay: uneven batches over several loci panels, captured once
  streamed Searcher.topk_streamed: references in pinned host memory
  queries  Searcher.build_queries: allele rows to packed query profiles
"""
import math
import random

import numpy as np
import torch

from paper_1707_00516_gb300 import binding as B
from paper_1707_00516_gb300.search import Searcher, words64

NONE = B.NO_THRESHOLD
FORMS = {"auto": B.FORM_AUTO, "plain": B.FORM_PLAIN, "fp8": B.FORM_TENSOR}
CHUNK_BYTES = 1 << 30  # allele bytes drawn at a time


def listed():
    return [
        # Two laboratories' worth of people: 64 unknown individuals against
        # 10,000 known ones, the whole uint16 matrix.  Latency and launches.
        dict(name="scores_small", kind="scores", n_q=64, n_refs=10_000, n_loci=1024, people="individuals", out_bytes=2),
        # A kinship or quality report: a ragged full uint32 matrix of a small
        # collection, N not a multiple of a word.
        dict(name="scores_report", kind="scores", n_q=500, n_refs=60_001, n_loci=1500, people="half", out_bytes=4),
        # One unknown looked up in a regional database: the smallest search.
        dict(name="topk_one", kind="topk", form="auto", n_q=1, n_refs=100_000, n_loci=1024, people="individuals", k=10,
             threshold=NONE),
        # A serving wave: the mean number of mixtures in flight at the serving
        # workload's load, against the national-size resident database.
        dict(name="topk_wave", kind="topk", form="auto", n_q=48, n_refs=20_000_000, n_loci=2048, people="mixtures", k=16,
             threshold=NONE),
        # The paper's headline shape: 2048 unknowns against 20M knowns.
        dict(name="topk_paper", kind="topk", form="auto", n_q=2048, n_refs=20_000_000, n_loci=2048, people="half", k=32,
             threshold=512),
        # The largest serving request end to end from host memory: 256
        # mixtures, pack, OR, search and results back on the host.
        dict(name="host_batch", kind="host", form="auto", n_q=256, n_refs=5_000_000, n_loci=2048, people="mixtures", k=16,
             threshold=NONE),
        # The FP8 form (its own operand copy), an ordinary batch.
        dict(name="topk_fp8", kind="topk", form="fp8", n_q=500, n_refs=2_000_000, n_loci=2048, people="half", k=32,
             threshold=512),
        # A latency-critical caller that may not allocate: the plain form.
        dict(name="noalloc", kind="noalloc", n_q=32, n_refs=1_000_000, n_loci=2048, people="half", k=16, threshold=NONE),
        # Exclusion screening: every pair within a few genotyping errors.
        dict(name="hits_screen", kind="hits", form="auto", n_q=512, n_refs=1_000_000, n_loci=1024, people="half",
             threshold=10, capacity=1 << 20),
        # Many small uneven batches over four loci panels in one graph replay.
        dict(name="plan_panels", kind="plan", n_refs=250_000, panels="512,2048,8192,16384", n_batches=64, max_batch=512,
             k=16, threshold=NONE),
        # A reference set that stays in host memory, sent in blocks.
        dict(name="streamed", kind="streamed", form="auto", n_q=2048, n_refs=4_000_000, n_loci=2048, people="half", k=32,
             threshold=512, block=1 << 20),
        # Query preparation: contributors' allele rows to packed profiles, a
        # panel whose rows are not 16-byte multiples.
        dict(name="queries_odd", kind="queries", n_q=2048, n_loci=1501, people="mixtures"),
    ]


def _log(rng, lo, hi):
    """An integer in [lo, hi], log-uniform."""
    return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(["scores", "topk", "topk", "topk", "host", "noalloc", "hits", "plan", "streamed", "queries"])
    people = rng.choice(["individuals", "mixtures", "half"])
    k = rng.randint(1, B.MAX_K)
    if kind == "scores":
        n_q, n_loci = _log(rng, 1, 1024), _log(rng, 100, 8192)
        n_refs = _log(rng, 1000, min(500_000, 60_000_000 // n_q))
        return dict(kind=kind, n_q=n_q, n_refs=n_refs, n_loci=n_loci, people=people, out_bytes=rng.choice([2, 4]))
    if kind == "topk":
        form = rng.choice(["auto", "auto", "auto", "fp8", "plain"])
        n_q, n_loci = _log(rng, 1, 2048), _log(rng, 200, 16384)
        top = 2e11 * 32 / (n_q + 128) if form == "plain" else 8e13 / (n_q + 128)
        n_refs = _log(rng, 10_000, int(min(20_000_000, 3e10 / n_loci / (2 if form == "fp8" else 1), top / n_loci)))
        threshold = rng.choice([NONE, NONE, n_loci // 4])
        return dict(kind=kind, form=form, n_q=n_q, n_refs=n_refs, n_loci=n_loci, people=people, k=k, threshold=threshold)
    if kind == "host":
        n_q, n_loci = _log(rng, 1, 1024), _log(rng, 200, 4096)
        n_refs = _log(rng, 10_000, int(2e10 / n_loci))
        return dict(kind=kind, form="auto", n_q=n_q, n_refs=min(n_refs, 10_000_000), n_loci=n_loci, people=people, k=k,
                    threshold=NONE)
    if kind == "noalloc":
        n_q, n_loci = _log(rng, 1, 512), _log(rng, 200, 4096)
        n_refs = _log(rng, 10_000, 2_000_000)
        return dict(kind=kind, n_q=n_q, n_refs=n_refs, n_loci=n_loci, people=people, k=k, threshold=NONE)
    if kind == "hits":
        n_q, n_loci = _log(rng, 16, 1024), _log(rng, 640, 4096)  # from 16 on some are in the database
        n_refs = _log(rng, 10_000, min(2_000_000, 500_000_000 // n_q))
        return dict(kind=kind, form=rng.choice(["auto", "auto", "fp8", "plain"]), n_q=n_q, n_refs=n_refs, n_loci=n_loci,
                    people=people, threshold=rng.randint(0, n_loci // 128), capacity=1 << 21)
    if kind == "plan":
        panels = sorted(_log(rng, 256, 16384) for _ in range(rng.randint(1, 4)))
        return dict(kind=kind, n_refs=_log(rng, 20_000, 300_000), panels=",".join(map(str, panels)),
                    n_batches=_log(rng, 4, 64), max_batch=_log(rng, 16, 512), k=k, threshold=NONE)
    if kind == "streamed":
        n_q, n_loci = _log(rng, 16, 2048), _log(rng, 200, 4096)
        n_refs = _log(rng, 100_000, int(min(4_000_000, 8e9 / n_loci)))
        return dict(kind=kind, form="auto", n_q=n_q, n_refs=n_refs, n_loci=n_loci, people=people, k=k, threshold=NONE,
                    block=_log(rng, 50_000, 1 << 20))
    return dict(kind=kind, n_q=_log(rng, 1, 16384), n_loci=_log(rng, 100, 16384), people=people)


# ---- inputs ---------------------------------------------------------------

def _rng(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1_000_003 + salt) & 0x7FFFFFFFFFFFFFFF)
    return g


def _freq(seed, n_loci):
    """P(bit set) per locus in 256ths."""
    u = torch.rand(n_loci, generator=_rng(seed, 1), device="cuda", dtype=torch.float64)
    p = 0.05 + 0.45 * u
    return (256.0 * (1.0 - (1.0 - p) ** 2)).to(torch.uint8)


def _people(g, n, thr):
    return (torch.empty((n, thr.numel()), dtype=torch.uint8, device="cuda").random_(generator=g) < thr).view(torch.uint8)


def _counts(n_q, people, rs):
    """People per query and its mode."""
    mixed = {"individuals": 0, "mixtures": n_q, "half": n_q - n_q // 2}[people]
    counts = np.ones(n_q, np.int64)
    modes = np.zeros(n_q, np.uint8)
    if mixed:
        counts[n_q - mixed:] = rs.randint(1 if people == "mixtures" else 2, 6, mixed)
        modes[n_q - mixed:] = B.MODE_UNEXPLAINED
    return counts, modes


def _sources(case, seed, thr, n_q, people, n_refs, salt=0):
    """Contributor alleles, group offsets and modes of the queries, and the
    contributors that are database rows: (source rows, their database rows)."""
    rs = np.random.RandomState((int(seed) + 7919 * salt) % (1 << 31))
    counts, modes = _counts(n_q, people, rs)
    offsets = np.zeros(n_q + 1, np.int64)
    offsets[1:] = np.cumsum(counts)
    src = _people(_rng(seed, 2 + salt), int(offsets[-1]), thr)
    planted = np.zeros(int(offsets[-1]), bool)
    planted[offsets[:-1][modes == B.MODE_UNEXPLAINED]] = True  # the first contributor
    more = rs.random_sample(planted.size) < 0.5
    rest = np.ones(planted.size, bool)
    rest[offsets[:-1][modes == B.MODE_UNEXPLAINED]] = False
    planted |= more & rest  # half of the others, and half of the individuals
    rows = np.nonzero(planted)[0]
    if rows.size > n_refs:
        rows = rows[:n_refs]
    at = np.sort(rs.choice(n_refs, rows.size, replace=False)) if n_refs < 4_000_000 else \
        np.unique(rs.randint(0, n_refs, rows.size))
    rows = rs.permutation(rows)[:at.size]
    return src, offsets, modes, rows, at


def _ref_chunks(seed, thr, n_refs, plant):
    """The database's allele rows, (first row, uint8 [n, N]) at a time.
    plant: list of (source alleles, source rows, database rows)."""
    n_loci = thr.numel()
    step = max(1, CHUNK_BYTES // n_loci)
    g = _rng(seed, 3)
    for r0 in range(0, n_refs, step):
        a = _people(g, min(step, n_refs - r0), thr)
        for src, rows, at in plant:
            lo, hi = np.searchsorted(at, [r0, r0 + a.shape[0]])
            if hi > lo:
                a[torch.from_numpy(at[lo:hi] - r0).cuda()] = src[torch.from_numpy(rows[lo:hi]).cuda()]
        yield r0, a


def _query_alleles(src, offsets):
    """Per-locus OR of each query's contributors."""
    off = torch.from_numpy(offsets).cuda()
    q = src[off[:-1]].clone()
    for c in range(1, int(np.max(np.diff(offsets))) if offsets.size > 1 else 0):
        has = (off[1:] - off[:-1]) > c
        q[has] |= src[off[:-1][has] + c]
    return q


def _pack(ctx, alleles):
    out = torch.empty((alleles.shape[0], words64(alleles.shape[1])), dtype=torch.int64, device="cuda")
    B.fastid_pack(ctx, alleles, alleles.shape[1], out)
    return out


def _packed_refs(ctx, seed, thr, n_refs, plant):
    packed = torch.empty((n_refs, words64(thr.numel())), dtype=torch.int64, device="cuda")
    for r0, a in _ref_chunks(seed, thr, n_refs, plant):
        B.fastid_pack(ctx, a, thr.numel(), packed[r0:r0 + a.shape[0]])
    return packed


def _flags(case):
    form = case.get("form", "auto")
    if case["kind"] == "noalloc" or form == "plain":
        return 0
    return B.REFS_TENSOR if form == "fp8" else B.REFS_FP4


# ---- the cases ---------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    s = Searcher(0, FORMS[case.get("form", "auto")])
    if kind == "plan":
        return _prepare_plan(case, seed, s)
    n_loci = case["n_loci"]
    thr = _freq(seed, n_loci)
    if kind == "queries":
        src, offsets, _, _, _ = _sources(case, seed, thr, case["n_q"], case["people"], 1)
        return dict(kind=kind, s=s, src=src, offsets=torch.from_numpy(offsets.astype(np.int32)).cuda(), n_loci=n_loci)
    src, offsets, modes, rows, at = _sources(case, seed, thr, case["n_q"], case["people"], case["n_refs"])
    packed = _packed_refs(s.ctx, seed, thr, case["n_refs"], [(src, rows, at)])
    st = dict(kind=kind, s=s, n_loci=n_loci, k=case.get("k"), threshold=case.get("threshold"))
    if kind == "host":
        st["src"] = src.cpu().pin_memory()
        st["offsets"] = torch.from_numpy(offsets.astype(np.int32)).pin_memory()
        st["modes"] = torch.from_numpy(modes).pin_memory()
    else:
        st["q"] = _pack(s.ctx, _query_alleles(src, offsets))
        st["modes"] = torch.from_numpy(modes).cuda()
    if kind == "streamed":
        refs = torch.empty(packed.shape, dtype=torch.int64, pin_memory=True)
        refs.copy_(packed)
        st.update(refs=refs, block=case["block"])
    else:
        st["db"] = B.fastid_load_refs(s.ctx, packed, n_loci, _flags(case))
    n_q = case["n_q"]
    if kind == "scores":
        st["dtype"] = torch.int16 if case["out_bytes"] == 2 else torch.int32
    if kind == "noalloc":
        st["out"] = (torch.empty((n_q, case["k"]), dtype=torch.int32, device="cuda"),
                     torch.empty((n_q, case["k"]), dtype=torch.int64, device="cuda"))
    if kind == "hits":
        cap = case["capacity"]
        st["out"] = (torch.full((cap,), -1, dtype=torch.int64, device="cuda"),
                     torch.full((cap,), -1, dtype=torch.int64, device="cuda"),
                     torch.full((cap,), -1, dtype=torch.int32, device="cuda"),
                     torch.zeros(1, dtype=torch.int64, device="cuda"))
    torch.cuda.synchronize()
    return st


def _batches(case, seed):
    """Panel and size of every batch: sizes log-uniform on 1..max_batch."""
    rs = random.Random(int(seed) * 31 + 5)
    n_panels = len(case["panels"].split(","))
    return [(rs.randrange(n_panels), _log(rs, 1, case["max_batch"])) for _ in range(case["n_batches"])]


def _plan_inputs(case, seed):
    """Per panel: loci, thresholds, and per batch its queries; batches in order."""
    loci = [int(x) for x in case["panels"].split(",")]
    thr = [_freq(seed * 8 + p, n) for p, n in enumerate(loci)]
    plants, queries = [[] for _ in loci], []
    for b, (p, n) in enumerate(_batches(case, 0)):  # the batch shapes belong to the case, not to the seed
        src, offsets, modes, rows, at = _sources(case, seed, thr[p], n, "half", case["n_refs"], salt=10 + b)
        plants[p].append((src, rows, at))
        queries.append((p, _query_alleles(src, offsets), modes))
    return loci, thr, plants, queries


def _prepare_plan(case, seed, s):
    loci, thr, plants, queries = _plan_inputs(case, seed)
    dbs = []
    for p in range(len(loci)):
        packed = _packed_refs(s.ctx, seed * 8 + p, thr[p], case["n_refs"], plants[p])
        dbs.append(B.fastid_load_refs(s.ctx, packed, loci[p], B.REFS_FP4))
        torch.cuda.synchronize()
    total, k = sum(q.shape[0] for _, q, _ in queries), case["k"]
    scores = torch.empty((total, k), dtype=torch.int32, device="cuda")
    idx = torch.empty((total, k), dtype=torch.int64, device="cuda")
    batches, o = [], 0
    for p, q, modes in queries:
        n = q.shape[0]
        batches.append((p, _pack(s.ctx, q), torch.from_numpy(modes).cuda(), scores[o:o + n], idx[o:o + n]))
        o += n
    plan = B.Plan(s.ctx, dbs, batches, k, case["threshold"])
    plan.capture()
    torch.cuda.synchronize()
    return dict(kind="plan", plan=plan, scores=scores, idx=idx, s=s)


def run(state):
    kind = state["kind"]
    if kind == "plan":
        state["plan"].replay()
        return state["scores"], state["idx"]
    s = state["s"]
    if kind == "queries":
        return s.build_queries(state["src"], state["offsets"], state["n_loci"])
    if kind == "scores":
        return s.scores(state["db"], state["q"], state["modes"], state["dtype"])
    if kind == "topk":
        return s.topk(state["db"], state["q"], state["modes"], state["k"], state["threshold"])
    if kind == "host":
        scores, idx, _, _ = s.search_host(state["db"], state["src"], state["offsets"], state["modes"], state["k"],
                                          state["threshold"])
        return scores.view(np.int32), idx
    if kind == "noalloc":
        scores, idx = state["out"]
        B.fastid_topk_noalloc(s.ctx, state["db"], state["q"], state["modes"], state["k"], state["threshold"], scores, idx)
        return scores, idx
    if kind == "streamed":
        return s.topk_streamed(state["refs"], state["n_loci"], state["q"], state["modes"], state["k"],
                               state["threshold"], state["block"])
    hq, hr, hs, hc = state["out"]
    B.fastid_compare(s.ctx, state["db"], state["q"], state["modes"], state["threshold"], hq, hr, hs, hc)
    return hq, hr, hs, hc


def work(case):
    """Packed references, queries and results once; a multiply-add a locus."""
    kind = case["kind"]
    if kind == "plan":
        loci = [int(x) for x in case["panels"].split(",")]
        sizes = _batches(case, 0)
        return {"bytes": sum(case["n_refs"] * words64(n) * 8 for n in loci)
                + sum(n * (words64(loci[p]) * 8 + 1 + 12 * case["k"]) for p, n in sizes),
                "flops": sum(2.0 * n * case["n_refs"] * loci[p] for p, n in sizes)}
    n_q, n_loci, w = case["n_q"], case["n_loci"], words64(case["n_loci"]) * 8
    people = {"individuals": 1.0, "mixtures": 3.0, "half": 2.25}[case["people"]]
    if kind == "queries":
        return {"bytes": n_q * (people * n_loci + w), "flops": 0}
    n_refs = case["n_refs"]
    bytes_ = n_refs * w + n_q * (people * n_loci if kind == "host" else w) + n_q
    if kind == "scores":
        bytes_ += n_q * n_refs * case["out_bytes"]
    elif kind != "hits":
        bytes_ += n_q * case["k"] * 12
    return {"bytes": bytes_, "flops": 2.0 * n_q * n_refs * n_loci}


# ---- the same results in plain torch, 64-bit, from the unpacked alleles ------------

def _score_chunk(a, q, modes):
    """int64 [n_q, n]: sum over loci of XOR (mode 0) or of R AND NOT Q (mode 1)."""
    r = a.double()
    both = (q.double() @ r.T).long()
    r_sum, q_sum = a.sum(1, dtype=torch.int64), q.sum(1, dtype=torch.int64)
    mis = r_sum[None, :] + q_sum[:, None] - 2 * both
    return torch.where((modes == B.MODE_MISMATCH)[:, None], mis, r_sum[None, :] - both)


def _exact_topk(seed, thr, n_refs, plant, q, modes, k, threshold):
    empty = torch.iinfo(torch.int64).max
    best = torch.full((q.shape[0], k), empty, dtype=torch.int64, device="cuda")
    for r0, a in _ref_chunks(seed, thr, n_refs, plant):
        for i in range(0, a.shape[0], 1 << 15):
            sc = _score_chunk(a[i:i + (1 << 15)], q, modes)
            key = (sc << 32) + torch.arange(r0 + i, r0 + i + sc.shape[1], device="cuda")
            if threshold != NONE:
                key[sc > threshold] = empty
            best = torch.cat([best, key], 1).topk(k, dim=1, largest=False, sorted=True).values
    none = best == empty
    return torch.where(none, -1, best >> 32).to(torch.int32), torch.where(none, -1, best & 0xFFFFFFFF)


def exact(case, seed):
    kind = case["kind"]
    if kind == "queries":
        thr = _freq(seed, case["n_loci"])
        src, offsets, _, _, _ = _sources(case, seed, thr, case["n_q"], case["people"], 1)
        q = _query_alleles(src, offsets)
        w = words64(case["n_loci"])
        q = torch.nn.functional.pad(q, (0, w * 64 - q.shape[1])).view(-1, w, 64)
        out = torch.zeros(q.shape[:2], dtype=torch.int64, device="cuda")
        for b in range(64):
            out |= q[:, :, b].long() << b
        return out
    if work(case)["flops"] > 5e12:
        return None
    if kind == "plan":
        loci, thr, plants, queries = _plan_inputs(case, seed)
        got = [_exact_topk(seed * 8 + p, thr[p], case["n_refs"], plants[p], q, torch.from_numpy(m).cuda(), case["k"],
                           case["threshold"]) for p, q, m in queries]
        return torch.cat([g[0] for g in got]), torch.cat([g[1] for g in got])
    thr = _freq(seed, case["n_loci"])
    src, offsets, modes, rows, at = _sources(case, seed, thr, case["n_q"], case["people"], case["n_refs"])
    q, modes, plant = _query_alleles(src, offsets), torch.from_numpy(modes).cuda(), [(src, rows, at)]
    if kind not in ("scores", "hits"):
        return _exact_topk(seed, thr, case["n_refs"], plant, q, modes, case["k"], case["threshold"])
    parts = []
    for r0, a in _ref_chunks(seed, thr, case["n_refs"], plant):
        for i in range(0, a.shape[0], 1 << 15):
            sc = _score_chunk(a[i:i + (1 << 15)], q, modes)
            if kind == "scores":
                parts.append(sc.to(torch.int16 if case["out_bytes"] == 2 else torch.int32))
            else:
                qi, ri = torch.nonzero(sc <= case["threshold"], as_tuple=True)
                parts.append(torch.stack([qi, ri + (r0 + i), sc[qi, ri]], 1))
    if kind == "scores":
        return torch.cat(parts, 1)
    h = torch.cat(parts)
    h = h[torch.argsort((h[:, 0] << 32) + h[:, 1])]
    out = torch.full((3, case["capacity"]), -1, dtype=torch.int64, device="cuda")
    out[:, :h.shape[0]] = h.T
    return out[0], out[1], out[2].to(torch.int32), torch.tensor([h.shape[0]], dtype=torch.int64, device="cuda")
