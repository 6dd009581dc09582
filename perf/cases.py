"""The work that a user of this library has it do, as cases that can be timed.

Two kinds of case, through the public Python entry points:

* ``search``: top-k of a batch of queries over an encoded corpus (rotate the
  queries, scan the codes, keep the k best), with the options a program sets:
  the code width, a tenant filter with per-query allowlists, an id map with
  deleted rows, a TQ+ calibration.  The corpus, its tables, the filter, the id
  map, the workspace and the result buffers are what a serving program keeps;
  the queries are what a request brings.
* ``encode``: rotate, quantise and pack a batch of vectors with the index's
  encode plan (bulk load and online ingest).

The data follow the library's synthetic workloads: a Gaussian mixture on the
unit sphere, queries that are corpus points with noise, Zipf-sized tenants in
shuffled order.  Corpora are drawn in the rotated basis (the mixture's
distribution does not depend on the basis) and quantised here with torch, so
that the codes a search reads do not depend on the encoder.  All
passes go through one created stream, as in a serving loop.
"""
import functools
import math

import numpy as np
import torch

import paper_2607_16973_gb300 as tq
from paper_2607_16973_gb300 import synth

_CHUNK = 32768


def listed():
    def search(name, nq, n, k, bits=4, d=1536, tenants=0, idmap=False, tqplus=False):
        return {"name": name, "kind": "search", "nq": nq, "n": n, "d": d, "bits": bits, "k": k,
                "tenants": tenants, "idmap": idmap, "tqplus": tqplus}

    def encode(name, n, bits=4, d=1536, mode="norm", tqplus=False):
        return {"name": name, "kind": "encode", "n": n, "d": d, "bits": bits, "mode": mode, "tqplus": tqplus}

    return [
        # one interactive query over a small, a mid-sized and a full corpus
        search("one-10k", 1, 10_000, 10),
        search("one-100k", 1, 100_000, 10),
        search("one-999k", 1, 999_000, 5),
        # one query of one tenant among 1000 that share the corpus
        search("tenant-100k", 1, 100_000, 10, tenants=1000),
        # a few queries that arrived together, an odd-sized corpus
        search("eight-250k", 8, 250_007, 10),
        # batches: a busy server, offline jobs, an evaluation run
        search("batch32-999k", 32, 999_000, 5),
        search("batch256-999k", 256, 999_000, 10),
        search("batch1024-999k", 1024, 999_000, 5),
        # another width and dimension, with deletions, external ids and a calibration
        search("mapped-2bit-300k", 50, 300_001, 20, bits=2, d=1024, idmap=True, tqplus=True),
        # ingest of a few documents, of a shard at 8 bits, and a bulk load
        encode("ingest-1000", 1_000),
        encode("ingest-8bit-40k", 40_003, bits=8, d=768, mode="unbiased"),
        encode("load-999k", 999_000),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    d = rng.choice([384, 512, 768, 1024, 1024, 1536, 1536, 1536, 2048])
    bits = rng.choice([4, 4, 4, 4, 4, 4, 2, 3, 8])
    if rng.random() < 0.25:
        n = min(_log_uniform(rng, 1, 999_000), 999_000 * 1536 * 1536 // (d * d))
        return {"kind": "encode", "n": n, "d": d, "bits": bits, "mode": rng.choice(["norm", "norm", "none", "unbiased"]),
                "tqplus": rng.random() < 0.2}
    nq = _log_uniform(rng, 1, 1024)
    n = _log_uniform(rng, 1_000, 999_000)
    n = min(n, 1024 * 999_000 * 1536 // (nq * d))
    tenants = rng.choice([0, 0, 0, 10, 100, 1000])
    return {"kind": "search", "nq": nq, "n": n, "d": d, "bits": bits, "k": rng.choice([1, 3, 5, 5, 10, 10, 20, 50, 100]),
            "tenants": min(tenants, n // 10), "idmap": rng.random() < 0.2, "tqplus": rng.random() < 0.2}


@functools.lru_cache(maxsize=64)
def _codebook(d, bits):
    c, t, _ = tq.codebook(d, bits)
    return c, t


@functools.lru_cache(maxsize=1)
def _stream():
    """The serving loop's stream: one for all states, so that passes follow one another."""
    return torch.cuda.Stream()


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _rotation(d, g):
    """A dense random orthogonal matrix, float32 [d, d] (y = R x)."""
    q, r = torch.linalg.qr(torch.randn(d, d, dtype=torch.float64, device="cuda", generator=g))
    return (q * torch.sign(torch.diagonal(r))).float().contiguous()


def _mixture(n, d, g):
    """Chunks (start, unit float32 rows) of a Gaussian mixture."""
    clusters = 64 if n < 50_000 else 256 if n < 500_000 else 1024
    centres = torch.randn(clusters, d, device="cuda", generator=g)
    for a in range(0, n, _CHUNK):
        m = min(_CHUNK, n - a)
        z = torch.randint(clusters, (m,), device="cuda", generator=g)
        y = torch.randn(m, d, device="cuda", generator=g).mul_(0.5).add_(centres[z])
        yield a, y.div_(y.norm(dim=1, keepdim=True))


def _pack(code, bits):
    """Codes uint8 [m, d] as a little-endian bit stream, uint8 [m, d*bits/8]."""
    m, d = code.shape
    if bits == 8:
        return code
    if bits in (2, 4):
        per = 8 // bits
        c = code.view(m, d // per, per)
        out = c[:, :, 0].clone()
        for i in range(1, per):
            out |= c[:, :, i] << (bits * i)
        return out
    word = torch.zeros(m, d // 8, dtype=torch.int32, device=code.device)
    for i in range(8):
        word |= code[:, i::8].to(torch.int32) << (3 * i)
    return torch.stack([(word >> s) & 255 for s in (0, 8, 16)], dim=2).to(torch.uint8).reshape(m, d * 3 // 8)


def _unpack(codes, d, bits):
    """The codes of packed rows, int64 [m, d]."""
    m = codes.shape[0]
    if bits == 8:
        return codes.long()
    if bits in (2, 4):
        return torch.stack([(codes >> s) & ((1 << bits) - 1) for s in range(0, 8, bits)], dim=2).reshape(m, d).long()
    b = codes.reshape(m, d // 8, 3).to(torch.int32)
    word = b[:, :, 0] | (b[:, :, 1] << 8) | (b[:, :, 2] << 16)
    return torch.stack([(word >> (3 * i)) & 7 for i in range(8)], dim=2).reshape(m, d).long()


def _calibration(d, g):
    """A TQ+ shift and scale of the size that a first batch of embeddings gives."""
    mu = torch.randn(d, device="cuda", generator=g) * (0.1 / math.sqrt(d))
    a = torch.exp(0.1 * torch.randn(d, device="cuda", generator=g))
    return mu, a


def prepare(case, seed):
    g = _generator(seed)
    d, bits, n = case["d"], case["bits"], case["n"]
    R = _rotation(d, g)
    c, t = (torch.from_numpy(v).cuda() for v in _codebook(d, bits))
    calib = _calibration(d, g) if case["tqplus"] else None
    s = {"case": case, "R": R, "c": c, "t": t, "calib": calib, "stream": _stream()}
    if case["kind"] == "encode":
        s["X"] = torch.empty(n, d, device="cuda")
        for a, y in _mixture(n, d, g):
            s["X"][a: a + len(y)] = y
        s["plan"] = tq.encode_plan(R)
        s["codes"] = torch.empty(n, d * bits // 8, dtype=torch.uint8, device="cuda")
        s["scale"] = torch.empty(n, device="cuda")
        return s

    nq, k = case["nq"], case["k"]
    s["codes"] = torch.empty(n, d * bits // 8, dtype=torch.uint8, device="cuda")
    s["scale"] = torch.empty(n, device="cuda")
    src = torch.randint(n, (nq,), device="cuda", generator=g)
    noisy = torch.empty(nq, d, device="cuda")
    for a, y in _mixture(n, d, g):
        z = y if calib is None else (y - calib[0]) / calib[1]
        code = torch.bucketize(z, t, out_int32=True).to(torch.uint8)
        rec = c[code.long()]
        if calib is not None:
            rec = rec * calib[1] + calib[0]
        s["codes"][a: a + len(y)] = _pack(code, bits)
        s["scale"][a: a + len(y)] = 1.0 / rec.norm(dim=1)
        here = (src >= a) & (src < a + len(y))
        noisy[here] = y[src[here] - a]
    noisy += 0.1 * torch.randn(nq, d, device="cuda", generator=g)
    noisy /= noisy.norm(dim=1, keepdim=True)
    s["Q"] = (noisy.double() @ R.double()).float().contiguous()  # y = R x, so x = R^T y

    rng = np.random.default_rng(seed)
    s["filter"] = s["off"] = s["ten"] = s["idmap"] = None
    if case["tenants"]:
        T = case["tenants"]
        values = torch.randperm(1 << 20, device="cuda", generator=g)[:T].to(torch.int32) * 2048 + 7
        ids = torch.repeat_interleave(values, torch.from_numpy(synth.zipf_sizes(n, T)).cuda())
        ids = ids[torch.randperm(n, device="cuda", generator=g)].contiguous()
        s["tenant_ids"] = ids
        s["filter"] = tq.Filter(ids, block=64)
        own, vals, lists = ids[src].cpu().numpy(), values.cpu().numpy(), []
        for i in range(nq):  # the source row's tenant; one list in ten has four more
            more = rng.choice(vals, size=min(4, T - 1), replace=False) if rng.random() < 0.1 else []
            lists.append([own[i]] + [v for v in more if v != own[i]])
        s["off"] = torch.from_numpy(np.cumsum([0] + [len(v) for v in lists]).astype(np.int64)).cuda()
        s["ten"] = torch.from_numpy(np.concatenate([np.asarray(v, np.int32) for v in lists])).cuda()
    if case["idmap"]:
        s["ext"] = rng.permutation(np.arange(1, n + 1, dtype=np.uint64) * np.uint64(2654435761))
        s["gone"] = rng.permutation(n)[: n // 100]
        s["idmap"] = tq.IdMap(n)
        s["idmap"].add(s["ext"])
        s["idmap"].remove(s["ext"][s["gone"]])
    s["workspace"] = torch.empty(tq.search_workspace(nq, n, d, bits, k, s["filter"]), dtype=torch.uint8, device="cuda")
    s["ids"] = torch.empty(nq, k, dtype=torch.int64, device="cuda")
    s["scores"] = torch.empty(nq, k, device="cuda")
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "encode":
        codes, scale = tq.encode(s["X"], s["R"], s["c"], s["t"], case["bits"], case["mode"], s["codes"], s["scale"],
                                 stream=s["stream"], calib=s["calib"], plan=s["plan"])
        return {"codes": codes, "scale": scale}
    ids, scores = tq.search(s["Q"], s["R"], s["c"], case["bits"], s["codes"], s["scale"], case["k"], filter=s["filter"],
                            allow_off=s["off"], allow_tenants=s["ten"], workspace=s["workspace"], out_ids=s["ids"],
                            out_scores=s["scores"], stream=s["stream"], idmap=s["idmap"], calib=s["calib"])
    return {"ids": ids, "scores": scores}


def work(case):
    d, n, rb = case["d"], case["n"], case["d"] * case["bits"] // 8
    if case["kind"] == "encode":
        # X in; codes and scalars out; the rotation matrix
        return {"bytes": n * (4 * d + rb + 4) + 4 * d * d, "flops": 2 * n * d * d}
    nq, k = case["nq"], case["k"]
    # the codes and scalars once, whatever the batch; R and the queries; the results.  (A filter may skip
    # code blocks: with 1000 Zipf tenants about half of the 64-vector blocks hold none of a query's vectors.)
    return {"bytes": n * (rb + 4 + (4 if case["tenants"] else 0)) + 4 * d * d + 4 * nq * d + 12 * nq * k,
            "flops": 2 * nq * n * d + 2 * nq * d * d}


def tolerance(case):
    if case["kind"] == "encode":
        # A coordinate within the arithmetic's error of a cell boundary may land in either cell, and its row's
        # scalar moves with it (by up to about 1e-3 of its value): against 64 bits about 6e-5 in the 2-norm.
        return {"rel": 2.5e-4, "max": 4e-3, "differ": 2e-3 if case["bits"] == 8 else 2e-4}
    # Scores: float32 sums below 16 queries (5e-8 against 64 bits), fp16 products with float32 sums from
    # there on (6.6e-5); neighbours in the ranking that differ by less than that may change places.
    if case["nq"] < 16:
        return {"rel": 5e-7, "differ": 1e-3}
    return {"rel": 3e-4, "differ": 1e-2}


def exact(case, seed):
    s = prepare(case, seed)
    d, bits, n = case["d"], case["bits"], case["n"]
    R, c = s["R"].double(), s["c"].double()
    mu, a = (v.double() for v in s["calib"]) if s["calib"] is not None else (0.0, 1.0)
    if case["kind"] == "encode":
        codes, scale = torch.empty_like(s["codes"]), torch.empty(n, dtype=torch.float64, device="cuda")
        for i in range(0, n, _CHUNK):
            x = s["X"][i: i + _CHUNK].double()
            nr = x.norm(dim=1)
            y = (x / nr[:, None]) @ R.T
            code = torch.bucketize((y - mu) / a, s["t"].double())
            rec = c[code] * a + mu
            codes[i: i + _CHUNK] = _pack(code.to(torch.uint8), bits)
            mode = case["mode"]
            scale[i: i + _CHUNK] = (nr if mode == "none" else nr / rec.norm(dim=1) if mode == "norm"
                                    else nr / (y * rec).sum(dim=1))
        return {"codes": codes, "scale": scale}
    nq, k = case["nq"], case["k"]
    q = s["Q"].double() @ R.T
    step = max(1, min(n, (1 << 28) // max(nq, d)))
    allowed = None
    if case["tenants"]:
        off, ten = s["off"].cpu().numpy(), s["ten"]
        allowed = [ten[off[i]: off[i + 1]] for i in range(nq)]
    live = torch.ones(n, dtype=torch.bool, device="cuda")
    if case["idmap"]:
        live[torch.from_numpy(s["gone"]).cuda()] = False
    best_s = torch.full((nq, k), -math.inf, dtype=torch.float64, device="cuda")
    best_i = torch.full((nq, k), -1, dtype=torch.int64, device="cuda")
    for i in range(0, n, step):
        e = min(n, i + step)
        sc = q @ (c[_unpack(s["codes"][i:e], d, bits)] * a + mu).T * s["scale"][i:e].double()
        sc[:, ~live[i:e]] = -math.inf
        if allowed is not None:
            for j in range(nq):
                sc[j, ~torch.isin(s["tenant_ids"][i:e], allowed[j])] = -math.inf
        both_s = torch.cat([best_s, sc], dim=1)
        both_i = torch.cat([best_i, torch.arange(i, e, device="cuda").expand(nq, -1)], dim=1)
        best_s, at = both_s.topk(k, dim=1)
        best_i = both_i.gather(1, at)
    best_i[best_s == -math.inf] = -1
    if case["idmap"]:
        ext = torch.from_numpy(s["ext"].view(np.int64)).cuda()
        best_i = torch.where(best_i >= 0, ext[best_i.clamp(min=0)], best_i)
    return {"ids": best_i, "scores": best_s}
