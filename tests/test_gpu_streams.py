"""Searches and encodes on created streams, where the kernels of a call are
programmatic dependents of one another, under graph capture, and from several
threads: the results are the default stream's, where nothing overlaps."""
import threading

import numpy as np
import pytest

import oracle as O
from paper_2607_16973_gb300 import synth

pytestmark = pytest.mark.gpu

ROUTES = [  # nq, n, d, bits, k, filtered, the scan
    (1, 20_000, 1536, 4, 10, False, "k_scan_tm (exact)"),
    (4, 60_001, 512, 4, 10, True, "k_scan_tm (exact)"),
    (20, 9_001, 512, 4, 10, True, "k_scan_tm"),
    (64, 30_001, 256, 2, 20, False, "k_scan_mma"),
    (300, 30_001, 256, 4, 5, True, "k_scan_mma"),
    (3, 12_000, 256, 8, 10, True, "k_scan_stream"),
    (2, 12_000, 256, 3, 33, False, "k_scan_ring"),
]


class Search:
    """One route's corpus and buffers; run() queues a search of batch `b` (of two)."""

    def __init__(self, tq, torch, route):
        self.tq, self.torch = tq, torch
        nq, n, d, bits, k, filtered, scan = route
        assert tq.search_kernel(nq, n, d, bits, k, filtered) == scan
        T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
        self.Q = [T(synth.gaussian_rows(nq, d, seed=s)) for s in (1, 2)]
        self.q = self.Q[0].clone()
        self.tail = (T(O.rotation(d, 5).astype(np.float32)), T(tq.codebook(d, bits)[0]), bits,
                     T(synth.random_codes(n, d * bits // 8, seed=n)), T(synth.random_scales(n, seed=n)), k)
        self.kw = {}
        if filtered:
            tenants, values = synth.zipf_tenants(n, 50)
            off, allow = synth.allowlists(synth.query_sources(n, nq), tenants, values)
            self.kw = dict(filter=tq.Filter(T(tenants.view(np.int32))), allow_off=T(off),
                           allow_tenants=T(allow.view(np.int32)))
        self.want = [tuple(x.clone() for x in tq.search(q, *self.tail, **self.kw)) for q in self.Q]
        self.ws = torch.empty(tq.search_workspace(nq, n, d, bits, k, self.kw.get("filter")), dtype=torch.uint8,
                              device="cuda")
        self.out = torch.empty(nq, k, dtype=torch.int64, device="cuda"), torch.empty(nq, k, device="cuda")
        torch.cuda.synchronize()

    def run(self, stream):
        self.tq.search(self.q, *self.tail, workspace=self.ws, out_ids=self.out[0], out_scores=self.out[1],
                       stream=stream, **self.kw)

    def check(self, b):
        assert all(self.torch.equal(x, y) for x, y in zip(self.out, self.want[b]))


class Encode:
    def __init__(self, tq, torch, n=300, d=1024):
        self.tq, self.torch = tq, torch
        T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
        self.Q = [T(synth.gaussian_rows(n, d, seed=s)) for s in (1, 2)]
        self.q = self.Q[0].clone()
        self.c, self.t = (T(a) for a in tq.codebook(d, 4)[:2])
        self.plan = tq.encode_plan(T(O.rotation(d, 5).astype(np.float32)))
        self.want = [tuple(x.clone() for x in tq.encode(q, None, self.c, self.t, 4, plan=self.plan)) for q in self.Q]
        self.ws = torch.empty(tq.encode_workspace(n, d, 4), dtype=torch.uint8, device="cuda")
        self.out = torch.empty(n, d // 2, dtype=torch.uint8, device="cuda"), torch.empty(n, device="cuda")
        torch.cuda.synchronize()

    def run(self, stream):
        self.tq.encode(self.q, None, self.c, self.t, 4, "norm", *self.out, stream=stream, plan=self.plan,
                       workspace=self.ws)

    check = Search.check


def _case(cuda_lib, route):
    import torch
    return torch, Encode(cuda_lib, torch) if route == "encode" else Search(cuda_lib, torch, route)


@pytest.mark.parametrize("route", [*ROUTES, "encode"], ids=str)
def test_back_to_back_and_captured(cuda_lib, route):
    torch, case = _case(cuda_lib, route)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        for b in (0, 1, 1, 0, 1):
            case.q.copy_(case.Q[b])
            case.run(side)
            case.run(side)
            side.synchronize()
            case.check(b)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            case.run(side)
            case.run(side)
        for b in (0, 1, 0):
            case.q.copy_(case.Q[b])
            for x in case.out:
                x.fill_(0)
            graph.replay()
            side.synchronize()
            case.check(b)


def test_from_several_threads(cuda_lib):
    import torch
    cases = [Search(cuda_lib, torch, r) for r in ROUTES] + [Encode(cuda_lib, torch)]
    errors = []

    def work(case):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                for b in (0, 1) * 4:
                    case.q.copy_(case.Q[b])
                    case.run(stream)
                    stream.synchronize()
                    case.check(b)
        except BaseException as e:  # noqa: BLE001 (reported by the main thread)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(c,)) for c in cases]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
