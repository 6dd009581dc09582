"""The small-batch tensor-core scan of 4-bit codes (k_scan_tm).

Below 16 queries it is the first half of an exact search: the scan keeps the
vectors whose upper score bounds are best and k_rescore takes the lookup
scan's float32 score of those, so ids and scores have to be the lookup scan's
bit for bit, also where the bounds cannot settle a query (ties, duplicates) or
do not cover the values (scales that are not finite) and the lookup scan runs
after all.  From 16 to 32 queries its scores are fp16 products like the
batched scan's and are checked against the oracle within its tolerance."""
import numpy as np
import pytest

import oracle as O
from paper_2607_16973_gb300 import synth
from parity import TOL_LUT, TOL_MMA, check_topk
from test_gpu_fold import _cb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tdev(cuda_lib):
    import torch
    dev = torch.device("cuda:0")
    return torch, (lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev))


def _data(n, d, nq, seed):
    packed = synth.random_codes(n, d // 2, seed=seed)
    scale = synth.random_scales(n, seed=seed)
    R = O.rotation(d, 5).astype(np.float32)
    Q = synth.gaussian_rows(nq, d, seed=seed)
    Q /= np.linalg.norm(Q, axis=1, keepdims=True)
    return packed, scale, R, Q


def _search(tq, torch, path, *a, **kw):
    tq.set_search_path(path)
    try:
        ids, sc = tq.search(*a, **kw)
        torch.cuda.synchronize()
    finally:
        tq.set_search_path("auto")
    return ids.cpu().numpy(), sc.cpu().numpy()


# rows x d x queries of 2^24 and more (2^27 for k > 16) take the tensor-core scan
@pytest.mark.parametrize("d,n,nq,k", [
    (256, 65_537, 1, 1),       # one raw code tile per vector tile, one row past a tile
    (256, 40_000, 15, 32),     # the largest batch and k
    (512, 60_000, 9, 16),
    (768, 25_001, 1, 10),
    (1536, 11_000, 1, 10),     # fewer tiles than SMs
    (1536, 70_001, 3, 7),      # four tiles per CTA
    (2048, 20_000, 8, 5),      # the largest d
])
def test_exact_search_is_the_lookup_scan(cuda_lib, tdev, d, n, nq, k):
    torch, T = tdev
    tq = cuda_lib
    packed, scale, R, Q = _data(n, d, nq, seed=d + nq)
    scale[::97] *= -1.0
    scale[5] = 0.0
    c32, _ = _cb(d)
    a = (T(Q), T(R), T(c32), 4, T(packed), T(scale), k)
    ids, sc = _search(tq, torch, "auto", *a)
    ids_l, sc_l = _search(tq, torch, "lut", *a)
    assert np.array_equal(ids, ids_l) and np.array_equal(sc, sc_l)
    ref = O.search(Q, R, c32, 4, packed, scale, k, d)
    check_topk(ids, sc, ref.ids, ref.scores64, np.ones_like(ref.scores64, bool), k, TOL_LUT)


def _all_equal(packed, scale, Q, c32):
    packed[:], scale[:] = packed[7], scale[7]


def _many_copies(packed, scale, Q, c32):  # more copies of a vector than a list holds, in one vector tile
    packed[256:320], scale[256:320] = packed[7], scale[7]
    Q[:] = Q[0]


def _infinite_scale(packed, scale, Q, c32):
    scale[100] = np.inf


def _nan_scale(packed, scale, Q, c32):
    scale[100] = np.nan


def _zero_query(packed, scale, Q, c32):
    Q[1] = 0.0


def _huge_query(packed, scale, Q, c32):
    Q *= np.float32(1e25)


def _nan_query(packed, scale, Q, c32):
    Q[1, 3] = np.nan


def _wide_scales(packed, scale, Q, c32):
    scale *= np.exp(synth.gaussian_rows(1, len(scale), seed=3)[0] * 4).astype(np.float32)


def _infinite_centroid(packed, scale, Q, c32):
    c32[15] = np.inf


@pytest.mark.parametrize("change", [_all_equal, _many_copies, _infinite_scale, _nan_scale, _zero_query, _huge_query,
                                    _nan_query, _wide_scales, _infinite_centroid])
def test_exact_search_on_odd_values(cuda_lib, tdev, change):
    torch, T = tdev
    tq = cuda_lib
    d, n, nq, k = 512, 20_000, 3, 10
    packed, scale, R, Q = _data(n, d, nq, seed=11)
    c32 = _cb(d)[0].copy()
    change(packed, scale, Q, c32)
    a = (T(Q), T(R), T(c32), 4, T(packed), T(scale), k)
    ids, sc = _search(tq, torch, "auto", *a)
    ids_l, sc_l = _search(tq, torch, "lut", *a)
    assert np.array_equal(ids, ids_l) and np.array_equal(sc, sc_l, equal_nan=True)


def test_exact_search_keeps_the_sign_of_zero(cuda_lib, tdev):
    """Rows of scale 0 score 0 or -0, by the sign of their product, and rank by
    id among them: the best results here, all other scores being negative."""
    torch, T = tdev
    tq = cuda_lib
    d, n, k = 512, 40_000, 8
    packed, scale, R, Q = _data(n, d, 1, seed=61)
    c32, _ = _cb(d)
    dot = c32.astype(np.float64)[O.unpack(packed, d, 4)] @ (R.astype(np.float64) @ Q[0])
    scale = (-np.abs(scale) * np.sign(dot)).astype(np.float32)
    zero = np.concatenate([np.nonzero(dot > 0)[0][100:500:100], np.nonzero(dot < 0)[0][100:400:100]])
    scale[zero] = 0.0
    a = (T(Q), T(R), T(c32), 4, T(packed), T(scale), k)
    assert tq.search_kernel(1, n, d, 4, k) == "k_scan_tm (exact)"
    ids, sc = _search(tq, torch, "auto", *a)
    ids_l, sc_l = _search(tq, torch, "lut", *a)
    assert np.array_equal(ids[0, :7], np.sort(zero)) and np.signbit(sc_l[0, :7]).sum() == 3
    assert np.array_equal(ids, ids_l) and np.array_equal(sc.view(np.int32), sc_l.view(np.int32))


def test_exact_search_with_deleted_rows_and_calibration(cuda_lib, tdev):
    torch, T = tdev
    tq = cuda_lib
    d, n, nq, k = 1024, 30_000, 5, 10
    packed, scale, R, Q = _data(n, d, nq, seed=21)
    c32, _ = _cb(d)
    mu = (synth.gaussian_rows(1, d, seed=4)[0] * 0.01).astype(np.float32)
    a_ = np.exp(synth.gaussian_rows(1, d, seed=5)[0] * 0.2).astype(np.float32)
    m = tq.IdMap(n)
    m.add(np.arange(n, dtype=np.uint64) + 10**9)
    first, _ = _search(tq, torch, "lut", T(Q), T(R), T(c32), 4, T(packed), T(scale), k, idmap=m, calib=(T(mu), T(a_)))
    m.remove(first[:, ::2].reshape(-1).view(np.uint64))  # half of what would be found
    args = (T(Q), T(R), T(c32), 4, T(packed), T(scale), k)
    got = _search(tq, torch, "auto", *args, idmap=m, calib=(T(mu), T(a_)))
    want = _search(tq, torch, "lut", *args, idmap=m, calib=(T(mu), T(a_)))
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    assert not set(got[0].reshape(-1).tolist()) & set(first[:, ::2].reshape(-1).tolist())


@pytest.mark.parametrize("d,n,nq,k", [
    (256, 1, 16, 3),          # one row, k - 1 empty slots
    (256, 129, 17, 1),        # one row past a tile, the wider query block
    (1536, 3_000, 32, 32),    # the largest batch and k
    (2048, 20_001, 20, 5),    # the largest d: two raw code stages
])
def test_fp16_batches(cuda_lib, tdev, d, n, nq, k):
    torch, T = tdev
    tq = cuda_lib
    packed, scale, R, Q = _data(n, d, nq, seed=d + nq)
    c32, _ = _cb(d)
    ids, sc = _search(tq, torch, "auto", T(Q), T(R), T(c32), 4, T(packed), T(scale), k)
    ref = O.search(Q, R, c32, 4, packed, scale, k, d)
    check_topk(ids, sc, ref.ids, ref.scores64, np.ones_like(ref.scores64, bool), k, TOL_MMA)


def test_fp16_batch_filtered(cuda_lib, tdev):
    torch, T = tdev
    tq = cuda_lib
    d, n, nq, k = 512, 9_001, 24, 10
    packed, scale, R, Q = _data(n, d, nq, seed=31)
    c32, _ = _cb(d)
    tenants, values = synth.zipf_tenants(n, 100)
    off, ids_allowed = synth.allowlists(synth.query_sources(n, nq), tenants, values)
    flt = tq.Filter(T(tenants.view(np.int32)), block=64)
    ids, sc = _search(tq, torch, "auto", T(Q), T(R), T(c32), 4, T(packed), T(scale), k, filter=flt, allow_off=T(off),
                      allow_tenants=T(ids_allowed.view(np.int32)))
    allowed = np.stack([np.isin(tenants, ids_allowed[off[i]:off[i + 1]]) for i in range(nq)])
    ref = O.search(Q, R, c32, 4, packed, scale, k, d, tenant_ids=tenants, allow_off=off, allow_ids=ids_allowed)
    check_topk(ids, sc, ref.ids, ref.scores64, allowed, k, TOL_MMA)


@pytest.mark.parametrize("order", ["interleaved", "sorted"])
@pytest.mark.parametrize("block", [32, 64])
def test_exact_search_filtered(cuda_lib, tdev, order, block):
    """Tiles no query allows are passed over; lists of one tenant, of five, of
    more than a warp looks up, with ids the corpus does not have, and empty."""
    torch, T = tdev
    tq = cuda_lib
    d, n, nq, k = 512, 60_001, 6, 10
    packed, scale, R, Q = _data(n, d, nq, seed=41)
    c32, _ = _cb(d)
    tenants, values = synth.zipf_tenants(n, 100)
    if order == "sorted":
        tenants = np.sort(tenants)
    lists = [values[:1], values[50:55], values[10:43], values[60:92], np.append(values[99:], [5, 7]).astype(np.uint32),
             values[:0]]
    off = np.cumsum([0] + [len(v) for v in lists]).astype(np.int64)
    ten = np.concatenate(lists).astype(np.uint32)
    flt = tq.Filter(T(tenants.view(np.int32)), block=block)
    a = (T(Q), T(R), T(c32), 4, T(packed), T(scale), k)
    kw = dict(filter=flt, allow_off=T(off), allow_tenants=T(ten.view(np.int32)))
    ids, sc = _search(tq, torch, "auto", *a, **kw)
    ids_l, sc_l = _search(tq, torch, "lut", *a, **kw)
    assert np.array_equal(ids, ids_l) and np.array_equal(sc, sc_l)
    allowed = np.stack([np.isin(tenants, v) for v in lists])
    ref = O.search(Q, R, c32, 4, packed, scale, k, d, tenant_ids=tenants, allow_off=off, allow_ids=ten)
    check_topk(ids, sc, ref.ids, ref.scores64, allowed, k, TOL_LUT)


def test_profile_events_cover_the_whole_exact_scan(cuda_lib, tdev):
    """The events stand around the bounding scan, the rescoring and the gated
    lookup scan.  One scale the bounds do not cover opens the gate, so between
    them lies more than the lookup scan alone takes."""
    torch, T = tdev
    tq = cuda_lib
    d, n = 1536, 200_000
    packed, scale, R, Q = _data(n, d, 1, seed=51)
    scale[100] = np.nan
    a = (T(Q), T(R), T(_cb(d)[0]), 4, T(packed), T(scale), 10)
    ms = {}
    for path in ("lut", "auto"):
        times = []
        for _ in range(7):
            ev = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            tq.profile_events(*ev)
            try:
                _search(tq, torch, path, *a)
            finally:
                tq.profile_events(None, None)
            times.append(ev[0].elapsed_time(ev[1]))
        ms[path] = sorted(times)[3]
    assert ms["auto"] > 1.3 * ms["lut"], ms


def test_exact_search_filtered_without_a_tile(cuda_lib, tdev):
    """Allowlists that name no tenant of the corpus: no CTA has a tile to scan."""
    torch, T = tdev
    tq = cuda_lib
    d, n, nq, k = 512, 60_001, 6, 10
    packed, scale, R, Q = _data(n, d, nq, seed=43)
    tenants, values = synth.zipf_tenants(n, 100)
    flt = tq.Filter(T(tenants.view(np.int32)), block=64)
    assert tq.search_kernel(nq, n, d, 4, k, filtered=True) == "k_scan_tm (exact)"
    none = np.setdiff1d(np.arange(200, dtype=np.uint32), values)[:40]
    for lists in ([none[:0]] * nq, [none[:2], none[:0], none[2:3], none, none[5:9], none[:1]]):
        off = np.cumsum([0] + [len(v) for v in lists]).astype(np.int64)
        ten = np.append(np.concatenate(lists), 1).astype(np.uint32)  # (never an empty tensor)
        ids, sc = _search(tq, torch, "auto", T(Q), T(R), T(_cb(d)[0]), 4, T(packed), T(scale), k, filter=flt,
                          allow_off=T(off), allow_tenants=T(ten.view(np.int32)))
        assert np.all(ids == -1) and np.all(np.isneginf(sc))


@pytest.mark.parametrize("d", [256, 2048])
@pytest.mark.parametrize("nq", [16, 32])
def test_accumulation_error_the_bounds_allow(cuda_lib, tdev, d, nq):
    """The exact search's bound gives the MMAs' float32 accumulation an error of
    d * 2^-23 of sum |q c|.  Here every operand is an fp16 number, so the fp16
    search's scores are off by that error alone: products far apart in
    magnitude, whose small ones are cut when aligned to the large."""
    torch, T = tdev
    tq = cuda_lib
    rng = np.random.default_rng(d)
    mag = np.array([2.0 ** -13, 2.0 ** -12, 1.5 * 2.0 ** -12, 2.0 ** -9, 2.0 ** -5, 0.25, 1.0, 1.9990234375])
    c = np.sort(np.concatenate([-mag, mag])).astype(np.float32)
    n = 32
    codes = rng.integers(0, 16, (n, d))
    small, one = 9, 14                       # codes of 2^-12 and 1
    codes[:8] = small
    codes[0, 0] = codes[1, d - 1] = codes[2, d // 2] = codes[3, ::16] = codes[4, 15::16] = one
    codes[5, ::2] = 15 - small               # -2^-12 between them: the cut sums have opposite signs
    codes[5, 1] = one
    Q = np.where(rng.random((nq, d)) < 0.5, rng.choice(mag, (nq, d)), rng.uniform(-1, 1, (nq, d)).astype(np.float16))
    Q[:4] = 2.0 ** -12
    Q[0, 0] = Q[1, d - 1] = Q[2, d // 2] = 1.0
    Q[3, ::16] = 1.0
    Q[4], Q[5] = 1.0, np.where(np.arange(d) % 3 == 0, -1.0, 1.0)
    Q = Q.astype(np.float32)
    assert np.array_equal(Q, Q.astype(np.float16)) and np.array_equal(c, c.astype(np.float16))
    assert tq.search_kernel(nq, n, d, 4, n) == "k_scan_tm"
    ids, sc = _search(tq, torch, "auto", T(Q), T(np.eye(d, dtype=np.float32)), T(c), 4,
                      T(O.pack(codes.astype(np.uint8), 4)), None, n)
    rec = c.astype(np.float64)[codes]
    exact = np.take_along_axis(Q.astype(np.float64) @ rec.T, ids, axis=1)
    total = np.take_along_axis(np.abs(Q.astype(np.float64)) @ np.abs(rec).T, ids, axis=1)
    share = np.abs(sc - exact) / (d * 2.0 ** -23 * total)
    assert share.max() <= 1.0, share.max()
