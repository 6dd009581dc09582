"""The fp16 tensor-core encoder (tq_encode_planned_ws, k_encode_h) at the sizes
where its work split changes: one row, a row past a panel, fewer items than
SMs (64- and 128-wide chunks, every panel split over CTAs), panels split
between two CTAs, partial last chunks.  Checked against the oracle as the
other encoders are, and against the TF32 encoder (tq_encode_planned): no more
codes off the 64-bit ones than that has."""
import numpy as np
import pytest

import oracle as O
from paper_2607_16973_gb300 import _lib, synth
from parity import check_encode
from test_gpu_encode_tc import _cb, _rate

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tdev(cuda_lib):
    import torch
    dev = torch.device("cuda:0")
    return torch, dev, (lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev))


def _tf32(tq, torch, X, plan, c, t, bits, mode):
    n, d = X.shape
    codes = torch.empty((n, d * bits // 8), dtype=torch.uint8, device=X.device)
    scale = torch.empty(n, device=X.device)
    _lib.check(tq.load().tq_encode_planned(X.data_ptr(), n, d, plan.data_ptr(), c.data_ptr(), t.data_ptr(), bits,
                                           _lib.SCALE_MODES[mode], None, None, codes.data_ptr(), scale.data_ptr(), 0))
    tq.encode_check(plan)
    torch.cuda.synchronize()
    return codes.cpu().numpy(), scale.cpu().numpy()


@pytest.mark.parametrize("n,d,bits,mode", [
    (1, 1024, 4, "norm"),           # one row, the smallest d of 4-bit codes
    (129, 1056, 3, "unbiased"),     # a row past a panel; a partial chunk
    (1_000, 1536, 4, "norm"),      # fewer items than SMs
    (2_500, 1536, 8, "none"),      # 20 panels
    (19_700, 1024, 2, "norm"),     # 154 panels split between CTAs, a partial chunk
])
def test_encode_h_parity(cuda_lib, tdev, n, d, bits, mode):
    torch, dev, T = tdev
    tq = cuda_lib
    X = synth.gaussian_rows(n, d, seed=n + d)
    if n > 3:
        X[3] = 0.0
        X[1] *= 1e-18   # rows far apart in magnitude: each is scaled by its own norm
        X[2] *= 1e15
    R = O.rotation(d, 7).astype(np.float32)
    c32, t32 = _cb(d, bits)
    plan = tq.encode_plan(T(R))
    codes, scale = tq.encode(T(X), None, T(c32), T(t32), bits, mode, plan=plan)
    tq.encode_check(plan)
    torch.cuda.synchronize()
    codes, scale = codes.cpu().numpy(), scale.cpu().numpy()
    enc = O.encode(X, R, c32, t32, bits, mode)
    off = check_encode(codes, scale, X, enc, c32, t32, d, bits, mode, max_rate=_rate(bits))
    codes_t, scale_t = _tf32(tq, torch, T(X), plan, T(c32), T(t32), bits, mode)
    off_t = check_encode(codes_t, scale_t, X, enc, c32, t32, d, bits, mode, max_rate=_rate(bits))
    # half of TF32's accumulation steps: fewer codes off (a handful either way is chance)
    assert off <= off_t + 3 * np.sqrt(off_t + 1)


def test_encode_h_values_out_of_range(cuda_lib, tdev):
    """Rows that are not finite or whose norm overflows come out as from the
    TF32 encoder; a matrix R of another scale is brought into fp16's range."""
    torch, dev, T = tdev
    tq = cuda_lib
    n, d, bits = 300, 1024, 4
    X = synth.gaussian_rows(n, d, seed=3)
    X[10, 5] = np.inf
    X[11, 6] = np.nan
    X[12] *= 1e25      # the norm overflows float32
    X[13] *= 1e-30     # the norm underflows to 0
    R = O.rotation(d, 7).astype(np.float32)
    c32, t32 = _cb(d, bits)
    plan = tq.encode_plan(T(R))
    codes, scale = tq.encode(T(X), None, T(c32), T(t32), bits, "norm", plan=plan)
    codes, scale = codes.cpu().numpy(), scale.cpu().numpy()
    codes_t, scale_t = _tf32(tq, torch, T(X), plan, T(c32), T(t32), bits, "norm")
    odd = [10, 11, 12, 13]
    assert np.array_equal(codes[odd], codes_t[odd])
    assert np.array_equal(scale[odd], scale_t[odd], equal_nan=True)
    Rs = (R * np.float32(3e6)).astype(np.float32)
    plan = tq.encode_plan(T(Rs))
    codes, scale = tq.encode(T(X), None, T(c32), T(t32 * np.float32(3e6)), bits, "norm", plan=plan)
    codes_t, _ = _tf32(tq, torch, T(X), plan, T(c32), T(t32 * np.float32(3e6)), bits, "norm")
    assert np.mean(codes.cpu().numpy()[20:] != codes_t[20:]) < 2e-4


@pytest.mark.parametrize("bits", [2, 4, 8])
@pytest.mark.parametrize("how", ["close", "equal", "infinite"])
def test_encode_h_boundaries_no_cell_separates(cuda_lib, tdev, bits, how):
    """Two boundaries in one lookup cell (close or equal), or a range that is not
    finite: the codes come from the search, as the TF32 encoder's do."""
    torch, dev, T = tdev
    tq = cuda_lib
    n, d = 120, 1024
    X, R = synth.gaussian_rows(n, d, seed=5), O.rotation(d, 7).astype(np.float32)
    c32, t32 = (a.copy() for a in tq.codebook(d, bits)[:2])
    m = len(t32) // 2
    if how == "infinite":
        t32[0], t32[-1] = -np.inf, np.inf
    else:
        t32[m] = t32[m - 1] + (np.float32(1e-6) if how == "close" else 0)
    plan = tq.encode_plan(T(R))
    codes, scale = tq.encode(T(X), None, T(c32), T(t32), bits, "norm", plan=plan)
    codes, scale = codes.cpu().numpy(), scale.cpu().numpy()
    codes_t, scale_t = _tf32(tq, torch, T(X), plan, T(c32), T(t32), bits, "norm")
    a, b = (O.unpack(x, d, bits).astype(np.int64) for x in (codes, codes_t))
    # where they differ the coordinate lies next to a boundary: a cell away, or two across the narrow one
    assert np.abs(a - b).max() <= (2 if how != "infinite" else 1) and np.mean(a != b) < (1e-3 if bits == 8 else 2e-4)
    same = (a == b).all(axis=1)
    assert same.any() and np.allclose(scale[same], scale_t[same], rtol=2e-6)
    y = (X.astype(np.float64) / np.linalg.norm(X, axis=1, keepdims=True)) @ R.T.astype(np.float64)
    want = np.searchsorted(t32.astype(np.float64), y)  # boundaries below y
    off = a != want
    near = np.abs(y[..., None] - t32[None, None].astype(np.float64)).min(axis=-1) < 1e-5
    assert np.all(near[off])


def test_encode_h_workspace(cuda_lib, tdev):
    """A kept workspace is reused, one that is too small is refused."""
    torch, dev, T = tdev
    tq = cuda_lib
    n, d, bits = 700, 1024, 4
    R = O.rotation(d, 7).astype(np.float32)
    c32, t32 = _cb(d, bits)
    plan = tq.encode_plan(T(R))
    ws = torch.empty(tq.encode_workspace(n, d), dtype=torch.uint8, device=dev)
    X = [T(synth.gaussian_rows(m, d, seed=m)) for m in (n, 130)]
    want = [tq.encode(x, None, T(c32), T(t32), bits, plan=plan) for x in X]
    for x, (codes, scale) in zip(X, want):
        got = tq.encode(x, None, T(c32), T(t32), bits, plan=plan, workspace=ws)
        assert torch.equal(got[0], codes) and torch.equal(got[1], scale)
    with pytest.raises(tq.TQError):
        tq.encode(X[0], None, T(c32), T(t32), bits, plan=plan, workspace=ws[:-1])
    assert tq.encode_workspace(n, 96) is None


def test_no_memory_for_the_workspace(cuda_lib, tdev, monkeypatch):
    """The encoder is the caller's choice, not the free memory's: a workspace
    that cannot be allocated is an error; without one on request, the codes are
    the TF32 encoder's."""
    torch, dev, T = tdev
    tq = cuda_lib
    n, d, bits = 300, 1024, 4
    c, t = (T(a) for a in _cb(d, bits))
    X, plan = T(synth.gaussian_rows(n, d, seed=9)), tq.encode_plan(T(O.rotation(d, 7).astype(np.float32)))
    out = torch.empty((n, d * bits // 8), dtype=torch.uint8, device=dev), torch.empty(n, device=dev)

    def no_memory(*a, **kw):
        raise torch.OutOfMemoryError("no memory")

    with monkeypatch.context() as m:
        m.setattr(torch, "empty", no_memory)
        with pytest.raises(torch.OutOfMemoryError):
            tq.encode(X, None, c, t, bits, "norm", *out, plan=plan)
        codes, scale = tq.encode(X, None, c, t, bits, "norm", *out, plan=plan, workspace=False)
    codes_t, scale_t = _tf32(tq, torch, X, plan, c, t, bits, "norm")
    assert np.array_equal(codes.cpu().numpy(), codes_t) and np.array_equal(scale.cpu().numpy(), scale_t)


@pytest.mark.parametrize("d,bits", [(384, 3), (992, 4), (736, 8)])
def test_below_its_range_the_tf32_encoder_runs(cuda_lib, tdev, d, bits):
    torch, dev, T = tdev
    tq = cuda_lib
    X, R = T(synth.gaussian_rows(500, d, seed=d)), O.rotation(d, 7).astype(np.float32)
    c32, t32 = (T(a) for a in tq.codebook(d, bits)[:2])
    plan = tq.encode_plan(T(R))
    codes, scale = tq.encode(X, None, c32, t32, bits, plan=plan)
    codes_t, scale_t = _tf32(tq, torch, X, plan, c32, t32, bits, "norm")
    assert np.array_equal(codes.cpu().numpy(), codes_t) and np.array_equal(scale.cpu().numpy(), scale_t)
