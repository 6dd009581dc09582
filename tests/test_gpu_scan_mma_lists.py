"""The batched tensor-core scan's lists and thresholds (k_scan_mma): a first
threshold from the first tile (group maxima, or a bisection for k > 16),
thresholds and list heads shared between the CTAs of a query (several tiles
per CTA), with deleted rows, ties and fewer live rows than k."""
import numpy as np
import pytest

import oracle as O
from paper_2607_16973_gb300 import synth
from parity import TOL_MMA, check_topk

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tdev(cuda_lib):
    import torch
    dev = torch.device("cuda:0")
    return torch, (lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev))


@pytest.mark.parametrize("n,nq,k,bits,dead", [
    (256, 40, 64, 4, 0.0),         # one whole tile
    (255, 33, 20, 2, 0.0),         # a short tile
    (90_001, 40, 20, 4, 0.3),      # three tiles per CTA: heads read at the second; deleted rows
    (90_001, 130, 8, 2, 0.0),      # two query tiles, the smallest k that reads heads
    (60_000, 300, 33, 4, 0.999),   # fewer live rows per CTA than k; heads of rank 3
    (90_001, 40, 7, 4, 0.3),       # the largest k of the kernel for short lists
    (90_001, 130, 1, 3, 0.0),      # its smallest, two query tiles
    (90_001, 40, 7, 8, 0.3),       # 8-bit codes have none: short lists in the general one
])
def test_mma_lists(cuda_lib, tdev, n, nq, k, bits, dead):
    torch, T = tdev
    tq = cuda_lib
    d = 128
    packed = synth.random_codes(n, d * bits // 8, seed=n + k)
    scale = synth.random_scales(n, seed=n)
    packed[n // 2: n // 2 + 40] = packed[0]      # ties, in rank order of the rows
    scale[n // 2: n // 2 + 40] = scale[0]
    R = O.rotation(d, 5).astype(np.float32)
    # (the oracle's own 8-bit codebook takes minutes)
    c32 = O.codebook(d, bits, "beta").centroids32 if bits < 8 else tq.codebook(d, bits)[0]
    Q = synth.gaussian_rows(nq, d, seed=nq)
    Q /= np.linalg.norm(Q, axis=1, keepdims=True)
    m, gone = None, np.zeros(n, bool)
    if dead:
        gone = np.random.default_rng(1).random(n) < dead
        m = tq.IdMap(n)
        m.add(np.arange(n, dtype=np.uint64))
        m.remove(np.nonzero(gone)[0].astype(np.uint64))
    tq.set_search_path("mma")
    try:
        ids, sc = tq.search(T(Q), T(R), T(c32), bits, T(packed), T(scale), k, idmap=m)
        torch.cuda.synchronize()
    finally:
        tq.set_search_path("auto")
    ref = O.search(Q, R, c32, bits, packed, scale, k, d, deleted=gone)
    allowed = np.repeat(~gone[None, :], nq, axis=0)
    check_topk(ids.cpu().numpy(), sc.cpu().numpy(), ref.ids, ref.scores64, allowed, k, TOL_MMA)
