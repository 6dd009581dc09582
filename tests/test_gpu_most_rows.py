"""Searches over the most rows that are accepted, 2^31 - 2: row and tile
numbers are int in the scans, so the last tile's must not wrap.  The corpus is
one code everywhere but in a few rows near both ends of the row range, which
score higher and have to be found.  (d = 32 and 64 at 2 and 3 bits: 17 to 35 GB.)"""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

N = 2 ** 31 - 2


@pytest.mark.parametrize("bits,d,nq", [
    (2, 32, 1),    # lookup scan, 32 rows a step
    (3, 32, 1),    # bulk-copy ring, whole steps of 4 rows and a rest of 2
    (2, 64, 16),   # batched tensor-core scan, tiles of 256 rows
])
def test_the_last_rows_are_found(cuda_lib, bits, d, nq):
    import torch
    tq = cuda_lib
    rb = d * bits // 8
    if torch.cuda.mem_get_info()[0] < N * rb + (8 << 30):
        pytest.skip("not enough device memory")
    rows = [0, 1, 2 ** 30, N - 300, N - 130, N - 129, N - 34, N - 33, N - 5, N - 2, N - 1]
    codes = torch.zeros((N, rb), dtype=torch.uint8, device="cuda")
    for i, r in enumerate(rows):  # the i-th row: all coordinates but the first i at the largest centroid
        c = np.full((1, d), (1 << bits) - 1, np.uint8)
        c[0, :i] = 0
        codes[r] = torch.from_numpy(O.pack(c, bits)[0]).cuda()
    c32 = torch.from_numpy(O.codebook(d, bits, "beta").centroids32).cuda()
    R = torch.eye(d, device="cuda")
    Q = torch.full((nq, d), 1.0 / np.sqrt(d), device="cuda")
    ids, scores = tq.search(Q, R, c32, bits, codes, None, len(rows))
    torch.cuda.synchronize()
    assert ids.cpu().tolist() == [rows] * nq
    del codes, ids, scores
    torch.cuda.empty_cache()
