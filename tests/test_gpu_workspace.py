"""A workspace kept for a program's largest search serves its smaller ones:
tq_search_workspace does not fall as the batch, k or the filter shrink, over
the sizes at which searches change path or split their work differently."""
import numpy as np
import pytest

import oracle as O
from paper_2607_16973_gb300 import synth
from test_gpu_fold import _cb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def filtered(cuda_lib):
    import torch
    tenants, values = synth.zipf_tenants(20_000, 50)
    return torch, cuda_lib.Filter(torch.from_numpy(tenants.view(np.int32)).cuda(), block=64), values


@pytest.mark.parametrize("d,bits", [(256, 4), (512, 4), (1536, 4), (96, 4), (128, 3), (256, 2), (1536, 8)])
def test_it_grows_with_batch_k_and_filter(cuda_lib, filtered, d, bits):
    tq, (_, flt, _) = cuda_lib, filtered
    n = 20_000
    batches = [*range(1, 36), 64, 127, 128, 129, 200, 256, 257, 300, 512, 513, 1000, 1024, 5000, 38_912, 39_000]
    ks = [1, 5, 8, 16, 17, 20, 32, 33, 50, 64, 65, 100, 256]
    before = {}
    for nq in batches:
        row = [(tq.search_workspace(nq, n, d, bits, k), tq.search_workspace(nq, n, d, bits, k, flt)) for k in ks]
        for k, (plain, with_filter), smaller in zip(ks, row, [(0, 0), *row]):
            assert plain <= with_filter, (nq, k)
            assert plain >= smaller[0] and with_filter >= smaller[1], (nq, k)
            assert plain >= before.get((k, 0), 0) and with_filter >= before.get((k, 1), 0), (nq, k)
            before[k, 0], before[k, 1] = plain, with_filter


@pytest.mark.parametrize("kept,then", [
    ((32, 1, False), (15, 1, False)),    # the exact small-batch search behind a larger batch
    ((15, 20, False), (15, 10, False)),  # its smaller k, for which fewer rows are enough
    ((1, 10, True), (1, 10, False)),     # without the filter
    ((300, 5, False), (256, 5, False)),  # fewer query tiles, more CTAs each
])
def test_a_kept_workspace_serves_a_smaller_search(cuda_lib, filtered, kept, then):
    tq, (torch, flt, values) = cuda_lib, filtered
    n, d = 20_000, 512
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    ws = torch.empty(tq.search_workspace(kept[0], n, d, 4, kept[1], flt if kept[2] else None), dtype=torch.uint8,
                     device="cuda")
    nq, k, _ = then
    Q = T(synth.gaussian_rows(nq, d, seed=2))
    a = (Q, T(O.rotation(d, 5).astype(np.float32)), T(_cb(d)[0]), 4, T(synth.random_codes(n, d // 2, seed=1)),
         T(synth.random_scales(n, seed=1)), k)
    got, want = tq.search(*a, workspace=ws), tq.search(*a)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
