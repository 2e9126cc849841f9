"""Searches at odd dimensions (every kernel's rows and codebooks end off the 16-byte grid) against the
oracle: in small batches, in batches past the tiled rotation's size, from host memory and without
allocation."""
import numpy as np
import pytest

import oracle
from paper_1804_09996_gb300 import lc
from test_gpu_full_walk_splits import index
from test_gpu_order import same
from test_gpu_parity import compare, gpu_search, handle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", [(41, 16, 10), (207, 16, 40)])
def test_parity_odd_dims(split):
    import torch
    ix, xq = index(split)
    h = handle(f"split{split}", ix)
    for beam, shortlist in ((1, 0), (4, 0), (1, -1)):
        ref = oracle.search(ix, xq, 10, 40, beam=beam, shortlist=shortlist)
        got = gpu_search(h, xq, 10, 40, shortlist, beam=beam)
        compare(ref, *got, max_exempt=0.01)                # the oracle: none
        same(got, gpu_search(h, xq, 10, 40, shortlist, device=False, beam=beam))
        big = gpu_search(h, np.tile(xq, (35, 1)), 10, 40, shortlist, beam=beam)
        for a in range(0, len(big[0]), len(xq)):
            same(got, [x[a:a + len(xq)] for x in big])
    q = torch.from_numpy(xq.astype(np.float32)).cuda()
    ids = torch.empty((len(xq), 10), dtype=torch.int32, device="cuda")
    ds = torch.empty((len(xq), 10), dtype=torch.float32, device="cuda")
    st = torch.empty((len(xq), 3), dtype=torch.int32, device="cuda")
    lc.lc_search_walk_noalloc(h, q, len(xq), 10, 40, ids, ds, st, torch.cuda.current_stream())
    same(got, [x.cpu().numpy() for x in (ids, ds, st)])
