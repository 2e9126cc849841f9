"""The full-decode walk in FP32 over level-1 splits without a compiled width (one to sixteen
coordinates per sub-space, odd dimensions, level-2 splits finer and coarser than level 1's)
against the oracle, in a small batch (teams of warps) and in a larger one: the codebook of level
2 is read for the nodes of a step one after another there."""
import numpy as np
import pytest

import oracle
from paper_1804_09996_gb300 import datagen as dg
from paper_1804_09996_gb300 import lc
from test_gpu_order import same
from test_gpu_parity import compare, gpu_search, handle

SPLITS = [(41, 16, 10), (128, 16, 16), (207, 16, 40), (64, 32, 16), (100, 64, 25)]
_ix = {}


def index(split):
    if split not in _ix:
        d, M1, M2 = split
        xt, xb, xq = (dg.make("mixture", n, d, 32, s) for n, s in ((1000, dg.STREAM_TRAIN), (900, dg.STREAM_BASE),
                                                                    (120, dg.STREAM_QUERY)))
        _ix[split] = oracle.build_index(xt, xb, M1, M2, False, codec_niter=5), xq
    return _ix[split]


@pytest.mark.gpu
@pytest.mark.parametrize("beam", [1, 4])
@pytest.mark.parametrize("split", SPLITS)
def test_parity_full_walk_splits(split, beam):
    ix, xq = index(split)
    h = handle(f"split{split}", ix)
    ref = oracle.search(ix, xq, 10, 40, beam=beam, walk_full=True)
    got = gpu_search(h, xq, 10, 40, 0, beam=beam, walk_full=1)
    compare(ref, *got, max_exempt=0.02)                # the oracle: <= 1.7 %
    big = gpu_search(h, np.tile(xq, (11, 1)), 10, 40, 0, beam=beam, walk_full=1)
    for a in range(0, len(big[0]), len(xq)):
        same(got, [x[a:a + len(xq)] for x in big])
