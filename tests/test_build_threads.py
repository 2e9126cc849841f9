"""The insertion's threads: the host build gives the same index whatever their number, in one
call or in several, and for batches too small to hand out (tests of the loops' hand-out; the
index itself is tested in test_host_build.py)."""
import numpy as np
import pytest

from paper_1804_09996_gb300 import datagen as dg
from paper_1804_09996_gb300 import lc


def build(nt, parts, batch_max):
    d = 32
    xt = dg.gaussian_mixture(600, d, 8, stream=dg.STREAM_TRAIN)
    xb = dg.gaussian_mixture(900, d, 8, stream=dg.STREAM_BASE)
    h = lc.lc_create(lc.lc_default_params(d, 16, 8, use_opq=0, kmeans_iters=3, beta_iters=1, beta_train_n=300, n_threads=nt,
                                          batch_max=batch_max))
    try:
        lc.lc_train(h, xt)
        for x in np.array_split(xb, parts):
            lc.lc_add(h, x)
        return lc.lc_export(h, d, 16, 8)
    finally:
        lc.lc_free(h)


@pytest.mark.parametrize("parts,batch_max", [(1, 256), (3, 256), (1, 1)])
def test_any_number_of_threads_gives_the_same_index(parts, batch_max):
    ref = build(1, parts, batch_max)
    for nt in (2, 5, 24):
        got = build(nt, parts, batch_max)
        assert all(np.array_equal(ref[k], got[k]) for k in ("codes1", "codes2", "beta", "B", "adj0", "levels", "upper_adj"))
        assert ref["ep"] == got["ep"]
