"""Device-side selection and linking of the GPU-assisted build over vector dimensions: the
compiled widths (96, 128), a multiple of eight, and dimensions that leave a remainder after the
groups of eight the distance is summed in.  The decoded-to-decoded arithmetic is the host
build's, so the rows are the host build's except where an FP32 search distance resolved a
near-tie the other way (the bound of the GPU build tests)."""
import numpy as np
import pytest

from paper_1804_09996_gb300 import datagen as dg
from paper_1804_09996_gb300 import lc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [96, 128, 64, 100, 41])
def test_rows_equal_the_host_builds(d):
    n = 1500
    xt = dg.gaussian_mixture(2000, d, 16, stream=dg.STREAM_TRAIN)
    xb = dg.gaussian_mixture(n, d, 16, stream=dg.STREAM_BASE)
    out = []
    for g in (0, 1):
        h = lc.lc_create(lc.lc_default_params(d, 16, 16, use_opq=0, kmeans_iters=4, beta_iters=1, beta_train_n=500,
                                              batch_max=200, build_gpu=g))
        try:
            lc.lc_train(h, xt)
            lc.lc_add(h, xb)
            out.append(lc.lc_export(h, d, 16, 16))
        finally:
            lc.lc_free(h)
    host, dev = out
    assert (host["adj0"] == dev["adj0"]).all(1).mean() > 0.95
    assert (host["adj0"] >= 0).sum(1).max() == 32                # rows that the heuristic shrank are among them
