"""The GPU-assisted build encodes in the host build's float arithmetic but for the centroids' norms,
which the host compiler of the device code may take by fused multiply-adds: its codes are the host
build's, except where two centroids are nearer to each other in distance than the rounding of
those distances."""
import numpy as np
import pytest

from oracle.codec import pq_decode, splits
from paper_1804_09996_gb300 import datagen as dg
from paper_1804_09996_gb300 import lc

pytestmark = pytest.mark.gpu


def near_ties(x, C, M, a, b):
    """Checks that where codes a and b of x differ, their centroids tie within the rounding of
    ||c||^2 - 2 <x, c> in FP32: each of the two sums of L products is off by at most L + 1 roundings
    of the sum of its terms' magnitudes.  Returns the number of differing codes."""
    x, C = x.astype(np.float64), C.astype(np.float64)
    off, ln = splits(x.shape[1], M)
    rows, subs = np.nonzero(a != b)
    for i, j in zip(rows, subs):
        s = slice(off[j], off[j] + ln[j])
        score, err = [], 0.0
        for code in (a[i, j], b[i, j]):
            c = C[code, s]
            score.append((c * c - 2 * x[i, s] * c).sum())
            err += 2 * (ln[j] + 1) * 2.0**-24 * (c * c + np.abs(2 * x[i, s] * c)).sum()
        assert abs(score[0] - score[1]) <= err, (i, j, score, err)
    return len(rows)


@pytest.mark.parametrize("d", [96, 128, 64, 100, 41])
def test_codes_are_the_host_builds_up_to_near_ties(d):
    xt = dg.gaussian_mixture(2000, d, 16, stream=dg.STREAM_TRAIN)
    xb = dg.gaussian_mixture(1500, d, 16, stream=dg.STREAM_BASE)
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
    assert np.array_equal(host["C1"], dev["C1"]) and np.array_equal(host["C2"], dev["C2"])
    n1 = near_ties(xb, host["C1"], 16, host["codes1"], dev["codes1"])
    same1 = (host["codes1"] == dev["codes1"]).all(1)
    res = xb - pq_decode(host["codes1"], host["C1"], 16).astype(np.float32)
    n2 = near_ties(res[same1], host["C2"], 16, host["codes2"][same1], dev["codes2"][same1])
    assert n1 + n2 <= 4                            # of 48,000 codes
