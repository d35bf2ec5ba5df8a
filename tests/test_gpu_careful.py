"""The careful passes at the edges of how their lists are dealt to the warps:
one listed track or seed, one per warp, one more than there are warps, several
per warp.  With the loose prior below every track and seed is listed (the
steps over the seed's hits then run in double); without it the listed ones are
the loopers near their largest radius, taken on from where the FP32 passes
stopped.  Tolerances are those of the parity tests.
"""
import numpy as np
import pytest

import oracle
from kfhelp import cov_close, param_close, tracker_for
from synth import make_batch
from synth.events import true_hit_lists

pytestmark = pytest.mark.gpu

LOOSE_VAR = (1.0, 1.0, 1.0, 1.0, 0.01, 0.01)  # a position prior of 1 cm against 0.01 cm hits


def _batch(n, loose, **kw):
    b = make_batch("c3", tracks=n, **kw)
    if loose:
        for i in range(6):
            b.cov[i * 6 - i * (i - 1) // 2] = LOOSE_VAR[i]
    return b


@pytest.mark.parametrize("loose", [True, False])
@pytest.mark.parametrize("n", [1, 33, 608, 609, 2500])
def test_careful_fit_list_sizes(n, loose):
    from paper_1906_11744_gb300 import KF_FIT_GIVEN
    b = _batch(n, loose)
    lists, nh = true_hit_lists(b, 0, b.det.n_layers)
    lists, nh = lists[b.seed_sim], nh[b.seed_sim]
    t = tracker_for(b)
    t.fit_tracks(KF_FIT_GIVEN, lists, nh)
    fit = t.get_fit()
    t.close()
    x, y, z, lay = b.event_hits(0)
    p, C, c2, st = oracle.fit(b.det, b.params, b.cov, lists, nh, x, y, z, lay, align=b.align)
    assert (fit["status"] == st).mean() >= 0.99
    ok = (st == 0) & (fit["status"] == 0)
    okp, ep = param_close(fit["params"].T[ok], p[ok])
    okc, ec = cov_close(fit["cov"].T[ok], C[ok], p[ok])
    assert okp.all(), ep
    assert okc.all(), ec
