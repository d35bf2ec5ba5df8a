"""The careful passes at the edges of how their lists are dealt to the warps:
one listed track or seed, one per warp, one more than there are warps, several
per warp.  With the loose prior below every track and seed is listed (the
steps over the seed's hits then run in double); without it the listed ones are
the loopers near their largest radius, taken on from where the FP32 passes
stopped.  Tolerances are those of the parity tests.
"""
import dataclasses

import numpy as np
import pytest

import oracle
from kfhelp import audit_mismatch, cov_close, found_cov_close, param_close, tracker_for
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


def _loopers(n):
    """The n tracks of lowest pT of many: most of them listed, many of them with double-precision steps."""
    b = make_batch("c3", tracks=12 * n + 200)
    sel = np.sort(np.argsort(-np.abs(b.params[3]))[:n])
    return dataclasses.replace(b, params=np.ascontiguousarray(b.params[:, sel]), cov=np.ascontiguousarray(b.cov[:, sel]),
                               seed_hits=np.ascontiguousarray(b.seed_hits[:, sel]), seed_sim=b.seed_sim[sel],
                               seed_off=np.array([0, n], np.int32))


@pytest.mark.parametrize("stride", [1, 4])
@pytest.mark.parametrize("n", [1, 33, 153, 1500])
def test_careful_adjoint_list_sizes(n, stride):
    """Gradients of loopers, norm-wise within the 1e-3 of the adjoint's parity test."""
    from paper_1906_11744_gb300 import KF_FIT_GIVEN
    b = _loopers(n)
    lists, nh = true_hit_lists(b, 0, b.det.n_layers)
    lists, nh = lists[b.seed_sim], nh[b.seed_sim]
    t = tracker_for(b, ckpt_stride=stride)
    t.fit_tracks(KF_FIT_GIVEN, lists, nh)
    g_align = np.zeros((b.det.n_layers, 2), np.float32)
    g_hits = np.zeros((b.n_hits, 3), np.float32)
    g_seed = np.zeros((6, n), np.float32)
    t.fit_adjoint(g_align, g_hits, g_seed)
    ok = t.get_fit()["status"] == 0
    t.close()
    assert ok.mean() >= 0.99
    x, y, z, lay = b.event_hits(0)
    _, ga, gh, gs, _ = oracle.fit_grad(b.det, b.params[:, ok], b.cov[:, ok], lists[ok], nh[ok], x, y, z, lay, b.align)
    for g, ref in ((g_align, ga), (g_hits, gh), (g_seed[:, ok].T, gs)):
        assert np.abs(g - ref).max() < 1e-3 * np.abs(ref).max()


@pytest.mark.parametrize("cap", [0, 1])
@pytest.mark.parametrize("n,loose,holes,cands", [(1, True, 3, 6), (40, True, 3, 4), (900, True, 3, 10),
                                                 (9000, False, 3, 6), (9000, False, 0, 10), (9000, False, 1, 16)])
def test_careful_finding(n, loose, holes, cands, cap):
    """Seeds given up by the main pass, with (cap 0) and without a record of
    their search: lists of a few seeds and of more than there are warps, and
    candidates without holes left, which stop on the surface with the state
    before it.  Hit lists and work counters equal the oracle's where the two
    agree on every seed looked at: those that meet a near-tangent crossing."""
    b = make_batch("c1", tracks=n)
    if loose:
        for i in range(6):
            b.cov[i * 6 - i * (i - 1) // 2] = LOOSE_VAR[i]
    t = tracker_for(b, max_cands=cands, max_holes=holes, find_regcap=cap)
    t.find_tracks()
    g = t.counters()
    trk = t.get_tracks()
    t.close()
    assert g["redone"] == b.n_seeds if loose else 1 <= g["redone"] < b.n_seeds
    # the low-pT tail: every seed that can meet a tangent crossing inside the barrel
    sel = np.arange(b.n_seeds) if loose else np.argsort(-np.abs(b.params[3]))[:max(100, b.n_seeds // 25)]
    from concurrent.futures import ThreadPoolExecutor
    with ThreadPoolExecutor(8) as ex:
        ref = list(ex.map(lambda s: oracle.find_event(b, 0, max_cands=cands, max_holes=holes, seeds=(int(s), int(s) + 1)),
                          sel))
    same = np.array([np.array_equal(trk["hits"][s], r["hits"][0]) for s, r in zip(sel, ref)])
    for s, r in zip(sel[~same], [r for r, k in zip(ref, same) if not k]):
        ok, kind, rel = audit_mismatch(b, 0, int(s), trk["hits"][s], r["hits"][0])
        assert ok, (int(s), kind, rel)
    assert same.mean() >= 0.98
    if loose and same.all():
        for k in ("steps", "updates", "holes"):
            assert abs(g[k] - sum(r["counters"][k] for r in ref)) <= 1e-3 * g[k]
    p = np.concatenate([r["p"] for r in ref])[same]
    C = np.concatenate([r["C"] for r in ref])[same]
    okp, ep = param_close(trk["params"].T[sel][same], p)
    okc, ec = found_cov_close(trk["cov"].T[sel][same], C, p)
    assert okp.all(), ep
    assert okc.all(), ec
