"""The device-side search of Eq. 14 and the warp tables of Eqs. 11-12 where they can go wrong: targets
at and outside the ends, tied, zero and infinite scores, few tokens, one token making up the whole
corpus, more distinct tokens than a warp's table holds, lengths that do not fill a warp."""
import numpy as np
import pytest
import torch

from tests import _parity as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sats():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2607_08991_gb300 import sats as s
    return s


def _tau_ref(score, ids, r_tar):
    """Every candidate in increasing order; the first of the nearest wins (0 before the scores, +inf last)."""
    sc = score[ids].astype(np.float64)
    cand = np.unique(np.concatenate([[0.0], sc[(sc > 0) & np.isfinite(sc)], [np.inf]]))
    m = max(1, ids.size)
    R = np.array([np.count_nonzero(sc < c) / m for c in cand])
    k = int(np.argmin(np.abs(R - r_tar)))
    return cand[k], R[k]


@pytest.mark.parametrize("V,m", [(1, 1), (3, 2), (40, 33), (5000, 4999), (200000, 60000)])
@pytest.mark.parametrize("kind", ["distinct", "ties", "zeros_and_inf"])
def test_tau(sats, V, m, kind):
    g = np.random.default_rng([V, m, len(kind)])
    score = g.exponential(0.1, V).astype(np.float32)
    if kind == "ties":
        score = (g.integers(0, 4, V) * 0.125).astype(np.float32)
    elif kind == "zeros_and_inf":
        score[::3] = 0.0
        score[1::5] = np.inf
        score[2::7] = -0.0
    ids = np.minimum((V * g.random(m) ** 3).astype(np.int32), V - 1)
    for r in (-0.5, 0.0, 1e-9, 0.25, 1.0 / 3.0, 0.5, 0.99999, 1.0, 2.0):
        tau, R, lut = sats.route_calibrate(P.dev(score), P.dev(ids), r)
        want_tau, want_R = _tau_ref(score, ids, r)
        assert tau == want_tau and R == want_R, (r, tau, want_tau)
        assert np.array_equal(lut.cpu().numpy(), (score >= np.float32(tau)).astype(np.uint8))


@pytest.mark.parametrize("n", [1, 31, 33, 4097, 250001])
@pytest.mark.parametrize("kind", ["one_token", "few", "spread"])
def test_scores(sats, n, kind):
    V = 70001
    g = np.random.default_rng([n, len(kind)])
    ids = {"one_token": np.full(n, V - 1), "few": g.integers(0, 5, n) * 512, "spread": g.integers(0, V, n)}[kind]
    ids = ids.astype(np.int32)
    lb = g.standard_normal(n).astype(np.float32)
    ls = lb + g.standard_normal(n).astype(np.float32)
    d = np.maximum(np.float32(0), ls - lb).astype(np.float64)
    total, count = np.bincount(ids, d, V), np.bincount(ids, minlength=V)
    score = sats.token_scores(P.dev(ids), P.dev(lb), P.dev(ls), V).cpu().numpy()
    assert np.array_equal(np.isinf(score), count == 0)
    seen = count > 0
    # sums of non-negative doubles in any order: n * 2^-53 relative, far below the rounding to fp32
    np.testing.assert_allclose(score[seen], total[seen] / count[seen], rtol=1.2e-7)
