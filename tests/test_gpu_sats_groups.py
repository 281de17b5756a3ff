"""Eq. 6 in groups of candidates, and the calibration with and without its blocks' inputs kept: sizes at
which the candidates of a block do not fit one group, and at which what would be kept passes 1 GiB.  The shares in
the calibration's table are the accurate gate activations', its errors those of separate evaluations, and
Eq. 6 of a few inputs is the definition's."""
import numpy as np
import pytest
import torch

from paper_2607_08991_gb300 import inputs
from tests import _parity as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sats():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2607_08991_gb300 import sats as s
    return s


@pytest.mark.parametrize("H,N,C,K0,K1", [
    (64, 264, 5, 36, 33),        # more candidates than a group holds
    (72, 261, 5, 12, 5),         # rows of a that no vector load can take
    (16, 40000, 1700, 8, 2),     # chunks of inputs; 1.1 GB of what the blocks' errors are formed from are not kept
])
def test_table_equals_separate_evaluations(sats, H, N, C, K0, K1):
    layers, gains = [], []
    for l in range(2):
        w = inputs.mlp_weights(H, N, layer=l, std=0.2, seed=1300)
        layers.append(sats.Layer(P.dev_u16(w.Wg), P.dev_u16(w.Wu), P.dev_u16(w.Wd)))
        gains.append(P.dev(inputs.norm_weight(H, layer=l)))
    x = P.dev(inputs.activations_f32(C, H, seed=1301))
    r = sats.sats_calibrate(layers, gains, 1e-5, x, 0.5, K0=K0, K1=K1, guardrail=True)
    n = torch.empty_like(x)
    sats.rmsnorm(x, gains[0], 1e-5, n)
    t, err, sp = (np.asarray(v[0]) for v in r["table"])
    # the shares: exactly those of the accurate gate activations, from which the thresholds come
    a = torch.empty(C, N, device="cuda")
    sats.gate_act_f32(layers[0], n, a)
    a = a.abs_()
    np.testing.assert_allclose(sp, [float((a < float(v)).double().mean()) for v in t], rtol=0, atol=1e-12)
    # the errors: those of separate evaluations, whose masks are the same ones.  Groups of other sizes take other
    # accumulator chains, common to both norms but for a few per cent of their 1e-5.
    one, sp1 = sats.layer_err(layers[0], n, [float(v) for v in t], eps=1e-6)
    np.testing.assert_allclose(sp, sp1, rtol=0, atol=1e-15)
    np.testing.assert_allclose(err, one, rtol=1e-5)
    assert (np.diff(sp[np.argsort(t)]) >= 0).all()
    for l in layers:
        l.close()


def test_ends_of_the_range(sats, oracle):
    """Outputs whose squares leave fp32's range, a candidate that drops nothing and one that drops all."""
    H, N, C = 64, 40, 4
    w = inputs.mlp_weights(H, N, std=0.3, seed=1310)
    x = inputs.activations_f32(C, H, seed=1311)
    for scale in (1.0, 2.0 ** 70, 2.0 ** -90):
        wd = inputs.to_bf16_bits((inputs.bf16_bits_to_f32(w.Wd) * np.float32(scale)).astype(np.float32))
        layer = sats.Layer(P.dev_u16(w.Wg), P.dev_u16(w.Wu), P.dev_u16(wd))
        a = np.abs(oracle.gate_act(x.astype(np.float64), w.Wg))
        v = np.sort(a.ravel())
        k = int(np.argmax(np.diff(v[40:120]))) + 40
        ts = [0.0, float(np.float32(0.5 * (v[k] + v[k + 1]))), float("inf")]
        err, sp = sats.layer_err(layer, P.dev(x), ts, eps=0.0)
        e_ref, s_ref = oracle.layer_err(x.astype(np.float64), w.Wg, w.Wu, wd, ts, eps=0.0)
        assert err[0] == 0.0 and abs(err[2] - 1.0) < 1e-5
        np.testing.assert_allclose(err, e_ref, rtol=1e-4, atol=1e-7)
        np.testing.assert_allclose(sp, s_ref, rtol=0, atol=1e-12)
        layer.close()
