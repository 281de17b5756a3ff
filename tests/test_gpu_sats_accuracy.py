"""How near Eq. 6's errors are to 64 bits, from the layer call and from the calibration's table, at input counts on
both sides of the down projection's batched and prefill kernels.  The bound, 1e-6 in the 2-norm over the candidates:
a and u are fp32 sums (about 1.5e-7 each), h's two bf16 parts leave 2^-17 of every neuron, rounded to nearest and
averaged over thousands of them, and the truncation of the down projection's accumulators (1e-5 at 4096 neurons) is
common to both norms but for a few per cent.  Taking h from accumulators truncated like that, or the two norms from
different chains, gives 1.5e-6 to 1.8e-5 on the larger of these shapes."""
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


def _block(sats, H, N, seed):
    w = inputs.mlp_weights(H, N, std=0.02, seed=seed)
    layer = sats.Layer(P.dev_u16(w.Wg), P.dev_u16(w.Wu), P.dev_u16(w.Wd))
    return layer, [inputs.bf16_bits_to_f32(m).astype(np.float64) for m in (w.Wg, w.Wu, w.Wd)]


def _h(n, W):
    g = n @ W[0]
    a = g / (1.0 + np.exp(-g))
    return a, a * (n @ W[1])


def _errors(h, drop, Wd, eps):
    y = np.linalg.norm(h @ Wd, axis=1) + eps
    return np.array([np.mean(np.linalg.norm(np.where(d, h, 0.0) @ Wd, axis=1) / y) for d in drop])


def _gap(v, s):
    """The middle of the widest gap within 1 % of the values around the s-quantile of the sorted v."""
    k, w = int(s * v.size), max(4, v.size // 100)
    i = max(0, k - w) + int(np.argmax(np.diff(v[max(0, k - w):k + w])))
    return float(np.float32(0.5 * (v[i] + v[i + 1])))


@pytest.mark.parametrize("H,N,C,K", [(2048, 5633, 48, 12), (1024, 2816, 120, 12), (4096, 6000, 9, 3), (512, 1408, 300, 4),
                                     (96, 261, 5, 7), (96, 40001, 400, 9), (104, 9, 3, 40)])   # several chunks of
                                     # inputs; several groups of candidates
def test_layer_err_against_fp64(sats, H, N, C, K):
    layer, W = _block(sats, H, N, 1400)
    x = inputs.activations_f32(C, H, seed=1401)
    a, h = _h(x.astype(np.float64), W)
    v = np.sort(np.abs(a).ravel())
    ts = [_gap(v, (k + 1) / (K + 1)) for k in range(K)]
    drop = [np.abs(a) < t for t in ts]
    err, sp = sats.layer_err(layer, P.dev(x), ts, eps=1e-6)
    ref = _errors(h, drop, W[2], 1e-6)
    np.testing.assert_allclose(sp, [d.mean() for d in drop], rtol=0, atol=1e-12)
    assert np.linalg.norm(err - ref) <= 1e-6 * np.linalg.norm(ref)
    layer.close()


def test_calibration_table_against_fp64(sats):
    H, N, C = 2048, 5633, 48
    layer, W = _block(sats, H, N, 1410)
    x, gain = P.dev(inputs.activations_f32(C, H, seed=1411)), P.dev(inputs.norm_weight(H))
    r = sats.sats_calibrate([layer], [gain], 1e-5, x, 0.5, K0=14, K1=3, guardrail=False)
    t, err, _ = (np.asarray(v[0]) for v in r["table"])
    n = torch.empty_like(x)
    sats.rmsnorm(x, gain, 1e-5, n)
    a = torch.empty((C, N), device="cuda")
    sats.gate_act_f32(layer, n, a)   # the calibration's own masks: its thresholds are values of these
    mask = np.abs(a.cpu().numpy())
    _, h = _h(n.cpu().numpy().astype(np.float64), W)
    ref = _errors(h, [mask < np.float32(v) for v in t], W[2], 1e-6)
    assert np.linalg.norm(err - ref) <= 1e-6 * np.linalg.norm(ref)
    layer.close()


@pytest.mark.parametrize("C", [2, 4, 40])   # the fused kernel; the tensor cores
def test_infinite_output_has_no_error(sats, C):
    """A kept neuron whose output overflows: y - y~ is infinity less infinity, not a small distortion."""
    H, N = 96, 24
    w = inputs.mlp_weights(H, N, std=0.02, seed=1420)
    Wg, Wu, Wd = (m.copy() for m in (w.Wg, w.Wu, w.Wd))
    Wg[:, 0] = Wu[:, 0] = inputs.to_bf16_bits(np.full(H, 0.02, np.float32))
    Wd[0, :] = inputs.to_bf16_bits(np.full(H, 3e38, np.float32))
    layer = sats.Layer(P.dev_u16(Wg), P.dev_u16(Wu), P.dev_u16(Wd))
    x = np.abs(inputs.activations_f32(C, H, seed=1421))
    err, sp = sats.layer_err(layer, P.dev(x), [0.05, 0.2], eps=1e-6)   # |a| of neuron 0: about 1.2; of the others: below 0.5
    assert np.isnan(err).all() and (np.asarray(sp) > 0).all() and (np.asarray(sp) < 1).all()
    layer.close()
