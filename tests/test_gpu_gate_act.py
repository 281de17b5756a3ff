"""Post-gate activations (Sec. 2, Eqs. 1-2) for calibration batches against fp64, at token and neuron
counts around the tile edges and hidden sizes that do not fill a K block.  The bound: fp32 arithmetic.
Each sum is H products in segments of 32, rounded once per segment, so its error is a few units of
2^-24 relative to the norm; 1e-6 allows eight, and a plain fp32-accumulator chain on the tensor cores
(1.2e-5 at H = 4096) or a dropped low part of x (4e-3) does not pass."""
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


def _silu(g):
    return g / (1.0 + np.exp(-g))


@pytest.mark.parametrize("H,N", [(8, 5), (72, 130), (512, 1408), (4096, 1009), (8192, 260)])
@pytest.mark.parametrize("B", [1, 16, 17, 128, 129, 300])
def test_against_fp64(sats, H, N, B):
    w = inputs.mlp_weights(H, N, std=1.0 / np.sqrt(H), seed=1200)
    layer = sats.Layer(P.dev_u16(w.Wg), P.dev_u16(w.Wu), P.dev_u16(w.Wd))
    W = inputs.bf16_bits_to_f32(w.Wg).astype(np.float64)
    a = torch.full((B, N), -7.0, device="cuda")
    x = inputs.activations_f32(B, H, seed=1201)
    sats.gate_act_f32(layer, P.dev(x), a)
    ref = _silu(x.astype(np.float64) @ W)
    assert np.linalg.norm(a.cpu().numpy() - ref) <= 1e-6 * np.linalg.norm(ref)
    xb = inputs.activations_bf16(B, H, seed=1202)
    a.fill_(-7.0)
    sats.gate_act(layer, P.dev_u16(xb), a)
    ref = _silu(inputs.bf16_bits_to_f32(xb).astype(np.float64) @ W)
    assert np.linalg.norm(a.cpu().numpy() - ref) <= 1e-6 * np.linalg.norm(ref)
    layer.close()


def test_fp32_range_of_the_activations(sats):
    """Values at the ends of fp32's range, infinities and NaN go through the cut into parts unharmed."""
    H, N = 64, 24
    w = inputs.mlp_weights(H, N, std=0.1, seed=1210)
    layer = sats.Layer(P.dev_u16(w.Wg), P.dev_u16(w.Wu), P.dev_u16(w.Wd))
    W = inputs.bf16_bits_to_f32(w.Wg).astype(np.float64)
    x = inputs.activations_f32(5, H, seed=1211)
    x[0, 3] = 3.0e38
    x[1, 5] = np.inf
    x[2, 7] = np.nan
    x[3] *= np.float32(1e-25)
    a = torch.zeros((5, N), device="cuda")
    sats.gate_act_f32(layer, P.dev(x), a)
    got = a.cpu().numpy().astype(np.float64)
    with np.errstate(all="ignore"):
        g = x.astype(np.float64) @ W
        ref = g / (1.0 + np.exp(-g))
    ref[0] = np.where(g[0] < 0, -0.0, g[0])    # exp of a large positive number is infinite in fp32
    for r in (0, 3, 4):
        np.testing.assert_allclose(got[r], ref[r], rtol=2e-5, atol=1e-30)
    assert np.array_equal(np.isposinf(got[1]), g[1] > 0) and np.isnan(got[1][g[1] < 0]).all()
    assert np.isnan(got[2]).all()
    layer.close()


@pytest.mark.parametrize("H,N,B,f32,bound", [
    (256, 1000, 130, False, 7.6e-8),   # roundings of the totals kept beside them
    (512, 1408, 130, False, 7.6e-8),
    (2048, 1000, 200, False, 7.6e-8),
    (2056, 1000, 60, False, 1.15e-7),  # sums in two levels
    (4096, 1009, 128, True, 1.4e-7),   # totals of tiles of more than 64 tokens
    (8192, 260, 100, True, 1.5e-7),
])
def test_no_further_from_fp64_than_fma_chains(sats, H, N, B, f32, bound):
    """The 2-norm of the error in units of the result's.  A rounding to nearest at the size of the result leaves
    2.1e-8 (2^-24 / sqrt(8) for values spread over a binade), the two truncated MMA steps 3e-8 that do not average out and
    twice 2.1e-8 in parts, SiLU's exponential and final rounding 4e-8: 6.4e-8 with no other rounding; two levels of 4 to
    16 additions bring 4 to 6 roundings more, fp32 parts one more bias of 3e-8.  FMA chains leave 7.1e-8 / 7.7e-8 / 9.5e-8
    at hidden 256 / 512 / 2048 (bf16) and 2.3e-7 / 3.1e-7 at 4096 / 8192 (fp32); sums of one level 9.0e-8 and more
    and 1.9e-7 / 2.4e-7."""
    w = inputs.mlp_weights(H, N, std=0.02, seed=1220)
    layer = sats.Layer(P.dev_u16(w.Wg), P.dev_u16(w.Wu), P.dev_u16(w.Wd))
    W = inputs.bf16_bits_to_f32(w.Wg).astype(np.float64)
    a = torch.full((B, N), -7.0, device="cuda")
    if f32:
        x = inputs.activations_f32(B, H, seed=1221)
        sats.gate_act_f32(layer, P.dev(x), a)
        x = x.astype(np.float64)
    else:
        xb = inputs.activations_bf16(B, H, seed=1222)
        sats.gate_act(layer, P.dev_u16(xb), a)
        x = inputs.bf16_bits_to_f32(xb).astype(np.float64)
    ref = _silu(x @ W)
    assert np.linalg.norm(a.cpu().numpy() - ref) <= bound * np.linalg.norm(ref)
    layer.close()


def test_bf16_range(sats):
    """Infinite, overflowing and not-a-number sums where totals keep their roundings (hidden 64) and where not (2112)."""
    for H in (64, 2112):
        N = 24
        w = inputs.mlp_weights(H, N, std=0.1, seed=1230)
        layer = sats.Layer(P.dev_u16(w.Wg), P.dev_u16(w.Wu), P.dev_u16(w.Wd))
        W = inputs.bf16_bits_to_f32(w.Wg).astype(np.float64)
        xb = inputs.activations_bf16(4, H, seed=1231)
        xb[1, 5], xb[2, 7] = 0x7F80, 0x7FC0   # inf, nan
        x = inputs.bf16_bits_to_f32(xb).astype(np.float64)
        a = torch.zeros((4, N), device="cuda")
        sats.gate_act(layer, P.dev_u16(xb), a)
        got = a.cpu().numpy().astype(np.float64)
        with np.errstate(all="ignore"):
            g = x @ W
        for r in (0, 3):
            np.testing.assert_allclose(got[r], _silu(g[r]), rtol=2e-5, atol=1e-30)
        assert np.array_equal(np.isposinf(got[1]), g[1] > 0) and np.isnan(got[1][g[1] < 0]).all()
        assert np.isnan(got[2]).all()
        layer.close()
