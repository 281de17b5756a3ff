"""LoRA batches beyond one pass of the fused kernel, at token counts around the tile edges, neuron
counts that do not fill a tile or a K block, the smallest hidden size of the path and every rank,
against the oracle element by element.  The bound is fp32 arithmetic's (both matrix products are
summed in segments of 32 products, of 64 with fp32 activations in tiles of more than 16 tokens, rounded once
each, a few units of 2^-24): 1e-6 relative, which a plain
accumulator chain on the tensor cores (1e-5) or h rounded to two bf16 parts (4e-6) does not meet."""
import numpy as np
import pytest
import torch

from paper_2607_08991_gb300 import inputs
from tests import _parity as P
from tests.test_gpu_lora import _call, _setup, _threshold

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sats():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2607_08991_gb300 import sats as s
    return s


@pytest.mark.parametrize("H,N,B,r,f32", [
    (96, 5, 3, 8, False),        # the smallest hidden size, one ragged tile
    (96, 200, 4, 32, True),
    (512, 1408, 16, 16, True),   # a full tile of 16 tokens
    (1032, 777, 17, 24, False),  # two token blocks, a hidden size that ends inside a K block
    (1032, 777, 32, 24, True),   # a full tile of 32 tokens
    (4096, 1009, 33, 16, False), # two token tiles
    (4096, 1009, 40, 16, True),
    (8192, 130, 3, 8, True),     # the largest hidden size (one token per fused pass; two would stay passes)
    (64, 100, 5, 8, False),      # below the path: passes of the fused kernel
])
def test_batches_match_oracle(sats, oracle, H, N, B, r, f32):
    scale = 0.75
    w, lo, layer, lora = _setup(sats, H, N, r, scale, seed=11)
    t = _threshold(oracle, w, H, 0.6)
    ws = sats.Workspace(H, N, B)
    if f32:
        xf = inputs.activations_f32(B, H, seed=inputs.SEED_X + 31)
        x64, xdev = xf.astype(np.float64), P.dev(xf)
    else:
        xb = inputs.activations_bf16(B, H, seed=inputs.SEED_X + 31)
        x64, xdev = oracle.bf16_to_f64(xb), P.dev_u16(xb)
    for _ in range(2):   # a second call on the same workspace
        y, keep = _call(sats, layer, lora, xdev, t, B, H, N, ws)
        y_ref, a_ref, keep_ref, _ = oracle.sparse_mlp_lora(x64, w.Wg, w.Wu, w.Wd, lo, scale, t, keep_hint=keep,
                                                           band_rel=P.BAND_REL)
        P.assert_keep_match(keep, keep_ref, a_ref, t)
        assert np.linalg.norm(y - y_ref) <= 1e-6 * np.linalg.norm(y_ref)
    # without the lists, on a workspace that other calls have used
    y2 = torch.full((B, H), float("nan"), device="cuda")
    if not f32:
        sats.sparse_mlp(layer, xdev, t, y2, ws)
    sats.sparse_mlp_lora(layer, lora, xdev, t, y2, ws)
    assert sats.get_error(ws) == sats.OK
    assert np.linalg.norm(y2.cpu().numpy() - y_ref) <= 1e-6 * np.linalg.norm(y_ref)
    lora.close()
    layer.close()


@pytest.mark.parametrize("H,N,B,f32", [(8192, 3584, 4, False), (8192, 3584, 17, True), (6000, 2001, 3, True),
                                       (2048, 3100, 8, False), (256, 400, 16, True)])
def test_no_further_from_fp64_than_single_tokens(sats, oracle, H, N, B, f32):
    """A batch's sums are no less accurate than the fused kernel's, which runs the same tokens one at a time."""
    r, scale = 16, 1.0
    w, lo, layer, lora = _setup(sats, H, N, r, scale, seed=12)
    if f32:
        xf = inputs.activations_f32(B, H, seed=inputs.SEED_X + 32)
        x64, x = xf.astype(np.float64), P.dev(xf)
    else:
        xb = inputs.activations_bf16(B, H, seed=inputs.SEED_X + 32)
        x64, x = oracle.bf16_to_f64(xb), P.dev_u16(xb)
    t = _threshold(oracle, w, H, 0.6)
    ws = sats.Workspace(H, N, B)
    y, keep = _call(sats, layer, lora, x, t, B, H, N, ws)
    ref, _, _, _ = oracle.sparse_mlp_lora(x64, w.Wg, w.Wu, w.Wd, lo, scale, t, keep_hint=keep, band_rel=P.BAND_REL)
    one = np.empty_like(y)
    for b in range(B):
        one[b], k1 = (v[0] for v in _call(sats, layer, lora, x[b:b + 1], t, 1, H, N, ws))
        if not np.array_equal(k1, keep[b]):   # a neuron at the threshold fell on the other side
            one[b] = ref[b]
    err, err1 = np.linalg.norm(y - ref), np.linalg.norm(one - ref)
    assert err1 > 0 and err <= err1
    lora.close()
    layer.close()
