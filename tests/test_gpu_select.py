"""Percentile selection (Eq. 3) against a sort: the m-th smallest |a| exactly, at sizes around
the vector width and the grid, on misaligned data, with ties, zeros and infinities; and the
shared passes over many ranks that the SATS calibration uses."""
import math

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


def _values(kind, n):
    g = np.random.default_rng([n, len(kind)])
    if kind == "normal":
        v = g.standard_normal(n)
    elif kind == "ties":
        v = g.integers(-3, 4, n) * 0.25
    else:   # every exponent, subnormals, zeros of both signs and infinities
        v = np.ldexp(g.standard_normal(n), g.integers(-149, 127, n))
        v[::7] = 0.0
        v[::11] = -0.0
        v[::13] = math.inf
    return v.astype(np.float32)


@pytest.mark.parametrize("n", [1, 3, 4, 2047, 2049, 311297, 1000003])
@pytest.mark.parametrize("kind", ["normal", "ties", "wide"])
def test_rank_is_exact(sats, n, kind):
    buf = torch.zeros(n + 4, device="cuda")
    sel = torch.zeros(sats.select_workspace_bytes(), dtype=torch.uint8, device="cuda")
    v = _values(kind, n)
    order = np.sort(np.abs(v))
    for off in (0, 1):   # 16-byte loads, and single ones
        a = buf[off:off + n]
        a.copy_(torch.from_numpy(v))
        for k in (1e-9, 0.1, 0.5, 0.937, 1.0):
            m = min(n, max(1, math.ceil(k * n * (1.0 - 2.0 ** -50))))
            assert sats.percentile_threshold(a, k, sel) == float(order[m - 1]), (off, k)


@pytest.mark.parametrize("K0", [2, 31, 40])   # one rank, a full group of 32, and a group and a rest
def test_shared_passes_equal_single_selections(sats, K0):
    H, N, C = 64, 136, 6
    layers, gains = [], []
    for l in range(2):
        w = inputs.mlp_weights(H, N, layer=l, std=0.1, seed=900)
        layers.append(sats.Layer(P.dev_u16(w.Wg), P.dev_u16(w.Wu), P.dev_u16(w.Wd)))
        gains.append(P.dev(inputs.norm_weight(H, layer=l)))
    x = P.dev(inputs.activations_f32(C, H, seed=901))
    r = sats.sats_calibrate(layers, gains, 1e-5, x, 0.5, K0=K0, K1=2, guardrail=True)
    n = torch.empty_like(x)
    a = torch.empty((C, N), device="cuda")
    sel = torch.zeros(sats.select_workspace_bytes(), dtype=torch.uint8, device="cuda")
    sats.rmsnorm(x, gains[0], 1e-5, n)
    sats.gate_act_f32(layers[0], n, a)
    want = [sats.percentile_threshold(a, k / K0, sel) for k in range(1, K0)]
    assert r["table"][0][0][:K0 - 1] == want
    for l in layers:
        l.close()
