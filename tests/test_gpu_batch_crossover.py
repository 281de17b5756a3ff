"""Batches of 65 to 256 tokens (224 with fp32 activations) around the line between the two gate/up
kernels: token counts at the tiles' edges, on layers that the rule sends each way, with the down
projection of the smaller batches behind either.  Same bounds as the other tensor-core batches."""
import pytest

from tests.test_gpu_route_stack import _stack
from tests.test_gpu_sparse_mlp import _run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sats():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2607_08991_gb300 import sats as s
    return s


@pytest.mark.parametrize("H,N", [
    (512, 1408),     # the prefill kernel throughout
    (72, 130),       # one tile of 16 neurons per SM and fewer; a partial K block
    (1024, 777),
    (128, 14600),    # more than one wave of tiles either way
])
@pytest.mark.parametrize("B,f32", [(65, False), (66, True), (97, True), (112, True), (113, True), (128, False), (129, False), (129, True),
                                   (208, False), (224, True), (256, False)])
def test_either_gate_up_kernel(sats, oracle, H, N, B, f32):
    _run(sats, oracle, H, N, B, 0.6, f32=f32)


@pytest.mark.parametrize("B", [113, 224])
def test_routed_stack(sats, oracle, B):
    keep, ids, lut = _stack(sats, oracle, 2, 512, 1408, B, [0.6] * 2, 1e-6, routed=True, p_dense=0.4, seed=B)
    assert keep[:, lut[ids] == 1].all()
