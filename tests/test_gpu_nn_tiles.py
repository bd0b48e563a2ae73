"""The tcgen05 convolution and weight-gradient kernels of the learned warm
start at the edges of their tiles (boxes of 8 x 16 voxels and up to 4 slices,
chunks of slices): single voxels, exact multiples, one more and one less, and
sizes at which the number of slices per block changes.

The tcgen05 and the mma.sync convolutions accumulate in the same order (taps,
then blocks of 16 channels, in FP32), so outputs, and with them the gradients
(the weight-gradient kernel is the same), must be the same bits.  The
gradients are also compared with the oracle, which rounds to BF16 where the
kernels do: 1e-2 of a tensor's largest value, as in test_gpu_nn.
"""
import numpy as np
import pytest

import paper_1701_06254_gb300 as R
from oracle import nn
from test_gpu_nn import _bf16_weights, _maxrel, _setup, _to_dict

pytestmark = pytest.mark.gpu


def _both(ws, F, T):
    out = []
    for tc in (True, False):
        ws.use_tcgen05(tc)
        y = ws.forward(F.astype(np.float32))
        ws.zero_grad()
        loss = ws.backward(F.astype(np.float32), T.astype(np.float32))
        out.append((np.asarray(y), np.asarray(ws.params(which=1)), loss))
    return out


@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 16, 8), (2, 17, 9), (3, 15, 7), (5, 33, 23), (4, 64, 64), (23, 61, 97),
                                   (1, 130, 261)])
def test_tcgen05_and_mma_sync_agree_bit_for_bit(shape):
    ws, P, F, T = _setup(shape=shape, seed=7)
    (y0, g0, l0), (y1, g1, l1) = _both(ws, F, T)
    assert np.array_equal(y0, y1)
    assert np.array_equal(g0, g1)
    assert l0 == l1


@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 2, 19), (2, 17, 9), (9, 16, 8)])
def test_weight_gradients_at_tile_edges(shape):
    ws, P, F, T = _setup(shape=shape, seed=8)
    ws.zero_grad()
    ws.backward(F.astype(np.float32), T.astype(np.float32))
    g = _to_dict(ws.params(which=1))
    Pb = _bf16_weights(P)
    yo, cache = nn.forward(Pb, F, rnd=nn.bf16_round)
    To = np.zeros(yo.shape); To[..., :2] = T
    go = nn.backward(Pb, cache, yo, To)
    for name, *_ in nn.LAYERS:
        for k in range(2):
            assert _maxrel(g[name][k], go[name][k]) <= 1e-2, (name, k, _maxrel(g[name][k], go[name][k]))
