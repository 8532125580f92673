"""The network's gradients at the edges of its kernels' work split: one pixel,
one row, one column, a pixel count next to a multiple of the 128-pixel chunks,
and more chunks than the weight gradient has blocks (each then adds several
up).  Bounds as in test_gpu_skipnet."""
import numpy as np
import pytest

from oracle import cnn
from test_gpu_skipnet import RTOL_BF16, _elementwise_err, _setup, _unflat

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nimg,H,W", [(1, 1, 1), (1, 1, 200), (2, 33, 1), (1, 3, 43), (5, 127, 129)])
def test_gradients_match_oracle_at_the_edges(nimg, H, W):
    from paper_2206_05761_gb300 import hwfv1 as Hh
    net, params, x, labels, xd, ld = _setup(11, nimg, H, W)
    loss, g = Hh.hwfv1_skipnet_gradients(net, xd, ld, nimg, H, W)
    again, g2 = Hh.hwfv1_skipnet_gradients(net, xd, ld, nimg, H, W)
    assert np.array_equal(g, g2)
    logits, cache = cnn.forward(params, x.transpose(0, 3, 1, 2), cnn.bf16)
    ref_loss, dl = cnn.loss_and_dlogits(logits, labels)
    ref = cnn.backward(params, cache, dl, cnn.bf16)
    assert abs(loss - ref_loss) <= RTOL_BF16 * ref_loss
    for name, a, b in zip(("w1", "b1", "w2", "b2", "w3", "b3"), _unflat(g, params), ref):
        if np.abs(b).max() == 0.0:
            assert not a.any(), name
        else:
            assert _elementwise_err(a, b) <= RTOL_BF16, name
    Hh.hwfv1_skipnet_destroy(net)
