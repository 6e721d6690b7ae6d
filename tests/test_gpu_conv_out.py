"""The correction network's output layer at inference, at the edges of its
tiles (32 columns by 8 rows, blocks of 4 to 32 planes).

The values are chosen so that every arithmetic step is exact: the step is +-1
(its RMS is exactly 1), the hidden layers pass small whole numbers that bf16
holds, and the output layer's weights are whole numbers, so each output is a
whole number below 2^24 that float32 sums hold in any order.  The tolerance
is therefore that of the last multiplication by the RMS and its reciprocal,
a few float32 roundings of the result: 1e-6 of the largest entry."""
import numpy as np
import pytest
import torch

from oracle import learned as NL
from tests.helpers import to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2103_10329_gb300 import build
    build.build()


def whole_params(seed):
    rng = np.random.default_rng(seed)
    layers = []
    for l, (ci, co) in enumerate(zip(NL.CIN, NL.COUT)):
        w = np.zeros((27, co, ci))
        if l == 3:
            w[:] = rng.integers(-3, 4, w.shape)
        else:  # centre tap only: each output channel is +- one input channel
            w[13, np.arange(co), rng.integers(0, ci, co)] = rng.choice([-1.0, 1.0], co) if l == 0 else 1.0
        layers.append((w, rng.integers(0, 3, co).astype(float)))
    return NL.pack(layers).astype(np.float32)


@pytest.mark.parametrize("shape", [(1, 1, 1, 1), (1, 2, 9, 33), (3, 5, 7, 31), (2, 33, 8, 32), (1, 36, 17, 65),
                                   (1, 65, 65, 97)])
def test_output_layer_exact(shape):
    from paper_2103_10329_gb300 import mgct
    net = mgct.Net()
    p = whole_params(sum(shape))
    net.set_params(p)
    step = np.random.default_rng(7).choice([-1.0, 1.0], shape)
    out = to_np(net.apply(torch.tensor(step, dtype=torch.float32, device="cuda")))
    net.check()
    y, _ = NL.forward(p.astype(np.float64), step, bf=True)
    ref = step + y
    assert np.abs(out - ref).max() <= 1e-6 * np.abs(ref).max()
