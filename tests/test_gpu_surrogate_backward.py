"""The fused backward pass of the bf16 network (16 channels in the finest
level) against the layer-by-layer pass: the same network with 16 dead channels
more in that level takes the latter."""

import math

import numpy as np
import pytest

from oracle import surrogate as S
from paper_1511_04633_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1511_04633_gb300 import dmrt
    return torch, dmrt


def _gradients(env, n, depth, channels, p, ra, wall, t):
    torch, dm = env
    sur = dm.Surrogate(n, depth, channels, storage=dm.STORE_BF16, max_batch=len(ra))
    sur.set_params(p)
    return sur.gradients(ra, wall, torch.from_numpy(t.reshape(len(ra), -1, 5)).cuda())


# depths 1 to 3, one and several samples, one and many weight-gradient tiles
# per block, two-plane tiles at the coarsest level, narrow and wide layers
@pytest.mark.parametrize("n,depth,channels,batch", [
    (16, 1, (16, 32), 1), (32, 1, (16, 16), 3), (32, 2, (16, 32, 64), 1), (32, 2, (16, 128, 32), 3),
    (64, 3, (16, 32, 64, 128), 1), (64, 3, (16, 32, 64, 128), 3), (64, 2, (16, 16, 16), 2),
])
def test_every_segment(env, n, depth, channels, batch):
    """Zero channels add nothing to any accumulation, so the forward passes
    agree to the bit up to the head, whose sums are ordered differently: its
    bfloat16 outputs and, from there on, the bfloat16 gradients that the
    convolutions read may round differently.  If every one of them did, each of
    the 4 depth + 3 roundings would contribute 2^-9 sqrt(2/3) of a gradient's
    norm, together 6e-3 at depth 3: bound 1e-2.  The loss of 20,000 outputs or
    more averages their roundings: bound 2e-4."""
    net, wide = S.UNet(n, depth, channels), S.UNet(n, depth, (32,) + channels[1:])
    p, q = np.zeros(net.count, np.float32), np.zeros(wide.count, np.float32)
    for i, ((wo, bo), (cin, cout, k, _)) in enumerate(zip(net.offsets, net.layers)):
        w = inputs.random_weights(bo - wo, seed=60 + i, scale=math.sqrt(6.0 / (k ** 3 * cin)))
        b = inputs.random_weights(cout, seed=90 + i, scale=0.1)
        p[wo:bo], p[bo:bo + cout] = w, b
        (xo, yo), (ci, co, _, _) = wide.offsets[i], wide.layers[i]
        q[xo:yo].reshape(k ** 3, co, ci)[:, :cout, :cin] = w.reshape(k ** 3, cout, cin)
        q[yo:yo + cout] = b
    ra, wall = [3e3 * 7 ** k for k in range(batch)], [1 + k % 3 for k in range(batch)]
    t = inputs.random_targets((batch, n, n, n, 5), seed=61)
    g, loss = _gradients(env, n, depth, channels, p, ra, wall, t)
    h, ref_loss = _gradients(env, n, depth, (32,) + channels[1:], q, ra, wall, t)
    assert abs(loss - ref_loss) <= 2e-4 * ref_loss
    for i, ((wo, bo), (cin, cout, k, _)) in enumerate(zip(net.offsets, net.layers)):
        (xo, yo), (ci, co, _, _) = wide.offsets[i], wide.layers[i]
        for name, a, b in (("weights", g[wo:bo], h[xo:yo].reshape(k ** 3, co, ci)[:, :cout, :cin].ravel()),
                           ("bias", g[bo:bo + cout], h[yo:yo + cout])):
            rel = np.linalg.norm(a - b) / np.linalg.norm(b)
            assert rel <= 1e-2, (name, i, cin, cout, k, rel)
