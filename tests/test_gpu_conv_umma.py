"""The tcgen05 convolutions (csrc/conv_umma.cu) at the edges of their tiles
and pipelines, against the oracle's convolution."""

import numpy as np
import pytest

from launch_shim import run_child
from oracle import surrogate as S
from paper_1511_04633_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1511_04633_gb300 import dmrt
    return torch, dmrt


# (n, batch, cin, cout, offset of y in elements): tiles of two planes (n not a
# multiple of 16) alone and four at a time, one and many stages, half-filled
# channel groups, every output width, runs that cross columns and samples,
# and outputs that are not 16-byte aligned (the mma.sync kernels)
@pytest.mark.parametrize("n,batch,cin,cout,shift", [
    (8, 1, 8, 16, 0), (8, 3, 128, 48, 0), (8, 2, 32, 128, 0), (24, 1, 48, 64, 0), (40, 1, 16, 32, 0),
    (16, 1, 8, 64, 0), (16, 3, 48, 80, 0), (16, 1, 96, 32, 0), (32, 1, 64, 16, 0), (48, 1, 8, 64, 0),
    (16, 1, 16, 16, 0), (16, 3, 32, 32, 0), (48, 2, 8, 16, 0),
    (16, 1, 16, 32, 2), (16, 1, 48, 64, 2), (8, 1, 16, 16, 2),
])
@pytest.mark.parametrize("out_f32", [False, True])
def test_convolution(env, n, batch, cin, cout, shift, out_f32):
    """Inputs exact in bf16: the FP32 accumulation and, for a bf16 output,
    the final rounding (half of 2^-7) are all that differs."""
    torch, dm = env
    x = torch.from_numpy(inputs.random_targets((batch, n, n, n, cin), seed=31)).to(torch.bfloat16)
    w = torch.from_numpy(inputs.random_weights(27 * cout * cin, seed=32, scale=0.2)).to(torch.bfloat16)
    b = torch.from_numpy(inputs.random_weights(cout, seed=33, scale=0.5))
    size = batch * n ** 3 * cout
    flat = torch.full((size + 8,), 7.0, dtype=torch.float32 if out_f32 else torch.bfloat16, device="cuda")
    y = flat[shift:shift + size]
    dm.dmrt_nn_conv3d(x.cuda(), w.cuda(), b.cuda(), y, batch, n, cin, cout, 3, act=1)
    assert dm.dmrt_nn_tensor_core_errors(reset=True) == 0
    ref = S.leaky(S.conv3d(x.double().numpy(), w.double().numpy().reshape(27, cout, cin), b.double().numpy(), 3))
    got = y.double().cpu().numpy().reshape(ref.shape)
    tol = 2e-5 if out_f32 else 8e-3
    assert np.abs(got - ref).max() <= tol * np.abs(ref).max()
    rest = torch.cat([flat[:shift], flat[shift + size:]])
    assert bool((rest == 7.0).all())


# (n, batch, cin, cout): one and many chunks, one and four tiles per CTA, tiles
# of two planes; the mma.sync kernel with 16 output channels per block (few
# blocks, or no multiple of 32) and with 32 (304 blocks or more); narrow layers
# of one K = 16 slice per tap
@pytest.mark.parametrize("n,batch,cin,cout", [
    (8, 2, 128, 64), (24, 1, 64, 128), (24, 8, 96, 128), (16, 1, 48, 80), (32, 3, 64, 64), (48, 1, 128, 32),
    (24, 8, 128, 16), (16, 2, 16, 16), (32, 4, 8, 32),
])
@pytest.mark.parametrize("out_f32", [False, True])
def test_the_two_tensor_core_paths_give_the_same_bits(env, n, batch, cin, cout, out_f32):
    """Outputs at 32-byte, 16-byte (other stores) and smaller alignments (the
    mma.sync kernels)."""
    torch, dm = env
    x = torch.from_numpy(inputs.random_targets((batch, n, n, n, cin), seed=51)).to(torch.bfloat16).cuda()
    w = torch.from_numpy(inputs.random_weights(27 * cout * cin, seed=52, scale=0.2)).to(torch.bfloat16).cuda()
    b = torch.from_numpy(inputs.random_weights(cout, seed=53, scale=0.5)).cuda()
    size = batch * n ** 3 * cout
    elt = 4 if out_f32 else 2
    outs = []
    for shift in (0, 16 // elt, 8 // elt):
        flat = torch.full((size + 8,), 7.0, dtype=torch.float32 if out_f32 else torch.bfloat16, device="cuda")
        y = flat[shift:shift + size]
        dm.dmrt_nn_conv3d(x, w, b, y, batch, n, cin, cout, 3, act=1)
        assert bool((flat[:shift] == 7.0).all()) and bool((flat[shift + size:] == 7.0).all())
        outs.append(y)
    assert dm.dmrt_nn_tensor_core_errors(reset=True) == 0
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])


def test_layers_take_the_faster_kernel(env, tmp_path):
    """Two-plane tiles with few input channels, or output channels that are no
    multiple of 32, go to mma.sync; wide ones and 16-voxel edges to tcgen05."""
    run_child(tmp_path, """
    import torch
    def umma(n, batch, cin, cout):
        x = torch.zeros((batch, n, n, n, cin), dtype=torch.bfloat16, device="cuda")
        w = torch.zeros((27, cout, cin), dtype=torch.bfloat16, device="cuda")
        y = torch.zeros((batch, n, n, n, cout), dtype=torch.bfloat16, device="cuda")
        torch.cuda.synchronize()
        shim.shim_forget()
        dm.dmrt_nn_conv3d(x, w, None, y, batch, n, cin, cout, 3, act=1)
        return b"conv3d_umma" in shim.shim_names()
    for c in ((24, 8, 16, 16), (40, 4, 32, 80), (40, 3, 16, 16), (56, 4, 32, 48)):
        assert not umma(*c), c
    for c in ((24, 8, 128, 128), (8, 4, 128, 128), (40, 4, 64, 64), (56, 2, 8, 64), (16, 1, 16, 16), (16, 4, 48, 48)):
        assert umma(*c), c
    """)
