"""Convolution paths that only larger volumes reach: the block tile of the layers with the largest operands, and the weight
gradient with several voxel chunks per CTA (both buffers, the table one stage ahead, the zero rows of unused taps).
Oracle and forward bound as in test_gpu_unet_conv."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import conv_ref as R  # noqa: E402
from tests.test_gpu_unet_conv import U, bf16, tohost  # noqa: E402,F401


@pytest.mark.parametrize("cin,cout", [(64, 32), (32, 96), (32, 64)])
@pytest.mark.parametrize("shape", [(8, 16, 2), (16, 16, 8), (32, 32, 24), (16, 48, 40)])   # 1, 8, 96, 120 tiles of 8 x 16 x 2
def test_conv_forward_block_tiles_of_large_layers(U, cin, cout, shape):  # noqa: F811
    nx, ny, nz = shape
    rng = np.random.default_rng(cin * 977 + cout + nx)
    x = R.bf16_round(rng.standard_normal((nz, ny, nx, cin)))
    w = R.bf16_round(rng.standard_normal((27, cout, cin)) / np.sqrt(27 * cin))
    b = rng.standard_normal(cout).astype(np.float32)
    wp = torch.empty(w.shape, dtype=torch.bfloat16, device="cuda")
    U.pack_weights(torch.from_numpy(w.astype(np.float32)).cuda(), cin, cout, 0, wp)
    ref, scale = R.conv_fwd(x, w, b.astype(np.float64), relu=False), R.conv_fwd(np.abs(x), np.abs(w))
    for relu in (False, True):
        y = torch.zeros((nz, ny, nx, cout), dtype=torch.bfloat16, device="cuda")
        err = torch.zeros(1, dtype=torch.int32, device="cuda")
        U.conv3d_fwd(bf16(x), wp, torch.from_numpy(b).cuda(), y, (nx, ny, nz), cin, cout, relu, err)
        torch.cuda.synchronize()
        assert int(err.item()) == 0
        r = np.maximum(ref, 0) if relu else ref
        assert np.all(np.abs(tohost(y) - r) <= 2 ** -8 * np.abs(r) + 1e-5 * scale + 1e-6)


# chunks of 128 voxels per CTA: 2, 6, 6, 12, 12, 4
@pytest.mark.parametrize("cin,cout,shape", [(16, 32, (32, 32, 32)), (32, 64, (64, 32, 32)), (48, 16, (32, 32, 32)),
                                           (96, 32, (32, 32, 32)), (128, 64, (32, 32, 32)), (64, 64, (24, 24, 32))])
def test_conv_weight_gradient_of_several_chunks(U, cin, cout, shape):  # noqa: F811
    """FP32 bound: a CTA adds at most 8 x 12 products of 16 voxels each in turn, the CTAs at most 152 partials: (8 x 12 + 16 +
    152) roundings of 2^-23 (the tensor cores may truncate) of the sum of the magnitudes."""
    nx, ny, nz = shape
    rng = np.random.default_rng(21 + cin)
    x = R.bf16_round(rng.standard_normal((nz, ny, nx, cin)))
    dy = R.bf16_round(rng.standard_normal((nz, ny, nx, cout)))
    ref, scale = R.conv_wgrad(x, dy), R.conv_wgrad(np.abs(x), np.abs(dy))
    dw = torch.zeros((27, cout, cin), dtype=torch.float32, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    U.conv3d_wgrad(bf16(x), bf16(dy), dw, (nx, ny, nz), cin, cout, err)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    np.testing.assert_array_less(np.abs(dw.cpu().numpy() - ref), (8 * 12 + 16 + 152) * 2.0 ** -23 * scale)
