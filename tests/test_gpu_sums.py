"""The means of a correction (k_sum4) keep FP64's precision: against exactly rounded sums.

Bound: a thread adds its values exactly (pairs of floats, at most 4 values here) or in FP64; what follows are at most 3
additions in a thread, 5 in a warp, 8 over a block's warps, one more over the blocks and 10 in the last block's tree,
each rounding by 2^-53 of the sum of the magnitudes: 32 in all with the division by N and the test's own."""
import ctypes
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from tests.native import load
    return load("sums")


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("N", [1, 27, 125, 128, 131, 512, 1000, 4096, 64 ** 3])
def test_means_against_exact_sums(lib, N, dtype):
    f = lib.sum4_f32 if dtype == torch.float32 else lib.sum4_f64
    partial = torch.zeros(4 * lib.sum4_blocks(), dtype=torch.float64, device="cuda")
    ticket = torch.zeros(4, dtype=torch.int32, device="cuda")
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    for seed in range(20 if N < 5000 else 2):
        rng = np.random.default_rng(seed)
        x = np.stack([rng.uniform(1, 2, N), rng.standard_normal(N), 2.0 ** rng.uniform(-25, 0, N), -rng.random(N)])
        x = x.astype(np.float32 if dtype == torch.float32 else np.float64)
        xt = torch.from_numpy(x).cuda()
        means = torch.zeros(4, dtype=torch.float64, device="cuda")
        assert f(ptr(xt), ctypes.c_longlong(N), ptr(partial), ptr(means), ptr(ticket)) == 0
        for a in range(4):
            v = x[a].astype(np.float64)
            assert abs(means[a].item() - math.fsum(v) / N) <= 32 * 2.0 ** -53 * np.abs(v).sum() / N, (a, seed)
