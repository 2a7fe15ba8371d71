"""The register-resident inverse of the coarsest psi row (k_invert_registers) by itself, at the edges of its register
tiles, against A G = I.

Matrices: a random permutation of the rows of a diagonally dominant matrix (zero or small diagonals: every step needs its
pivot search), and a bordered one, singular without the border, as on periodic boxes.
Bound: Gauss-Jordan elimination with partial pivoting leaves |A G - I| <= 8 m u |A| |G| times the growth of the pivots (Higham,
Accuracy and Stability of Numerical Algorithms, section 14.4, per column of I), which is at most 2 for these matrices."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from tests.native import load
    return load("inverse")


def dominant(rng, m):
    A = rng.standard_normal((m, m)) / m
    A[np.arange(m), np.arange(m)] = 2 + rng.random(m)
    return A[rng.permutation(m)]


def bordered(rng, m):
    """A periodic 1D Laplacian, bordered by ones: the multiplier's row and column with a zero corner."""
    A = np.zeros((m, m))
    n = m - 1
    for i in range(n):
        A[i, i] = -2 - 1e-3 * rng.random()
        A[i, (i + 1) % n] += 1
        A[i, i - 1] += 1
    A[n, :n] = A[:n, n] = 1
    return A


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("m", [1, 2, 7, 28, 32, 33, 48, 64, 65, 91, 96, 97, 126, 133, 160])
def test_product_with_the_matrix_is_the_identity(lib, m, precision):
    dt, u, f = (np.float32, 2.0 ** -24, lib.invert_f32) if precision == "fp32" else (np.float64, 2.0 ** -53, lib.invert_f64)
    for seed in range(4):
        rng = np.random.default_rng(100 * m + seed)
        A = (bordered(rng, m) if seed == 3 and m > 3 else dominant(rng, m)).astype(dt)
        aug = np.zeros((m, 2 * m), dt)
        aug[:, :m] = A
        aug[:, m:] = np.nan   # the identity block is not read
        at = torch.from_numpy(aug).cuda()
        gt = torch.full((m, m), float("nan"), dtype=at.dtype, device="cuda")
        assert f(ctypes.c_void_p(at.data_ptr()), m, ctypes.c_void_p(gt.data_ptr())) == 0
        A, G = A.astype(np.longdouble), gt.cpu().numpy().astype(np.longdouble)
        assert np.isfinite(G).all()
        bound = 16 * m * u * (np.abs(A) @ np.abs(G)).max()
        assert np.abs(A @ G - np.eye(m)).max() <= bound, (seed, float(np.abs(A @ G - np.eye(m)).max()), float(bound))
