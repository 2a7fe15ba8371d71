"""The cluster form of the V-cycle's bottom (k_cluster_cycle), the register-resident coarsest inverse, the
zero-start colour pass and the blocked prolongation against the one-kernel-per-step path (smoother = 1):
one outer iteration from psi = 1, so the state afterwards is the correction itself.  Sizes: a problem that
fits the cluster whole, three coarsest orders of the inverse (28, 91, 126: its register tiles), shares that do
not divide evenly, symmetry planes; one cycle (zero start) and two (the second continues from the first).

Both paths apply the same operator and differ in summation order only.  Bound: 1e-4 of each field's
largest value in FP32 (as for the tiled kernels; a wrong neighbour changes a cell by a fraction of order one),
1e-10 in FP64.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2501_13046_gb300 import fields  # noqa: E402


@pytest.fixture(scope="module")
def mg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_13046_gb300 import _build
    _build.build()
    from paper_2501_13046_gb300 import mg as m
    return m


def problem(n, order, bc):
    """Smooth matter on a box of cubic cells (h = 1)."""
    lo = [0.0 if bc != "robin" else -m / 2 for m in n]
    hi = [a + m for a, m in zip(lo, n)]
    X, Y, Z = fields.cell_centres(list(n), lo, hi)
    k = [2 * np.pi / m for m in n]
    w = np.cos(k[0] * X + 0.3) * np.cos(k[1] * Y - 0.2) * np.cos(k[2] * Z + 0.5)
    rho0 = 1e-4 * (2.0 + w)
    S = 1e-5 * np.stack([np.sin(k[0] * X + c) * np.cos(k[1] * Y + 2 * c) * np.cos(k[2] * Z - c) for c in (0.1, 0.7, 1.9)])
    robin = bc != "periodic"
    return dict(n=list(n), lo=lo, hi=hi, order=order, bc=fields.ROBIN if robin else fields.PERIODIC,
                kmode=fields.K_FIXED if robin else fields.K_INTEGRABILITY, K=0.0, punctures=[],
                reflect=7 if bc == "octant" else 0, rho0=rho0, rho2=0.1 * rho0, S=S)


def one_iteration(mg, p, precision, **over):
    cfg = mg.config_for(p, precision, max_outer=1, tol=1e-30, nu_pre=1, nu_post=1, **over)
    ctx = mg.mg_create(cfg, torch.cuda.current_stream().cuda_stream)
    try:
        mg.mg_set_sources(ctx, *[np.ascontiguousarray(a) for a in (p["rho0"], p["rho2"], *p["S"])])
        mg.mg_solve(ctx)
        u, W = np.empty(p["rho0"].shape), np.empty(p["S"].shape)
        mg.mg_get_solution(ctx, u, W)
    finally:
        mg.mg_destroy(ctx)
    return u, W


@pytest.mark.parametrize("cycles", [1, 2])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("n,order,bc", [((24, 20, 12), 4, "periodic"), ((12, 12, 12), 2, "periodic"),
                                        ((20, 20, 20), 4, "periodic"), ((48, 48, 48), 4, "robin"),
                                        ((12, 16, 24), 4, "robin"), ((32, 16, 16), 4, "octant")])
def test_cluster_matches_the_per_kernel_path(mg, n, order, bc, precision, cycles):
    p = problem(n, order, bc)
    prec, tol = (mg.MG_MIXED, 1e-4) if precision == "mixed" else (mg.MG_FP64, 1e-10)
    u0, W0 = one_iteration(mg, p, prec, inner_cycles=cycles, smoother=0)
    u1, W1 = one_iteration(mg, p, prec, inner_cycles=cycles, smoother=1)
    assert np.abs(u1).max() > 0
    assert np.abs(u0 - u1).max() <= tol * np.abs(u1).max()
    for a in range(3):
        assert np.abs(W1[a]).max() > 0
        assert np.abs(W0[a] - W1[a]).max() <= tol * np.abs(W1[a]).max()
