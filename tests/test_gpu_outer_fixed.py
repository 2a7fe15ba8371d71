"""The fused FP64 residual (stencils in 64-bit fixed point) against the oracle, cell by cell, where its
tiling and its units can go wrong: grids of a few cells, tile edges and remainders (16 x 8 tiles, chunks of
planes), unequal spacings, every boundary variant, values that grow from plane to plane (the tile's unit
is rescaled on the way), and a NaN (the direct path).

Tolerance, derived: both sides sum at most 32 products per output, each rounded to 2^-53 of terms whose
weights total 16 / h^2 (Laplacian: 3 * 64/12) or 20 / h^2 (momentum row with its mixed terms); the later
factors psi^-5, psi^-6 and the nonlinear terms add a few units of 2^-53 of the value (1e-13 with margin).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import oracle as O  # noqa: E402
from paper_2501_13046_gb300 import fields  # noqa: E402

EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def mg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_13046_gb300 import _build
    _build.build()
    from paper_2501_13046_gb300 import mg as m
    return m


def problem(n, order, bc, box):
    rng = np.random.default_rng(3)
    shape = (n[2], n[1], n[0])
    robin = bc != "periodic"
    lo = [0.0 if bc == "octant" else -b / 2 if robin else 0.0 for b in box]
    hi = [l + b for l, b in zip(lo, box)]
    return dict(n=list(n), lo=lo, hi=hi, order=order, bc=fields.ROBIN if robin else fields.PERIODIC,
                kmode=fields.K_FIXED if robin else fields.K_INTEGRABILITY, K=0.3 if robin else 0.0, punctures=[],
                reflect=7 if bc == "octant" else 0, extrap=0b000110 if bc == "extrap" else 0,
                rho0=0.5 + 0.1 * rng.standard_normal(shape), rho2=0.01 * rng.random(shape),
                S=0.01 * rng.standard_normal((3,) + shape))


def gpu_fields(mg, p, u, W):
    ctx = mg.mg_create(mg.config_for(p, mg.MG_FP64), torch.cuda.current_stream().cuda_stream)
    try:
        mg.mg_set_sources(ctx, *[np.ascontiguousarray(a) for a in (p["rho0"], p["rho2"], *p["S"])])
        mg.mg_set_initial_guess(ctx, np.ascontiguousarray(u), np.ascontiguousarray(W))
        H, M = np.empty_like(u), np.empty_like(W)
        mg.mg_constraint_fields(ctx, H, M)
    finally:
        mg.mg_destroy(ctx)
    return H, M


def check(p, u, W, H, M, per_plane=False):
    g = O.make_grid(p["n"], p["lo"], p["hi"], p["order"], p["bc"], p["punctures"], reflect=p["reflect"],
                    extrap=p["extrap"])
    ref = O.residual(g, u, W, p["rho0"], p["rho2"], p["S"], p["kmode"], K2=p["K"] ** 2)
    h2 = min((p["hi"][a] - p["lo"][a]) / p["n"][a] for a in range(3)) ** 2
    # a plane's unit follows the largest value met so far: planes up to two further on
    top = lambda f: np.array([np.nanmax(np.abs(f[..., :k + 3, :, :])) for k in range(p["n"][2])])[:, None, None] \
        if per_plane else np.nanmax(np.abs(f))
    psi = np.abs(1.0 + np.nan_to_num(u)).min()
    tol_H = 8 * psi ** -5 * 2 * 32 * EPS * 16 / h2 * top(u) + 1e-13 * np.nanmax(np.abs(ref["H"]))
    tol_M = psi ** -6 * (2 * 32 * EPS * 20 / h2 * top(W) + 1e-13 * 8 * np.pi * np.abs(p["S"]).max() * (1 + np.nanmax(u)) ** 6)
    assert np.array_equal(np.isnan(H), np.isnan(ref["H"])) and np.array_equal(np.isnan(M), np.isnan(ref["M"]))
    assert (np.abs(np.nan_to_num(H - ref["H"])) <= tol_H).all(), np.nanmax(np.abs(H - ref["H"]) / tol_H)
    assert (np.abs(np.nan_to_num(M - ref["M"])) <= tol_M).all(), np.nanmax(np.abs(M - ref["M"]) / tol_M)


CASES = [((3, 3, 3), 2, "periodic", (3.0, 3.0, 3.0)), ((5, 4, 6), 4, "periodic", (5.0, 4.0, 6.0)),
         ((16, 8, 32), 4, "periodic", (16.0, 8.0, 32.0)), ((17, 9, 33), 4, "periodic", (17.0, 7.0, 40.0)),
         ((33, 15, 7), 2, "periodic", (33.0, 20.0, 7.0)), ((18, 10, 35), 4, "robin", (9.0, 5.0, 17.5)),
         ((31, 24, 6), 2, "robin", (20.0, 24.0, 5.0)), ((20, 17, 12), 4, "octant", (10.0, 8.5, 6.0)),
         ((19, 12, 14), 4, "extrap", (9.5, 6.0, 7.0))]


@pytest.mark.parametrize("n,order,bc,box", CASES)
def test_fields_match_the_oracle_cell_by_cell(mg, n, order, bc, box):
    p = problem(n, order, bc, box)
    rng = np.random.default_rng(11)
    u, W = 0.05 * rng.standard_normal(p["rho0"].shape), 0.02 * rng.standard_normal(p["S"].shape)
    check(p, u, W, *gpu_fields(mg, p, u, W))


@pytest.mark.parametrize("bc", ["periodic", "robin"])
def test_growing_values_rescale_the_unit(mg, bc):
    """W grows fourfold and u twofold per plane: the unit of every plane follows its own neighbourhood."""
    p = problem((18, 9, 24), 4, bc, (18.0, 9.0, 24.0))
    p["S"] = 0.0 * p["S"]
    rng = np.random.default_rng(5)
    k = np.arange(24)[:, None, None]
    u = 0.05 * 2.0 ** (k - 23) * rng.standard_normal(p["rho0"].shape)
    W = 0.02 * 4.0 ** (k - 23) * rng.standard_normal(p["S"].shape)
    H, M = gpu_fields(mg, p, u, W)
    # (a periodic box's first planes reach the last, largest ones; momentum sources and their mean are zero)
    check(p, u, W, H, M, per_plane=bc == "robin")


def test_a_nan_stays_local(mg):
    p = problem((20, 11, 13), 4, "robin", (10.0, 5.5, 6.5))
    rng = np.random.default_rng(6)
    u, W = 0.05 * rng.standard_normal(p["rho0"].shape), 0.02 * rng.standard_normal(p["S"].shape)
    W[1, 9, 6, 17] = np.nan
    H, M = gpu_fields(mg, p, u, W)
    assert np.isnan(M).any() and np.isfinite(M).any()
    check(p, u, W, H, M)
