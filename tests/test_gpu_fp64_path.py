"""The FP64 path's kernels (fixed-point near field and translations, symmetry-shared expansions)
against the oracle's direct sum on every cell, at the sizes and settings where their index
arithmetic changes: leaf levels 2, 3 and 5 (subtree depths, cluster splits), near radii 1, 2, 3
and 5, orders at the edges of the row groups (8, 15, 16, 19, 20, 23) and 24 (the generic kernels).

Tolerance: truncation.  A pair accepted by r_A + r_B < theta d contributes with an error below
theta^(p+1) of the sum of |q log r|; the relative l2 of the field is allowed ten times that, and
1e-13 where the series is exact to rounding.
"""
import numpy as np
import pytest

import oracle
from paper_1610_04398_gb300 import synth
from gpu_cases import rel_l2, run_gpu, run_oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1610_04398_gb300 as pkg
    pkg.build()
    oracle.build()


@pytest.mark.parametrize("n,order,theta", [(32, 20, 0.5), (64, 8, 0.95), (64, 23, 0.25), (64, 24, 0.25), (64, 15, 0.4),
                                           (128, 16, 0.6), (128, 19, 0.75), (256, 20, 0.5)])
def test_fp64_grid_matches_direct_sum(n, order, theta):
    snap = synth.cylinder_flow(n, diameter=0.3, centre=(0.5, 0.5), n_surface=130, seed=n + order)
    g = run_gpu(snap, "fp64", order, theta)
    r = run_oracle(snap)
    tol = max(10 * theta ** (order + 1), 1e-13)
    e, es = rel_l2(g["P"].ravel(), r["P_cells"]), rel_l2(g["per_point"][:, 0], r["P_surf"])
    print(f"n {n} p {order} theta {theta}: grid {e:.2e} surface {es:.2e} (allowed {tol:.1e})")
    assert np.max(np.abs(g["f"] - r["f"])) <= 1e-12 * np.max(np.abs(r["f"]))
    assert e <= tol
    assert es <= max(10 * min(theta, 0.6) ** (order + 1), 1e-13)
    g["plan"].destroy()


def test_fp64_non_finite_source_reaches_every_cell():
    snap = synth.lamb_oseen(64)
    snap.u[20, 30] = np.inf
    g = run_gpu(snap, "fp64", 12, 0.5)
    assert not np.isfinite(g["P"]).any()
    g["plan"].destroy()


def test_fp64_dynamic_range():
    """Weights of one corner 2^-300 of the other's: the fixed-point exponents follow the tile."""
    snap = synth.lamb_oseen(64)
    rng = np.random.default_rng(3)
    snap.u[:] = rng.normal(size=snap.u.shape)
    snap.v[:] = rng.normal(size=snap.v.shape)
    snap.u[:, :32] *= 2.0 ** -150
    snap.v[:, :32] *= 2.0 ** -150
    g = run_gpu(snap, "fp64", 20, 0.5)
    r = run_oracle(snap)
    assert rel_l2(g["P"].ravel(), r["P_cells"]) < 1e-6
    g["plan"].destroy()
