"""Rounding of mixed-precision adaptive solves on cells of three to five sizes, against the direct sum in
FP64 on the same FP32 weights.  Acceptance 0.5 at order 20 leaves truncation far below FP32.

Allowed: 1.5 times the error of the direct sum in FP32, terms added in pairs (numpy): FP32 products and
sums over blocks of cells, whose partial sums are added with their errors kept, should not do worse.
"""
import numpy as np
import pytest

from paper_1610_04398_gb300 import api, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1610_04398_gb300 as pkg
    pkg.build()


@pytest.mark.parametrize("kind", ["noise", "patch", "smooth", "levels"])
@pytest.mark.parametrize("levels", [(2, 4), (1, 5), (2, 6)])
def test_mixed_solve(levels, kind):
    lv, ix, iy = synth.adaptive_blocks(*levels, centre=(0.4, 0.5), radius=0.1, band=2.0)
    xs, ys, hs = synth.block_cells(lv, ix, iy)
    rng = np.random.default_rng(len(lv))
    q = rng.normal(size=xs.size)
    if kind == "smooth":
        q = np.exp(-((xs - 0.4) ** 2 + (ys - 0.5) ** 2) / 0.02)
    if kind != "levels":  # else weights of one size on cells of all sizes
        q *= hs ** 2
    if kind == "patch":
        q[np.hypot(xs - 0.45, ys - 0.5) < 0.03] *= 1e6
    q = q.astype(np.float32)
    at = np.sort(rng.choice(q.size, 300, replace=False))
    c0 = np.pi / 4 - 1.5 - 0.5 * np.log(2.0)
    r2 = np.maximum((xs[at, None] - xs) ** 2 + (ys[at, None] - ys) ** 2, (np.exp(c0) * hs) ** 2)
    K = np.log(r2) / 2
    want = (K * q.astype(np.float64)).sum(1)
    plain = (K.astype(np.float32) * q).sum(1, dtype=np.float32)
    tree = api.AdaptiveTree(lv, ix, iy, theta=0.5)
    P = torch.empty(q.size, dtype=torch.float32, device="cuda")
    tree.solve_mixed(torch.tensor(q, device="cuda"), 20, P)
    got = 2 * np.pi * P.double().cpu().numpy()[at]
    e, allowed = (np.linalg.norm(a - want) / np.linalg.norm(want) for a in (got, plain))
    print(f"{kind} levels {levels}: {e:.2e}, plain FP32 {allowed:.2e}")
    assert e <= 1.5 * allowed
