"""The FFT solve at the sizes where the lines per block of its row and column kernels change (512 and
1024: two and two, 2048: one and two, 4096: one and one in mixed precision), sampled cells against
the oracle's exact sums.

Tolerance: rms error ~ eps log2(M^2) ||q||_2 ||K||_2 / M of a transform pair of M^2 = 4 n^2 points
(Higham, Accuracy and Stability of Numerical Algorithms, Sec. 24.1, and Parseval), four times that
for the rms of the samples and forty times for the largest.
"""
import math

import numpy as np
import pytest

import oracle
from paper_1610_04398_gb300 import api, synth
from gpu_cases import to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,precision", [(512, "mixed"), (1024, "mixed"), (1024, "fp64"), (2048, "mixed"), (4096, "mixed")])
def test_fft_pairs_of_rows(n, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1610_04398_gb300 as pkg
    pkg.build()
    oracle.build()
    snap = synth.cylinder_flow(n, seed=n)
    plan = api.Plan(n, snap.h, 12, 0.75, x0=snap.x0, y0=snap.y0, precision=precision)
    dt = plan.dtype
    f = torch.empty(n * n, dtype=dt, device="cuda")
    P = torch.full((n * n,), float("nan"), dtype=dt, device="cuda")
    plan.rhs(*[to_dev(a, dt) for a in (snap.u, snap.v, snap.chi, snap.usx, snap.usy)], snap.lam, f_out=f)
    plan.pressure_solve_fft(P)
    torch.cuda.synchronize()
    npdt = np.float64 if dt == torch.float64 else np.float32
    q = (f.cpu().numpy().reshape(n, n) * (npdt(snap.h) * npdt(snap.h))).astype(np.float64)
    cells = np.unique(np.concatenate([np.random.default_rng(n).choice(n * n, 96, replace=False),
                                      [0, 1, n - 1, n, n * n - 1]]))
    X, Y = synth.cell_centres(n, snap.h, snap.x0, snap.y0)
    ref = oracle.green_sum_grid(q, snap.h, X.ravel()[cells], Y.ravel()[cells], snap.x0, snap.y0)
    d = np.arange(-(n - 1), n)
    K2 = math.sqrt(sum(float(np.sum(np.log(np.maximum(snap.h * np.hypot(d, y), oracle.rho_h(snap.h))) ** 2)) for y in d))
    eps = 2.0 ** (-53 if precision == "fp64" else -24)
    b = 4 * eps * math.log2(4 * n * n) * np.linalg.norm(q) * K2 / (2 * math.pi) / (2 * n)
    err = P.double().cpu().numpy()[cells] - ref
    print(f"{n} {precision}: rms {np.sqrt(np.mean(err ** 2)):.2e} max {np.max(np.abs(err)):.2e} bound {b:.2e}")
    assert np.isfinite(P.double().cpu().numpy()).all()
    assert np.sqrt(np.mean(err ** 2)) <= b
    assert np.max(np.abs(err)) <= 10 * b
    plan.destroy()
