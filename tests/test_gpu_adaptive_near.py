"""The adaptive solve's near field over every relation of two leaves' levels: the same level and
one level apart (kernel values held in registers), two and three apart (read per pair), four apart
(summed directly), each with the fine block on either side of the coarse ones, against the
oracle's direct sum on every cell.

Tolerances.  FP64 at p = 30, theta = 0.4: truncation below theta^31 = 5e-13 of the sum of |q log r|,
allowed 1e-11 relative l2.  Mixed: the FP32 level of the adaptive mixed path's tests, 1e-5.
"""
import numpy as np
import pytest

import oracle
from paper_1610_04398_gb300 import api, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1610_04398_gb300 as pkg
    pkg.build()
    oracle.build()


def _jump(fine):
    """Level-2 blocks, one of them (1, 2) split straight down to level ``fine``."""
    lv, ix, iy = [], [], []
    n = 1 << (fine - 2)
    for y in range(4):
        for x in range(4):
            if (x, y) != (1, 2):
                lv.append(2), ix.append(x), iy.append(y)
            else:
                lv += [fine] * n * n
                ix += [x * n + k % n for k in range(n * n)]
                iy += [y * n + k // n for k in range(n * n)]
    return tuple(np.array(a, np.int32) for a in (lv, ix, iy))


@pytest.mark.parametrize("fine", [2, 3, 4, 5, 6])
def test_level_differences_match_direct_sum(fine):
    lay = _jump(fine)
    xs, ys, hs = synth.block_cells(*lay)
    q = (np.random.default_rng(fine).normal(size=xs.size) + 0.5) * hs ** 2
    ref = oracle.green_sum_var(xs, ys, q, hs, xs, ys)
    t = api.AdaptiveTree(*lay, theta=0.4)
    P = t.solve(torch.from_numpy(q).cuda(), 30).cpu().numpy()
    # the mixed solve reads q at any alignment
    buf = torch.zeros(q.size + 1, dtype=torch.float32, device="cuda")
    buf[1:] = torch.from_numpy(q).float()
    Pm = t.solve_mixed(buf[1:], 20).double().cpu().numpy()
    t.destroy()
    e, em = (np.linalg.norm(a - ref) / np.linalg.norm(ref) for a in (P, Pm))
    print(f"levels 2 and {fine}: FP64 {e:.2e}, mixed {em:.2e}")
    assert e < 1e-11 and em < 1e-5


@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_non_finite_weight_reaches_every_cell(value):
    lay = _jump(4)
    _, _, hs = synth.block_cells(*lay)
    q = np.random.default_rng(0).normal(size=hs.size) * hs ** 2
    q[70] = value
    t = api.AdaptiveTree(*lay, theta=0.5)
    P = t.solve(torch.from_numpy(q).cuda(), 12)
    Pm = t.solve_mixed(torch.from_numpy(q).float().cuda(), 12)
    assert not torch.isfinite(P).any() and not torch.isfinite(Pm).any()
    t.destroy()
