"""Mixed-precision translations against the FP64 plan of the same order and acceptance parameter
(the same lists and the same truncation, so only rounding differs), on every cell: at 2048^2 the
sources at rotated offsets are grouped, at 1024^2 and below threads share a box and take the sources
one by one; the multipoles lie in planes of coefficient pairs at every size.

Tolerance 2e-5 of the field in l2, worst cell 1e-4 of the largest value: FP32 rounding (some hundred
terms a cell at 6e-8 each, summed).  A source left out or rotated the wrong way in a list of tens
moves the field by percents.
"""
import pytest

from paper_1610_04398_gb300 import synth
from gpu_cases import rel_l2, run_gpu, worst_cell

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1610_04398_gb300 as pkg
    pkg.build()


@pytest.mark.parametrize("n,order,theta,tile", [(2048, 12, 0.75, 128), (2048, 12, 0.4, 16), (2048, 16, 0.6, 128),
                                                (2048, 20, 0.5, 16), (2048, 24, 0.25, 16), (1024, 24, 0.5, 16),
                                                (1024, 12, 0.95, 16), (256, 16, 0.5, 128)])
def test_mixed_matches_fp64_plan(n, order, theta, tile):
    snap = synth.cylinder_flow(n, diameter=0.2, centre=(0.4, 0.45), n_surface=100, seed=order)
    a = run_gpu(snap, "mixed", order, theta, tile=tile)
    b = run_gpu(snap, "fp64", order, theta)
    e, w = rel_l2(a["P"], b["P"]), worst_cell(a["P"], b["P"])
    print(f"n {n} p {order} theta {theta}: l2 {e:.2e} worst cell {w:.2e}")
    assert e <= 2e-5
    assert w <= 1e-4
    a["plan"].destroy()
    b["plan"].destroy()
