"""Multipoles of every box and level against their definition, M_k = sum q w^k / k with w = (z - c) / s,
for orders with and without compile-time kernels, odd and even (the last coefficient alone in its
plane), up to the largest, on grids from one leaf up, in both precisions; and the fields that the
mixed layout's other kernels give, into aligned and unaligned outputs.

Tolerance of M_k: each of the 64 cells, and each of the shifts up to the box, rounds terms whose
absolute values sum to at most (1/sqrt 2)^k sum |q| (the powers of a child's offset and of its
coefficients add up to that bound), so 64 + 4 (k + 4) units per level above the leaves of it.
"""
import numpy as np
import pytest

from paper_1610_04398_gb300 import api

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1610_04398_gb300 as pkg
    pkg.build()


def fields(n, dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return [torch.randn(n * n, generator=g, device="cuda", dtype=torch.float64).to(dtype) for _ in range(5)]


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("n,order", [(8, 2), (16, 3), (32, 9), (64, 10), (128, 12), (64, 20), (128, 23), (64, 24),
                                     (128, 31), (32, 40)])
def test_multipoles_are_their_definition(n, order, precision):
    plan = api.Plan(n, 1.0 / n, order, 0.6, precision=precision)
    f = torch.empty(n * n, dtype=plan.dtype, device="cuda")
    plan.rhs(*fields(n, plan.dtype, n + order), 3.0, f_out=f)
    plan.pressure_solve(torch.empty_like(f))
    h = torch.tensor(1.0 / n, dtype=plan.dtype).item()
    q = (f.double().cpu().numpy() * h * h).reshape(n, n)
    unit = 2.0 ** (-53 if precision == "fp64" else -24)
    k = np.arange(order + 1)
    L = int(np.log2(n // 8))
    for level in range(L + 1):
        side, m = 2 ** level, n >> level  # m cells a box
        c = (np.arange(m) + 0.5) / m - 0.5
        w = c[None, :] + 1j * c[:, None]
        W = w.ravel()[:, None] ** k / np.maximum(k, 1)
        qb = q.reshape(side, m, side, m).transpose(0, 2, 1, 3).reshape(side * side, m * m)
        got = plan.get_expansion("multipole", level).cpu().numpy()
        allowed = unit * (64 + 4 * (k + 4) * (L - level + 1)) * 0.7072 ** k * np.abs(qb).sum(1)[:, None]
        err = np.abs(got - qb @ W)
        assert (err <= allowed).all(), (level, np.max(err / allowed))
    plan.destroy()


@pytest.mark.parametrize("n,order,theta", [(64, 10, 0.6), (256, 15, 0.75), (512, 18, 0.5), (2048, 10, 0.75),
                                           (8192, 20, 0.75)])
def test_mixed_fields_on_the_plane_layout(n, order, theta):
    """Orders without compile-time kernels, and leaf multipoles beyond the L2 (8192^2, order 20: a thread
    a box, the sources one by one).  The mixed plan against the FP64 plan of the same order, lists and fields: rounding only, below the
    mixed path's bar of 1e-4; and into an output off the 16-byte boundary."""
    P64 = torch.empty(n * n, dtype=torch.float64, device="cuda")
    plan = api.Plan(n, 1.0 / n, order, theta, precision="fp64")
    f32 = fields(n, torch.float32, n)
    plan.rhs(*[a.double() for a in f32], 0.0)
    plan.pressure_solve(P64)
    plan.destroy()
    buf = torch.empty(n * n + 1, dtype=torch.float32, device="cuda")
    plan = api.Plan(n, 1.0 / n, order, theta, precision="mixed", tile=128)
    plan.rhs(*f32, 0.0)
    for out in (buf[:-1], buf[1:]):
        plan.pressure_solve(out)
        assert float((out.double() - P64).norm() / P64.norm()) < 1e-4
    plan.destroy()
