"""Rounding of the FP64 paths, without the truncation that hides it elsewhere: plans against the same
multipole sum (lists, order, truncation) in long double, adaptive solves at an acceptance and order whose
truncation (0.25^31) is below rounding against the direct sum in long double.

Allowed for plans: 10 units (2^-53) of the field in l2.  A value is the sum of a constant, a far and a near part, each
up to a few times the field and each rounded once or twice at its own size, and of sums of some hundred
terms whose roundings add up to a few units more.  Allowed for adaptive solves, where the terms of some
fields cancel to a hundredth of their size: the error of the direct sum in FP64, term after term.
The fields cover what weights relative to a
common exponent could lose: smooth ones, a wall of large weights in small ones, a violent patch, halves of
very different size, and noise.
"""
import numpy as np
import pytest

import fmm_reference as ref
from paper_1610_04398_gb300 import api, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
ALLOWED = 10 * 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1610_04398_gb300 as pkg
    pkg.build()


def fields(kind, n):
    rng = np.random.default_rng(n)
    if kind == "wall":
        s = synth.cylinder_flow(n, diameter=0.3, centre=(0.5, 0.5), n_surface=128, seed=11)
        return [s.u, s.v, s.chi, s.usx, s.usy], s.lam
    if kind == "smooth":
        s = synth.lamb_oseen(n)
        return [s.u, s.v, s.chi, s.usx, s.usy], 0.0
    f = [rng.normal(size=(n, n)) for _ in range(5)]
    for a in f:
        if kind == "patch":
            a[n // 4:n // 4 + 6, n // 4:n // 4 + 6] *= 1e4
        if kind == "halves":  # sources 2^-20 of the other half's
            a[:, :n // 2] *= 2.0 ** -10
    return f, 0.0


def rel(a, b):
    return float(np.sqrt(((a - b) ** 2).sum() / (b ** 2).sum()))


@pytest.mark.parametrize("kind", ["wall", "smooth", "patch", "halves", "noise"])
@pytest.mark.parametrize("n,order,theta", [(64, 20, 0.5), (64, 8, 0.95), (64, 23, 0.25), (32, 12, 0.6), (128, 16, 0.75)])
def test_plan(n, order, theta, kind):
    F, lam = fields(kind, n)
    plan = api.Plan(n, 1.0 / n, order, theta, precision="fp64")
    f = torch.empty(n * n, dtype=torch.float64, device="cuda")
    P = torch.empty_like(f)
    plan.rhs(*[torch.tensor(np.ascontiguousarray(a), device="cuda").view(-1) for a in F], lam, f_out=f)
    plan.pressure_solve(P)
    q = f.cpu().numpy().reshape(n, n) * (1.0 / n) ** 2  # h^2 a power of two: exact
    M = ref.multipoles(q, order)
    near = ref.near(q, 1.0 / n, theta)
    L = len(M) - 1
    far = ref.far(ref.locals_(M, 1.0 / n, n, order, theta)[L], n)
    two_pi = 8 * np.arctan(ref.LD(1))
    got = P.cpu().numpy().reshape(n, n)
    # the plan's own locals evaluated exactly: what remains is the near field's and the evaluation's error
    own = ref.far(plan.get_expansion("local", L).cpu().numpy().astype(ref.CLD), n)
    size = np.sqrt(((near + far) ** 2).mean())
    e_far, e_near = (float(np.sqrt((x ** 2).mean()) / size) for x in (own - far, got * two_pi - own - near))
    e = rel(got, (near + far) / two_pi)
    print(f"{kind} n {n} p {order} theta {theta}: {e / 2 ** -53:.1f} units (far {e_far / 2 ** -53:.1f}, near {e_near / 2 ** -53:.1f})")
    assert e <= ALLOWED and e_far <= ALLOWED and e_near <= ALLOWED
    plan.destroy()


@pytest.mark.parametrize("kind", ["noise", "patch", "smooth", "levels"])
@pytest.mark.parametrize("levels", [(2, 4), (1, 5)])
def test_adaptive(levels, kind):
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
    tree = api.AdaptiveTree(lv, ix, iy, theta=0.25)
    P = torch.empty(q.size, dtype=torch.float64, device="cuda")
    tree.solve(torch.tensor(q, device="cuda"), 30, P)
    at = np.sort(rng.choice(q.size, 200, replace=False))
    X, Y, Q = (a.astype(ref.LD) for a in (xs, ys, q))
    rho = np.exp(ref.C0) * hs.astype(ref.LD)
    r2 = np.maximum((X[at, None] - X) ** 2 + (Y[at, None] - Y) ** 2, rho ** 2)
    K, two_pi = np.log(r2) / 2, 8 * np.arctan(ref.LD(1))
    want = K @ Q / two_pi
    plain = np.add.accumulate(K.astype(np.float64) * q, axis=1)[:, -1] / two_pi
    e, allowed = rel(P.cpu().numpy()[at], want), rel(plain, want)
    print(f"{kind} levels {levels} ({len(lv)} leaves): {e / 2 ** -53:.1f} units, allowed {allowed / 2 ** -53:.1f}")
    assert e <= allowed


@pytest.mark.parametrize("h", [1e-9, 3.7, 1e8])
def test_cell_sizes_beyond_the_table(h):
    """log h beyond what the near-field table holds enters through the monopoles: against the plan with
    h = 1 on the same q = h^2 f, which differs by log h sum q / (2 pi)."""
    n, order = 64, 12
    rng = np.random.default_rng(1)
    u, v = (torch.tensor(rng.normal(size=n * n), device="cuda") for _ in range(2))
    z = torch.zeros_like(u)
    out = []
    for s in (1.0, h):
        plan = api.Plan(n, s, order, 0.6, precision="fp64")
        f, P = torch.empty_like(u), torch.empty_like(u)
        plan.rhs(u, v, z, z, z, 0.0, f_out=f)  # f scales by 1 / h^2: the weights are the same
        plan.pressure_solve(P)
        out.append((P.cpu().numpy(), f.cpu().numpy() * s * s))
        plan.destroy()
    (P0, q), (P1, q1) = out
    assert rel(q1, q) < 8 * 2.0 ** -53
    size = np.abs(q).sum() * (abs(np.log(h)) + 5) / (2 * np.pi)  # a bound of the terms
    assert np.max(np.abs(P1 - P0 - np.log(h) * q.sum() / (2 * np.pi))) < 8 * 2.0 ** -53 * size
