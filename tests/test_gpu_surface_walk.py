"""The surface pass (tree-code walk, tractions and force sums in one launch) where its lists and
its grid change: the strictest acceptance (a lane's list of accepted boxes fills and is flushed),
points outside the domain (the walk starts at the root), point counts that leave part of a CTA idle
and more points than one sweep of the grid covers, in both precisions, against the oracle.

Tolerances: FP64 truncation 10 theta^(p+1); mixed 1e-4 (the mixed path's bar)."""
import numpy as np
import pytest

import oracle
from paper_1610_04398_gb300 import api, synth
from gpu_cases import rel_l2, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1610_04398_gb300 as pkg
    pkg.build()
    oracle.build()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("npts,theta_s", [(1, 0.5), (9, 0.25), (533, 0.25), (20001, 0.6)])
def test_surface_pressure_and_forces(precision, npts, theta_s):
    snap = synth.cylinder_flow(256, diameter=0.3, centre=(0.5, 0.5), n_surface=max(npts, 3), seed=npts)
    pts, nrm = snap.points[:npts].copy(), snap.normals[:npts].copy()
    if npts > 8:
        pts[5], pts[6] = (1.4, 0.5), (-0.3, -0.2)
    plan = api.Plan(256, snap.h, 12, 0.6, precision=precision, lift=snap.lift, theta_surface=theta_s)
    f = [to_dev(a, plan.dtype) for a in (snap.u, snap.v, snap.chi, snap.usx, snap.usy)]
    per = torch.empty(npts * 5, dtype=torch.float64, device="cuda")
    forces = torch.empty(6, dtype=torch.float64, device="cuda")
    dS = torch.full((npts,), 0.01, dtype=torch.float64, device="cuda")
    plan.rhs(*f, snap.lam)
    for _ in range(2):  # the arrival counter is reset
        plan.surface_traction(f[0], f[1], to_dev(pts, torch.float64), to_dev(nrm, torch.float64), snap.nu, dS=dS,
                              per_point=per, forces=forces)
    per = per.view(npts, 5).cpu().numpy()
    at = np.arange(npts) if npts < 1000 else np.unique(np.r_[0:40, np.random.default_rng(0).choice(npts, 400), npts - 1])
    q = oracle.source_weights(oracle.rhs(snap.u, snap.v, snap.chi, snap.usx, snap.usy, h=snap.h, lam=snap.lam), snap.h)
    ref = oracle.green_sum_grid(q, snap.h, pts[at, 0], pts[at, 1])
    tol = max(10 * theta_s ** 13, 1e-12) if precision == "fp64" else 1e-4
    assert rel_l2(per[at, 0], ref) < tol
    assert np.allclose(per[:, 1:3], -per[:, :1] * nrm, rtol=1e-14, atol=0)
    F = 0.01 * per[:, 1:].sum(0)
    assert np.allclose(forces.cpu().numpy()[:4], F, rtol=1e-9, atol=1e-9 * np.abs(0.01 * per[:, 1:]).sum())
    plan.destroy()


@pytest.mark.parametrize("order", [10, 12, 16, 20, 24])
def test_more_points_than_one_wave(order):
    """The form for more points than a wave holds (from 3649 on 152 SMs) against the other on the
    first points: the same FP32 operations, so rounding of the contracted ones at most (1e-6)."""
    npts = 24 * torch.cuda.get_device_properties(0).multi_processor_count + 1
    snap = synth.cylinder_flow(128, diameter=0.3, centre=(0.5, 0.5), n_surface=npts, seed=order)
    plan = api.Plan(128, snap.h, order, 0.6, precision="mixed", lift=snap.lift)
    f = [to_dev(a, plan.dtype) for a in (snap.u, snap.v, snap.chi, snap.usx, snap.usy)]
    plan.rhs(*f, snap.lam)
    out = []
    for m in (npts, npts - 1):
        per = torch.full((m * 5,), float("nan"), dtype=torch.float64, device="cuda")
        plan.surface_traction(f[0], f[1], to_dev(snap.points[:m], torch.float64), to_dev(snap.normals[:m], torch.float64),
                              snap.nu, per_point=per)
        out.append(per.view(m, 5).cpu().numpy())
    assert np.isfinite(out[0]).all()
    assert rel_l2(out[0][:-1], out[1]) < 1e-6
    plan.destroy()


def test_fp64_strict_walk_flushes_its_list():
    """Acceptance 0.25 at 1024^2: more than 224 accepted boxes a point, so a walk evaluates its list
    before its levels are done.  Allowed at each point: truncation theta^21 and 1e-14 for rounding (some
    90 units), both of sum |q log r| there (every r is below 1): one wrong or missing box shows."""
    npts = 533
    snap = synth.cylinder_flow(1024, diameter=0.3, centre=(0.5, 0.5), n_surface=npts, seed=7)
    plan = api.Plan(1024, snap.h, 20, 0.6, precision="fp64", lift=snap.lift, theta_surface=0.25)
    f = [to_dev(a, plan.dtype) for a in (snap.u, snap.v, snap.chi, snap.usx, snap.usy)]
    plan.rhs(*f, snap.lam)
    pts, nrm = to_dev(snap.points, torch.float64), to_dev(snap.normals, torch.float64)
    out = []
    for _ in range(4):
        per = torch.empty(npts * 5, dtype=torch.float64, device="cuda")
        plan.surface_traction(f[0], f[1], pts, nrm, snap.nu, per_point=per)
        out.append(per)
    assert all(torch.equal(out[0], o) for o in out)
    q = oracle.source_weights(oracle.rhs(snap.u, snap.v, snap.chi, snap.usx, snap.usy, h=snap.h, lam=snap.lam), snap.h)
    ref = oracle.green_sum_grid(q, snap.h, snap.points[:, 0], snap.points[:, 1])
    size = -oracle.green_sum_grid(np.abs(q), snap.h, snap.points[:, 0], snap.points[:, 1])
    assert (np.abs(out[0].view(npts, 5)[:, 0].cpu().numpy() - ref) < (0.25 ** 21 + 1e-14) * size).all()
    plan.destroy()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_captured_step_outlives_a_larger_call(precision):
    """A step captured with few points, a call with more than the plan's scratch held so far, a replay:
    the scratch grows without moving, so the replay gives the first launch's values bit for bit."""
    snap = synth.cylinder_flow(128, diameter=0.3, centre=(0.5, 0.5), n_surface=20001, seed=3)
    plan = api.Plan(128, snap.h, 12, 0.6, precision=precision, lift=snap.lift)
    f = [to_dev(a, plan.dtype) for a in (snap.u, snap.v, snap.chi, snap.usx, snap.usy)]
    pts, nrm = to_dev(snap.points, torch.float64), to_dev(snap.normals, torch.float64)
    few, few_nrm = pts[:400].clone(), nrm[:400].clone()  # held while the step exists
    per = torch.empty(5 * 400, dtype=torch.float64, device="cuda")
    forces = torch.zeros(6, dtype=torch.float64, device="cuda")
    P = torch.empty(128 * 128, dtype=plan.dtype, device="cuda")
    step = plan.capture_step(*f, snap.lam, p_out=P, points=few, normals=few_nrm, nu=snap.nu, per_point=per,
                             forces=forces)
    step.launch()
    first = per.clone(), forces.clone()
    before = plan.info().workspace_bytes
    plan.surface_traction(f[0], f[1], pts, nrm, snap.nu)
    assert plan.info().workspace_bytes > before  # it did grow
    spoil = torch.full((1 << 16,), float("nan"), dtype=torch.float64, device="cuda")
    per.zero_(), forces.zero_()
    step.launch()
    torch.cuda.synchronize()
    assert torch.equal(per, first[0]) and torch.equal(forces, first[1]) and torch.isnan(spoil).all()
    step.destroy()
    plan.destroy()


def test_adaptive_walk_takes_nan_points():
    """A point with a NaN coordinate accepts no box and lies within every cell's clamp: its value is sum q
    log rho_h / (2 pi), the call succeeds and the other points are what they are without it."""
    lv, ix, iy = synth.adaptive_blocks(3, 6, centre=(0.4, 0.5), radius=0.1, band=2.0)
    _, _, hs = synth.block_cells(lv, ix, iy)
    q = np.random.default_rng(0).normal(size=hs.size) * hs ** 2
    tree = api.AdaptiveTree(lv, ix, iy, theta=0.5)
    qd = to_dev(q, torch.float64)
    tree.solve(qd, 12)
    pts = synth.circle_surface(40, (0.4, 0.5), 0.1)[0]
    clean = tree.surface_pressure(qd, to_dev(pts, torch.float64), 0.5).cpu().numpy()
    bad = [3, 17]
    pts[3, 0] = pts[17, 1] = np.nan
    P = tree.surface_pressure(qd, to_dev(pts, torch.float64), 0.5).cpu().numpy()
    keep = np.setdiff1d(np.arange(40), bad)
    assert np.array_equal(P[keep], clean[keep])
    terms = q * np.log(oracle.rho_h(1.0) * hs) / (2 * np.pi)
    assert np.max(np.abs(P[bad] - terms.sum())) < 1e-14 * np.abs(terms).sum()
    tree.destroy()
