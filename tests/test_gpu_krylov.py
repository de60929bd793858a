"""The node-shared Krylov kernel (the default route) against the per-pole
kernel (forced by a launch shape) on the same inputs, at the sizes where it
can go wrong: every stencil order, regions from one point up, odd batches of
unequal regions, projectors that wrap, the 32-step updates of the solution
vectors, iteration caps, changed potentials.

Tolerances: both sides stop at ||r|| <= tol with ||e_j|| = 1.  x_jp(j) is a
bilinear form, in error by r^T (H - z)^-1 r <= tol^2 / Im z, far below
rounding; at tol = 1e-11 and the poles used (Im z > 0.02) the densities agree
to 1e-11 of their size (rounding amplified by |w_p| |x|, at most a few
thousand ulp).  Solution vectors differ by 2 tol / Im z <= 1e-9, sums over
the poles by |w_p| times that: 1e-8 of the largest entry.
"""
import numpy as np
import pytest

from synthetic import make_workload
from tests.gpu_helpers import rel_err

pytestmark = pytest.mark.gpu

PER_POLE = dict(kernel="generic", block=256, ctas_per_sm=1)


def _system(halfwidth=None, **kw):
    from paper_1907_02604_gb300 import Hamiltonian, make_poles
    w = make_workload("tiny", **kw)
    if halfwidth is not None:
        w.halfwidth = np.array(halfwidth, dtype=np.int32)
    ham = Hamiltonian.from_workload(w)
    z, wt = make_poles(w.kT, w.mu, *ham.spectral_bounds(), w.n_poles)
    return w, ham, z, wt


def _both(w, ham, z, wt, tol=1e-11, precision="fp64", **kw):
    from paper_1907_02604_gb300 import SolverOptions, density
    out = []
    for shape in ({}, PER_POLE):
        o = SolverOptions(tol=tol, precision=precision if not shape else "fp64", **shape, **kw)
        rho, e, st = density(ham, z, wt, w.nodes, w.halfwidth, o, energy=True, strict=False)
        out.append((rho.cpu().numpy(), e.cpu().numpy(), st))
    return out


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("order", [2, 4, 6, 8])
@pytest.mark.parametrize("nonlocal_proj", [False, True])
def test_orders_and_unequal_regions(order, nonlocal_proj, precision):
    # nine sizes in one batch, one point to 17^3; with projectors every region
    # meets atoms through the periodic boundary
    w, ham, z, wt = _system(shape=(20, 18, 22), n_nodes=9, n_atoms=5, fd_order=order, spacing=(0.5, 0.55, 0.5),
                            nonlocal_proj=nonlocal_proj, halfwidth=[0, 1, 2, 3, 4, 5, 6, 7, 8])
    (r0, e0, s0), (r1, e1, s1) = _both(w, ham, z, wt, precision=precision)
    assert s0["n_converged"] == s1["n_converged"] == w.n_systems
    assert rel_err(r0, r1) <= 1e-10 and rel_err(e0, e1) <= 1e-10
    # the same Krylov spaces: the steps to tol agree but for rounding
    assert abs(s0["total_iters"] - s1["total_iters"]) <= 0.03 * s1["total_iters"] + w.n_systems


def test_more_sizes_than_classes():
    w, ham, z, wt = _system(shape=(36, 36, 36), n_nodes=15, n_atoms=6, spacing=(0.6, 0.6, 0.6), fd_order=4,
                            halfwidth=[14, 2, 7, 1, 13, 3, 11, 5, 12, 4, 10, 6, 9, 8, 0], n_poles=4)
    (r0, e0, _), (r1, e1, _) = _both(w, ham, z, wt)
    assert rel_err(r0, r1) <= 1e-10 and rel_err(e0, e1) <= 1e-10


@pytest.mark.parametrize("n_poles", [2, 34, 64])
def test_pole_counts_and_rows(n_poles):
    """Poles beyond one warp, and rows of the density matrix (solution
    vectors over the region) against the per-pole kernel's."""
    from paper_1907_02604_gb300 import SolverOptions, density_matrix_rows
    w, ham, z, wt = _system(shape=(18, 18, 18), n_nodes=4, n_atoms=6, fd_order=8, spacing=(0.5, 0.5, 0.5),
                            nonlocal_proj=True, halfwidth=[3, 6, 7, 1], n_poles=n_poles)
    rows = []
    for shape in ({}, PER_POLE):
        r = density_matrix_rows(ham, z, wt, w.nodes, w.halfwidth, SolverOptions(tol=1e-11, **shape))
        rows.append([t.cpu().numpy() for t in r[:3]])
    assert rel_err(rows[0][0], rows[1][0]) <= 1e-10
    assert rel_err(rows[0][2], rows[1][2]) <= 1e-8


@pytest.mark.parametrize("maxit", [1, 31, 32, 33, 64])
def test_checkpoint_at_the_iteration_cap(maxit):
    """The iterate at a capped step is the same Galerkin solution on both
    routes, whatever part of a 32-step update the cap leaves."""
    from paper_1907_02604_gb300 import SolverOptions, Workspace, density, density_adjoint
    import torch
    w, ham, z, wt = _system(shape=(16, 15, 14), n_nodes=3, n_atoms=4, fd_order=8, spacing=(0.5, 0.5, 0.5),
                            halfwidth=[5, 6, 4])
    a = torch.linspace(-1, 1, 3, dtype=torch.float64, device="cuda")
    out = []
    for shape in ({}, PER_POLE):
        ws = Workspace(ham, w.nodes, w.halfwidth, w.n_poles)
        o = SolverOptions(tol=1e-13, maxit=maxit, **shape)
        rho, _, st = density(ham, z, wt, w.nodes, w.halfwidth, o, checkpoint=ws, strict=False)
        g, f = density_adjoint(ham, z, wt, w.nodes, w.halfwidth, a, None, o, checkpoint=ws, forces=True)
        assert st["iters_max"] <= maxit
        out.append((rho.cpu().numpy(), g.cpu().numpy(), f.cpu().numpy()))
    # unconverged iterates depend on the step alone: 64 steps of rounding, conditioned by |H| / Im z ~ 1e3
    for x, y in zip(*out):
        assert rel_err(x, y) <= 1e-9


def test_fused_adjoint_and_checkpoint_agree():
    from paper_1907_02604_gb300 import SolverOptions, Workspace, density, density_adjoint, density_fused_adjoint
    import torch
    w, ham, z, wt = _system(shape=(20, 18, 16), n_nodes=5, n_atoms=6, fd_order=8, spacing=(0.5, 0.5, 0.5),
                            halfwidth=[3, 7, 5, 2, 6], n_poles=16)
    b = torch.linspace(0.5, 2, 5, dtype=torch.float64, device="cuda")
    o = SolverOptions(tol=1e-10, precision="mixed")
    ws = Workspace(ham, w.nodes, w.halfwidth, w.n_poles)
    density(ham, z, wt, w.nodes, w.halfwidth, o, checkpoint=ws)
    g0, f0 = density_adjoint(ham, z, wt, w.nodes, w.halfwidth, torch.zeros_like(b), b, o, checkpoint=ws, forces=True)
    _, _, g1, f1, _ = density_fused_adjoint(ham, z, wt, w.nodes, w.halfwidth, None, b, o, forces=True)
    assert rel_err(g1.cpu().numpy(), g0.cpu().numpy()) <= 1e-12      # the same vectors, summed in another order
    assert rel_err(f1.cpu().numpy(), f0.cpu().numpy()) <= 1e-10


def test_plan_follows_a_potential_of_another_scale():
    """A plan captured for one spectral range and relaunched after a potential
    that needs a larger fixed-point scale."""
    from paper_1907_02604_gb300 import Plan, SolverOptions, density
    w, ham, z, wt = _system(shape=(16, 16, 16), n_nodes=4, s=4, n_atoms=4, spacing=(0.5, 0.5, 0.5))
    plan = Plan(ham, z, wt, w.nodes, w.halfwidth, SolverOptions(tol=1e-11))
    plan.launch()
    plan.stats()
    V = ham.potential()
    ham.set_potential(V * 400.0)
    plan.launch()
    plan.stats()
    ref, _, _ = density(ham, z, wt, w.nodes, w.halfwidth, SolverOptions(tol=1e-11, **PER_POLE))
    assert rel_err(plan.rho.cpu().numpy(), ref.cpu().numpy()) <= 1e-10


@pytest.mark.parametrize("strength", [5.0, 20.0, 100.0])
@pytest.mark.parametrize("nonlocal_proj", [False, True])
def test_potential_dominated(strength, nonlocal_proj):
    """Where |alpha| exceeds beta an error of the recurred norms would grow from
    step to step, until a norm of zero or less ends the recurrence.  H is
    perturbed by rounding, 1e-16 ||H|| <= 1e-13, and a sum of x_jp(j) by that
    times the sum of |w_p| / Im z^2, below 1e4: 1e-9."""
    n = 20 if nonlocal_proj else 16   # (a projector has to fit the box)
    w, ham, z, wt = _system(shape=(n, n, n), n_nodes=4, s=4, n_atoms=4, spacing=(0.5, 0.5, 0.5),
                            nonlocal_proj=nonlocal_proj)
    ham.set_potential(ham.potential() * strength)
    (r0, e0, s0), (r1, e1, s1) = _both(w, ham, z, wt)
    assert s0["n_converged"] == s1["n_converged"] == w.n_systems
    assert rel_err(r0, r1) <= 1e-9 and rel_err(e0, e1) <= 1e-9


def test_non_finite_potential_is_reported():
    from paper_1907_02604_gb300 import SolverOptions, density
    w, ham, z, wt = _system(shape=(12, 12, 12), n_nodes=2, s=3, n_atoms=2, spacing=(0.5, 0.5, 0.5))
    V = ham.potential()
    bad = V.clone()
    bad[int(w.nodes[0])] = float("nan")
    ham.set_potential(bad)
    _, _, st = density(ham, z, wt, w.nodes, w.halfwidth, SolverOptions(tol=1e-10, maxit=50), strict=False)
    assert st["n_converged"] < w.n_systems
    ham.set_potential(V)
    _, _, st = density(ham, z, wt, w.nodes, w.halfwidth, SolverOptions(tol=1e-10))
    assert st["n_converged"] == w.n_systems


@pytest.mark.parametrize("shape", [(33, 9, 17), (31, 8, 8), (65, 7, 23)])
@pytest.mark.parametrize("periodic", [(True, True, True), (False, True, False)])
def test_potential_tiles(shape, periodic):
    """Grids that leave part of a 32 x 8 x 8 tile empty, wells wider than the
    box: the separable sums against the oracle's direct ones (three factors
    instead of one exponential: a few ulp of the depth per atom)."""
    from oracle import hamiltonian as oh
    from paper_1907_02604_gb300 import Hamiltonian
    w = make_workload("tiny", shape=shape, periodic=periodic, n_atoms=7, s=1, n_nodes=1)
    V = Hamiltonian.from_workload(w).potential().cpu().numpy()
    assert np.max(np.abs(V - oh.local_potential(w))) < 1e-13


@pytest.mark.parametrize("n_nodes,K", [(1, 1), (3, 128), (700, 8)])
def test_gauss_rules_grouping(n_nodes, K):
    """One node, the largest rule, and more nodes than one a warp: moments of
    the rules are those of H (exact for the node's region)."""
    from paper_1907_02604_gb300 import lssgq_rules
    w, ham, z, wt = _system(shape=(12, 12, 12), n_nodes=n_nodes, s=2, n_atoms=3, spacing=(0.6, 0.6, 0.6), fd_order=4)
    r = lssgq_rules(ham, w.nodes, w.halfwidth, K=K)
    lam, wt_ = r.lam.cpu().numpy(), r.weight.cpu().numpy()
    np.testing.assert_allclose(wt_.sum(1), 1.0, rtol=0, atol=1e-12)
    assert np.all(np.diff(lam, axis=1) >= 0)
    # the first moment is H_jj = the stencil's diagonal + V_j
    V = ham.potential().cpu().numpy()[w.nodes]
    first = (lam * wt_).sum(1) - V
    assert np.max(np.abs(first - first[0])) <= 1e-11 * np.abs(lam).max()
