"""FP64 calls on the node-shared kernel are as exact as on the FP64 kernels."""
import numpy as np
import pytest

from synthetic import make_workload

pytestmark = pytest.mark.gpu


def _spiked(spike, nodes=24, s=8):
    """Bulk cell whose potential is `spike` at one point outside every region:
    the regions' operators are untouched, the fixed-point scale follows it."""
    from paper_1907_02604_gb300 import Hamiltonian
    w = make_workload("bulk_mixed").subset(np.arange(nodes))
    w.halfwidth[:] = s
    n = np.array(w.shape)
    c = w.node_coords()
    for g in range(0, w.n_grid, 977):
        p = np.array([g % n[0], g // n[0] % n[1], g // (n[0] * n[1])])
        d = np.abs(c - p)
        if (np.minimum(d, n - d).max(1) > s + 4).all():
            break
    ham = Hamiltonian.from_workload(w)
    if spike:
        V = ham.potential()
        V[g] = spike
        ham.set_potential(V)
    return w, ham


@pytest.mark.parametrize("spike", [0.0, 400.0])
def test_rules_as_exact_as_the_fp64_kernel(spike):
    """The two kernels' lowest nodes.  Both round the Jacobi matrix (entries of
    10 to 20 Ha) and its QR to half an ulp, 2e-15 Ha; nodes of small weight
    answer with about three times that, 5e-15 a side.  Products cut to 2^-57 of
    the scale were off by 1e-13 Ha in alpha after 40 steps."""
    from paper_1907_02604_gb300 import lssgq_rules
    w, ham = _spiked(spike)
    lam = [lssgq_rules(ham, w.nodes, w.halfwidth, K=40, precision="fp64", block=b).lam.cpu().numpy()[:, :6]
           for b in (0, 1024)]
    assert np.sqrt(np.mean((lam[0] - lam[1]) ** 2)) <= 1.2e-14


def _both(f):
    per_pole = dict(kernel="generic", block=256, ctas_per_sm=1)
    return [x.cpu().numpy() for x in (f({}), f(per_pole))]


@pytest.mark.parametrize("spike", [1e5, 1e7])
def test_potential_that_is_high_elsewhere(spike):
    """FP64 calls whose regions do not touch a high potential: rules are the FP64
    kernel's, densities and a plan made before the potential rose those of the
    per-pole kernels to 1e-11 (tol 1e-11; x_jp(j) is in error by tol^2 / Im z
    and by rounding, a few 1e-13).  Steps of 2^-62 of the scale were off by up to
    1e-7 and 6e-9."""
    import torch
    from paper_1907_02604_gb300 import Plan, SolverOptions, density, lssgq_rules, make_poles
    w, ham = _spiked(0.0, nodes=8)
    low = ham.potential()
    _, high = _spiked(spike, nodes=8)
    z, wt = make_poles(0.01, 0.2, -10.0, 46.0, 16)
    o = SolverOptions(tol=1e-11)
    plan = Plan(ham, z, wt, w.nodes, w.halfwidth, o)
    plan.launch()
    plan.stats()
    before = plan.rho.clone()
    V = high.potential()
    ham.set_potential(V)
    lam = [lssgq_rules(ham, w.nodes, w.halfwidth, K=40, precision="fp64", block=b).lam for b in (0, 1024)]
    assert torch.equal(*lam)
    r, ref = _both(lambda k: density(ham, z, wt, w.nodes, w.halfwidth, SolverOptions(tol=1e-11, **k))[0])
    assert np.abs(r - ref).max() <= 1e-11 * np.abs(ref).max()
    for _ in range(2):
        plan.launch()
        st = plan.stats()
        assert st["n_converged"] == 8 * 16
        assert np.abs(plan.rho.cpu().numpy() - ref).max() <= 1e-11 * np.abs(ref).max()
    ham.set_potential(low)
    plan.launch()
    plan.stats()
    assert np.abs((plan.rho - before).cpu().numpy()).max() <= 1e-11 * np.abs(ref).max()


@pytest.mark.parametrize("tol,spike", [(1e-11, 0.0), (1e-12, 0.0), (1e-13, 0.0), (1e-10, 1e3), (1e-10, 1e5)])
def test_mixed_calls_converge_to_their_tolerance(tol, spike):
    """Tolerances near the fixed-point kernel's own steps, and steps made coarse
    by a potential that is high elsewhere: the true residual has to meet tol, as
    it does with the FP32 kernels' refreshed residuals.  An x_jp(j) is in error by
    e_j^T (H - z)^-1 r <= tol / Im z (FP32 iterates are not Galerkin solutions),
    a density by 2 / dV sum |w_p| of that, and by rounding, 1e-12."""
    from paper_1907_02604_gb300 import Plan, SolverOptions, density, make_poles
    w, ham = _spiked(0.0, nodes=8)
    _, high = _spiked(spike, nodes=8)
    z, wt = make_poles(0.01, 0.2, -10.0, 46.0, 16)
    per_pole = dict(kernel="generic", block=256, ctas_per_sm=1)
    ref = density(ham, z, wt, w.nodes, w.halfwidth, SolverOptions(tol=1e-12, **per_pole))[0]
    bound = 2 / ham.dV * tol * np.sum(np.abs(wt) / z.imag) + 1e-12 * float(ref.abs().max())
    o = SolverOptions(tol=tol, precision="mixed")
    plan = Plan(ham, z, wt, w.nodes, w.halfwidth, o)     # made before the potential rises
    ham.set_potential(high.potential())
    rho, _, st = density(ham, z, wt, w.nodes, w.halfwidth, o, strict=False)
    plan.launch()
    for r, q in ((rho, st), (plan.rho, plan.stats(strict=False))):
        assert q["n_converged"] == 8 * 16 and q["max_resid"] <= tol
        assert float((r - ref).abs().max()) <= bound


@pytest.mark.parametrize("n_nodes,K", [(1, 1), (3, 128), (700, 8)])
def test_first_moment_is_the_diagonal(n_nodes, K):
    """sum_k w_k lambda_k = H_jj, the stencil's diagonal plus V_j: the QR keeps
    it to a few ulp of max |lambda| a sweep, 300 sweeps at most (K = 128)."""
    from paper_1907_02604_gb300 import Hamiltonian, fd_weights, lssgq_rules
    w = make_workload("tiny", shape=(12, 12, 12), n_nodes=n_nodes, s=2, n_atoms=3, spacing=(0.6, 0.55, 0.5))
    ham = Hamiltonian.from_workload(w)
    r = lssgq_rules(ham, w.nodes, w.halfwidth, K=K)
    lam, wt = r.lam.cpu().numpy(), r.weight.cpu().numpy()
    diag = sum(-0.5 * fd_weights(w.fd_order)[0] / h ** 2 for h in w.spacing)
    want = diag + ham.potential().cpu().numpy()[w.nodes]
    assert np.abs((lam * wt).sum(1) - want).max() <= 1e-12 * np.abs(lam).max()
