"""The default route gives the same bits run after run: records, projections
and norms are summed in an order (or in integers) that no race decides."""
import numpy as np
import pytest

from synthetic import make_workload

pytestmark = pytest.mark.gpu


def _bulk(nodes, hw):
    from paper_1907_02604_gb300 import Hamiltonian, make_poles
    w = make_workload("bulk_mixed").subset(np.arange(nodes))
    w.halfwidth[:] = hw
    ham = Hamiltonian.from_workload(w)
    z, wt = make_poles(w.kT, w.mu, *ham.spectral_bounds(), w.n_poles)
    return w, ham, z, wt


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_overlapping_projectors(precision):
    """Up to four atoms' rows meet at a point here; two sizes of region."""
    from paper_1907_02604_gb300 import SolverOptions, density
    w, ham, z, wt = _bulk(12, [10, 6] * 6)
    o = SolverOptions(tol=1e-10, precision=precision)
    first = None
    for _ in range(12):
        rho, e, st = density(ham, z, wt, w.nodes, w.halfwidth, o, energy=True)
        first = first or (rho, e, st)
        assert rho.equal(first[0]) and e.equal(first[1])
        assert all(st[k] == first[2][k] for k in ("total_iters", "max_resid"))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_asynchronous_calls(precision):
    """Calls that only enqueue fork to side streams, a class of sizes on each."""
    import torch
    from paper_1907_02604_gb300 import SolverOptions, density
    w, ham, z, wt = _bulk(10, [8, 3, 6, 2, 5, 4, 7, 1, 3, 0])
    o = SolverOptions(tol=1e-10, precision=precision)
    rho, e, _ = density(ham, z, wt, w.nodes, w.halfwidth, o, energy=True)
    for _ in range(5):
        r, f, st = density(ham, z, wt, w.nodes, w.halfwidth, o, energy=True, sync=False)
        torch.cuda.synchronize()
        assert st is None and r.equal(rho) and f.equal(e)
