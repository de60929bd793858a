"""What the node-shared kernel reports where it cannot solve: the same as the
kernels it stands in for."""
import numpy as np
import pytest

from synthetic import make_workload

pytestmark = pytest.mark.gpu


def _system(**kw):
    from paper_1907_02604_gb300 import Hamiltonian
    w = make_workload("tiny", **kw)
    return w, Hamiltonian.from_workload(w)


@pytest.mark.parametrize("precision,block", [("fp64", 0), ("fp64", 1024), ("mixed", 0)])
def test_rules_of_a_potential_that_is_not_finite(precision, block):
    """A NaN in a region gives a Jacobi matrix of NaNs, whose QR does not
    converge: an error, never rules of zeros."""
    from paper_1907_02604_gb300 import lssgq_rules
    from paper_1907_02604_gb300._lib import MacroDFTError
    w, ham = _system(shape=(14, 14, 14), n_nodes=2, s=2, n_atoms=2, spacing=(0.5, 0.5, 0.5))
    w.nodes[:] = [3 + 14 * (3 + 14 * 3), 10 + 14 * (10 + 14 * 10)]   # regions apart
    good = lssgq_rules(ham, w.nodes, w.halfwidth, K=1, precision=precision, block=block).lam.cpu().numpy()
    V = ham.potential()
    V[int(w.nodes[0]) + 1] = float("nan")
    ham.set_potential(V)
    with pytest.raises(MacroDFTError, match="MD_ERR_BREAKDOWN"):
        lssgq_rules(ham, w.nodes, w.halfwidth, K=8, precision=precision, block=block)
    # one node a rule: nothing to iterate, and the NaN is the answer
    lam = lssgq_rules(ham, w.nodes, w.halfwidth, K=1, precision=precision, block=block).lam.cpu().numpy()
    assert np.isnan(lam[0, 0]) and lam[1, 0] == good[1, 0]
