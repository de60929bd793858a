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


def test_time_budget_of_many_region_sizes():
    """Twelve classes of region size, each with nodes for the whole device, and
    poles in the middle of the spectrum that none of them can reach: the budget
    is the call's, not each class's.  On top of it every node left takes its
    set-up and one step, well under 0.1 ms on a tenth of the device: 0.2 s for
    all."""
    import time
    import torch
    from paper_1907_02604_gb300 import SolverOptions, density
    from paper_1907_02604_gb300._lib import MacroDFTError
    sizes = np.repeat(np.arange(3, 15), 160)
    w, ham = _system(shape=(36, 36, 36), n_nodes=len(sizes), n_atoms=4, spacing=(0.5, 0.5, 0.5), fd_order=8)
    w.halfwidth = sizes.astype(np.int32)
    z = np.array([10.0, 12.0, 14.0, 16.0]) + 1e-9j

    def run(budget):
        with pytest.raises(MacroDFTError, match="MD_ERR_TIMEOUT"):
            density(ham, z, np.ones(4), w.nodes, w.halfwidth, SolverOptions(tol=1e-12, maxit=10 ** 8, timeout_s=budget))
        torch.cuda.synchronize()
    run(1e-6)   # allocations of a first call
    t = time.time()
    run(0.3)
    assert time.time() - t < 0.5


def test_rules_on_a_device_that_is_nearly_full():
    """FP64 rules of 33^3 regions with projectors need 131 MB on the FP64 kernel
    and 380 on the node-shared one: with 240 MB free they come from the former."""
    import torch
    from paper_1907_02604_gb300 import Hamiltonian, lssgq_rules
    w = make_workload("bulk_mixed").subset(np.arange(160))
    tw, tham = _system(shape=(20, 20, 20), n_nodes=2, s=4, n_atoms=2, spacing=(0.5, 0.5, 0.5), nonlocal_proj=True, fd_order=8)
    for block in (0, 1024):   # both kernels loaded
        lssgq_rules(tham, tw.nodes, tw.halfwidth, K=4, block=block)
    ref = Hamiltonian.from_workload(w)
    want = lssgq_rules(ref, w.nodes, w.halfwidth, K=8, block=1024).lam
    ref.close()
    ham = Hamiltonian.from_workload(w)
    torch.cuda.synchronize()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - 240 * 10 ** 6, dtype=torch.uint8, device="cuda")
    try:
        lam = lssgq_rules(ham, w.nodes, w.halfwidth, K=8).lam
        assert torch.equal(lam, want)
    finally:
        del hog
        torch.cuda.empty_cache()
