"""The cluster mailbox of the node-shared kernel.  Between rank 0's reads of
the last step's words and the FP64 check of another CTA lies no barrier of the
cluster when there are neither projectors nor solution vectors, so the check
stores to a word that no step reads.  A lost race would show on the GPU as a
wrong alpha or as unmatched barriers, so the words are compared in the source;
the GPU test runs that path on clusters whose CTAs have next to nothing to
check."""
import os
import re

import numpy as np
import pytest

from synthetic import make_workload
from tests.gpu_helpers import rel_err

SRC = os.path.join(os.path.dirname(__file__), "..", "paper_1907_02604_gb300", "csrc", "md_krylov.cu")


def test_check_has_a_mailbox_word_of_its_own():
    src = open(SRC).read()
    words = int(re.search(r"mbox\[kMaxC\]\[(\d+)\]", src).group(1))
    head, check = src.split("mixed precision: the last step once more", 1)
    stored = {int(k) for k in re.findall(r"smem_addr\(&S\.mbox\[rank\]\[(\d+)\]\)", check)}
    # words 0..3 through lane & 3 and the loop over k, the rest by number
    read = {0, 1, 2, 3} | {int(k) for k in re.findall(r"S\.mbox\[\w+\]\[(\d+)\]", head)} | {5, 6}
    assert stored and max(stored) < words
    assert not stored & read


def test_cluster_meets_before_the_first_remote_store():
    """Shared memory of another CTA may be written once that CTA runs."""
    src = open(SRC).read()
    kernel = src[src.index("k_krylov(const __grid_constant__ KrylovParams P) {"):]
    start = kernel[:kernel.index("st.shared::cluster")]
    assert "k_sync();" in start


@pytest.mark.gpu
def test_mixed_check_on_thin_slabs():
    """Without projectors every sum of a mixed call has a fixed order: the same
    bits run after run, and those of the FP64 call to 1e-11 (x_jp(j) is in error
    by tol^2 / Im z and by rounding)."""
    from paper_1907_02604_gb300 import Hamiltonian, SolverOptions, density, make_poles
    hw = [0, 1, 2, 3, 4, 5, 6, 7, 8, 0, 1, 1, 3, 6]   # one point among 17^3: CTAs without a plane
    w = make_workload("tiny", shape=(24, 24, 24), n_nodes=len(hw), n_atoms=6, spacing=(0.6, 0.6, 0.6), fd_order=4,
                      n_poles=4)
    w.halfwidth = np.array(hw, dtype=np.int32)
    ham = Hamiltonian.from_workload(w)
    z, wt = make_poles(w.kT, w.mu, *ham.spectral_bounds(), w.n_poles)
    want = density(ham, z, wt, w.nodes, w.halfwidth, SolverOptions(tol=1e-10), energy=True)
    first = None
    for _ in range(30):
        rho, e, st = density(ham, z, wt, w.nodes, w.halfwidth, SolverOptions(tol=1e-10, precision="mixed"), energy=True)
        assert st["n_converged"] == w.n_systems
        first = first or (rho, e)
        assert rho.equal(first[0]) and e.equal(first[1])
    assert rel_err(first[0].cpu().numpy(), want[0].cpu().numpy()) <= 1e-11
