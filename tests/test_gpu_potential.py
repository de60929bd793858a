"""The local potential bit for bit.  Mixed solves amplify its last bits (the
entropies of a mixed call move by 2e-9 with them, beyond what two calls on the
same atoms may differ by), so the terms and their order are part of what a
build promises.  Digests of the potentials of the one-exponential-per-term sum
over the 27 cells around a point, taken on a GB300."""
import hashlib

import numpy as np
import pytest

from synthetic import make_workload
from synthetic.rng import stream

pytestmark = pytest.mark.gpu

DIGESTS = {
    "small_fp64": "d720ab39e57a5b64",
    "bulk_mixed": "115dabba5e154c5f",
}


def _digest(w, **kw):
    from paper_1907_02604_gb300 import Hamiltonian
    h = Hamiltonian(w.shape, w.spacing, kw.get("periodic", w.periodic), w.fd_order, kw.get("atoms", w.atoms),
                    w.depth, w.sigma, cutoff_sigmas=kw.get("cutoff", w.cutoff_sigmas), v_ext=w.v_ext)
    return hashlib.sha256(h.potential().cpu().numpy().tobytes()).hexdigest()[:16]


@pytest.mark.parametrize("name", ["small_fp64", "bulk_mixed"])
def test_workload_potential_bits(name):
    assert _digest(make_workload(name)) == DIGESTS[name]


# grids of odd sizes, open and periodic axes, one to five cells an axis, atoms
# on grid points and half a box apart (ties of the minimum image), outside the
# box, far from it
CASES = {
    "open_x": ("1dbd7eb3e9ee1d0f", dict(shape=(37, 21, 30), n_atoms=40), dict(periodic=(False, True, True), cutoff=3.0), None),
    "one_cell": ("f55db44ec702dfdb", dict(shape=(9, 11, 7), n_atoms=5), dict(cutoff=8.0), None),
    "ties": ("8519137b8b526b3f", dict(shape=(16, 12, 20), n_atoms=60, spacing=(0.5, 0.25, 0.5)), dict(cutoff=4.0), "grid"),
    "outside": ("d7452215dbd36cec", dict(shape=(41, 33, 18), n_atoms=50), dict(cutoff=2.0), "outside"),
    "far": ("c449754cdfb6f21c", dict(shape=(25, 40, 19), n_atoms=30), dict(cutoff=4.0), "far"),
}


@pytest.mark.parametrize("name", list(CASES))
def test_potential_bits(name):
    digest, sizes, kw, move = CASES[name]
    w = make_workload("tiny", **sizes)
    atoms = w.atoms
    box = np.array(w.meta["box"])
    if move == "grid":
        atoms = np.round(atoms / 0.25) * 0.25
    elif move == "outside":
        atoms = atoms + np.floor(7 * stream(3, atoms.size).reshape(atoms.shape) - 3) * box
    elif move == "far":
        atoms = atoms + 1000.0
    assert _digest(w, atoms=np.ascontiguousarray(atoms), **kw) == digest
