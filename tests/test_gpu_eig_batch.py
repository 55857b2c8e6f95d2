"""The block-per-matrix eigensolver (csrc/eig.cu) where several matrices share a
launch: the sizes only a batch sends to it (65 to 88 functions), mixed sizes
(the largest sets the shared memory), members above the limit beside members
below it, more matrices than one launch takes; and matrices that hold no
finite decomposition.

A batch member's first energy comes from the same core-Hamiltonian orbitals as
its own solve, whatever else is in the batch: within the 1e-8 Eh of the batched
solver's contract.
"""
import numpy as np
import pytest

from synth import h_line

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1303_4916_gb300 as hf
    return hf


@pytest.fixture(scope="module")
def ctx(hf):
    return hf.Context(0)


BATCHES = {
    "largest": [65, 88],
    "mixed": [1, 2, 63, 64, 65, 87, 88, 89],
    "alone": [88, 100],
    "many": [2 + k % 7 for k in range(40)],
}



@pytest.mark.parametrize("name", sorted(BATCHES))
def test_batch_members_match_their_own_solve(hf, ctx, name):
    mols = []
    for n in BATCHES[name]:
        m = h_line(n, seed=n)
        m.n_electrons = max(2, n // 2 * 2)  # closed shells
        mols.append(m)
    res, st = hf.scf_solve_batch([hf.Basis(ctx, m) for m in mols], max_iter=2, e_tol=0.0)
    for m, r, s in zip(mols, res, st):
        own = hf.Basis(ctx, m).scf(max_iter=2, e_tol=0.0)
        assert np.isfinite(own.energy) and abs(r.energy - own.energy) <= 1e-8, (m.nshell, s)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("n", [2, 5, 33])
def test_no_finite_energy_from_a_fock_matrix_that_is_not_finite(hf, ctx, n, bad):
    """A starting density with a NaN or an infinity makes F such a matrix: the solve must not report numbers."""
    import torch
    m = h_line(n, seed=n)
    m.n_electrons = 2  # one occupied orbital
    b = hf.Basis(ctx, m)
    D0 = torch.full((b.nbf, b.nbf), 0.1, dtype=torch.float64, device="cuda:0")
    D0[0, 0] = bad
    r = b.scf(max_iter=3, D0=D0)
    assert not r.converged and not np.isfinite(r.energy)
    assert not torch.isfinite(r.tensors["eps"]).any()
