"""The block-per-matrix eigensolver (csrc/eig.cu) at the sizes where it can go
wrong: one function, odd sizes (padded), the largest it takes alone and the
first that goes to the library, and exactly degenerate levels.

The first RHF iteration diagonalises the core Hamiltonian, so its orbitals must
satisfy H C = S C eps and C^T S C = 1, with eps ascending.  Rounding: X = S^{-1/2},
F' = X H X and C = X C' are five products of length n on top of the
eigendecomposition, each n 2^-53 of its operands' norms, amplified by at most
1 / lambda_min(S): 64 n 2^-53 ||H|| / lambda_min(S).
"""
import numpy as np
import pytest

from synth import h_line
from synth.molecules import _pack

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


def _ring(n):
    """n hydrogens on a regular polygon with the same shell: pairs of degenerate levels."""
    r = 1.6 / (2 * np.sin(np.pi / n))
    a = 2 * np.pi * np.arange(n) / n
    xyz = np.stack([r * np.cos(a), r * np.sin(a), np.zeros(n)], axis=1)
    return _pack([1] * n, xyz, [(k, 0, [0.4, 1.9], [0.6, 0.5]) for k in range(n)], "ring", -1)


CASES = [("line", n) for n in (1, 2, 3, 17, 63, 64, 65)] + [("ring", 6), ("ring", 48)]


@pytest.mark.parametrize("kind,n", CASES)
def test_first_iteration_diagonalises_the_core_hamiltonian(hf, ctx, kind, n):
    mol = h_line(n) if kind == "line" else _ring(n)
    b = hf.Basis(ctx, mol)
    assert b.nbf == n
    S, T, V, _ = b.one_electron()
    S, H = S.cpu().numpy(), (T + V).cpu().numpy()
    r = b.scf(max_iter=1)
    C, eps = r.tensors["C"].cpu().numpy(), r.tensors["eps"].cpu().numpy()
    lam = np.linalg.eigvalsh(S)[0]
    tol = 64 * n * 2.0 ** -53 * max(1.0, np.linalg.norm(H, 2)) / lam
    assert np.all(np.diff(eps) >= 0)
    assert np.max(np.abs(C.T @ S @ C - np.eye(n))) <= tol
    assert np.max(np.abs(H @ C - S @ C * eps)) <= tol
