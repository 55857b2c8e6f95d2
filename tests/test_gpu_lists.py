"""The work lists keep exactly the quartets that the Schwarz rule keeps: counts
against a direct count over the shell pairs, for molecules with many equal
Schwarz factors (a ring, whose bras tie), with ragged contractions (ket units of
many sizes) and with pairs that hold no significant primitives (a long chain).
J and K of the same lists agree with the oracle at the same threshold.
"""
import numpy as np
import pytest

import oracle
from synth import h_line, lattice_molecule
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
    a = 2 * np.pi * np.arange(n) / n
    r = 0.8 / np.sin(np.pi / n)
    xyz = np.stack([r * np.cos(a), r * np.sin(a), np.zeros(n)], axis=1)
    shells = [(k, l, [0.4, 1.9], [0.6, 0.5]) for k in range(n) for l in (0, 1)]
    return _pack([1] * n, xyz, shells, "ring", -1)


MOLS = {"ring": lambda: _ring(8), "chain": lambda: h_line(40, seed=4, spacing=2.2), "ragged": lambda: lattice_molecule(4, 53, "spd")}


@pytest.mark.parametrize("name", sorted(MOLS))
@pytest.mark.parametrize("tau", [0.0, 1e-12, 1e-5])
@pytest.mark.parametrize("bound", [0.0, 1e-7, 1e-3])
def test_lists_keep_what_the_schwarz_rule_keeps(hf, ctx, name, tau, bound):
    import torch
    mol = MOLS[name]()
    b = hf.Basis(ctx, mol)
    Q = b.schwarz()
    q = Q[np.tril_indices(mol.nshell)]
    prod = np.outer(q, q)[np.tril_indices(len(q))]
    kept = prod >= tau
    total, low = b.count_quartets(hf.jk_opts(tau, fp32_bound=bound))
    assert total == int(kept.sum())
    assert low == int((kept & (prod < bound)).sum())
    if bound == 0.0:
        ob = oracle.Basis(mol)
        C = np.random.default_rng(2).normal(size=(ob.nbf, 3)) / np.sqrt(ob.nbf)
        J0, K0, _ = ob.jk(C @ C.T, tau=tau, nthreads=oracle.oracle_threads())
        J, K = b.fock_jk(torch.tensor(C @ C.T, device="cuda:0"), opts=hf.jk_opts(tau))
        # a quartet whose product is within rounding of tau may be on either side: it weighs below 4 tau max|D|
        slack = 1e-10 + (4 * tau * np.max(np.abs(C @ C.T)) if tau > 1e-10 else 0.0)
        assert np.max(np.abs(J.cpu().numpy() - J0)) <= slack
        assert np.max(np.abs(K.cpu().numpy() - K0)) <= slack
