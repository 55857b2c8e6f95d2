"""The stored integral tensor is a function of the basis alone: every element is
the same to the last bit on every call, whatever the launches' order (long
contractions, warp-cooperative classes, f shells), and equal to the oracle's
within 1e-12.
"""
import numpy as np
import pytest

import oracle
from synth import random_shells_molecule
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


def _contracted(spec, seed):
    """Shells (atom, l, primitives) on three atoms: up to 256 primitive pairs a shell pair."""
    rng = np.random.default_rng(seed)
    xyz = np.array([[0.0, 0.0, 0.0], [1.7, 0.3, -0.4], [-0.6, 2.1, 0.9]])
    shells = [(a, l, np.exp(rng.uniform(np.log(0.08), np.log(30.0), k)), rng.uniform(0.2, 1.0, k)) for a, l, k in spec]
    return _pack([6, 1, 8], xyz, shells, "contracted", -1)


CASES = {
    "s16": _contracted([(0, 0, 16), (1, 0, 16), (2, 0, 3)], 1),
    "sp": _contracted([(0, 0, 11), (0, 1, 6), (1, 0, 5), (2, 1, 7)], 2),
    "spd": _contracted([(0, 0, 9), (0, 2, 6), (1, 1, 6), (2, 2, 5), (2, 0, 1)], 3),
    "fg": random_shells_molecule((4, 3, 1, 0), 61, nprim=(2, 4), exp_range=(0.2, 5.0), box=3.0),
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_tensor_repeats_to_the_last_bit(hf, ctx, case):
    import torch
    mol = CASES[case]
    b = hf.Basis(ctx, mol)
    G = b.eri_tensor()
    for _ in range(5):
        assert torch.equal(b.eri_tensor(), G)
    assert torch.equal(hf.Basis(ctx, mol).eri_tensor(), G)  # another handle, the same molecule
    for p in ((1, 0, 2, 3), (0, 1, 3, 2), (2, 3, 0, 1)):
        assert torch.equal(G.permute(*p), G)
    G0 = oracle.Basis(mol).eri_tensor()
    assert np.max(np.abs(G.cpu().numpy() - G0)) <= 1e-12 * max(1.0, np.max(np.abs(G0)))


def test_tensor_of_a_class_too_large_for_slots(hf, ctx):
    """34 p shells of 5 primitives: the (pp|pp) quartets' unit slots would pass 256 MB, so the class takes whole kets.
    J and K from the tensor against the direct build, which has lists of its own."""
    import torch
    rng = np.random.default_rng(8)
    n = 34
    xyz = np.array([[i % 4, i // 4 % 3, i // 12] for i in range(n)]) * 1.3 + rng.uniform(-0.1, 0.1, (n, 3))
    shells = [(a, 1, np.exp(rng.uniform(np.log(0.3), np.log(3.0), 5)), rng.uniform(0.2, 1.0, 5)) for a in range(n)]
    b = hf.Basis(ctx, _pack([1] * n, xyz, shells, "p34", -1))
    G = b.eri_tensor()
    assert torch.equal(b.eri_tensor(), G)
    C = rng.normal(size=(b.nbf, 10)) / np.sqrt(b.nbf)
    D = torch.tensor(C @ C.T, device="cuda:0")
    J, K = b.jk_stored(G, D)
    J0, K0 = b.fock_jk(D, opts=hf.jk_opts(0.0))
    assert float((J - J0).abs().max()) <= 1e-10 and float((K - K0).abs().max()) <= 1e-10
