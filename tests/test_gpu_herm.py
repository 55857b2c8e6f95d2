"""The Hermite-bra kernels of the s/p/d classes (csrc/herm.cuh) and their ket
units against the CPU oracle.

(ss|ss) integrals of single-primitive shells over the whole range of T pin the
tabulated S_m: near rows (y = 2T below 120, grid 1/32), the change to the far
rows, and far rows scaled by several powers of four.  Tolerance: the value is
a product of about 30 correctly rounded FP64 factors and sums, so 32 roundings
of 2^-53 relative.

Contractions of 1 to 16 primitives give shell pairs of 1 to 256 primitive
pairs, i.e. kets cut into up to 22 units of unequal size and bra parts of one
primitive pair; J and K must meet the package's 1e-10 in every tier that meets
it, screened and not, and the FP32 split its own bound at a split that sends
nothing to FP32.
"""
import numpy as np
import pytest

import oracle
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


# (alpha, distances): T = alpha R^2 from 0 through the grid steps, the change of
# range at T = 60 and up to 4e6 (k = 8)
T_CASES = {
    "near": (1.0, np.sqrt(np.concatenate([np.linspace(0.0, 1.0, 20), np.arange(1, 20) * 3.0 + 1 / 128]))),
    "change": (1.0, np.sqrt(np.concatenate([60 + np.linspace(-0.5, 0.5, 21), [59.9999999, 60.0, 60.0000001, 63.99, 64.0, 64.01]]))),
    "far": (1.0, np.sqrt(np.geomspace(50.0, 4.0e6, 40))),
    "tiny": (1.0, np.concatenate([[0.0], np.geomspace(1e-9, 1e-2, 30)])),
}


@pytest.mark.parametrize("case", sorted(T_CASES))
def test_ssss_over_the_range_of_T(hf, ctx, case):
    alpha, dist = T_CASES[case]
    n = len(dist) + 1
    xyz = np.zeros((n, 3))
    xyz[1:, 0] = dist  # centre 0 against every other: T = alpha R^2
    mol = _pack([0] * n, xyz, [(a, 0, [alpha], [1.0]) for a in range(n)], "line", -1, n_electrons=2)
    b = hf.Basis(ctx, mol)
    Q = b.eri_tensor().cpu().numpy()
    got = np.array([Q[0, 0, i, i] for i in range(1, n)])
    T = alpha * dist ** 2
    # (aa|bb) of unit-norm Gaussians: 2 pi^(5/2) / (p q sqrt(p + q)) N^4 F_0, p = q = 2 alpha, T = alpha R^2
    want = np.array([2 * np.pi ** 2.5 / (4 * alpha ** 2 * np.sqrt(4 * alpha)) * (2 * alpha / np.pi) ** 3 * oracle.boys(0, t)
                     for t in T])
    assert np.max(np.abs(got / want - 1)) <= 32 * 2.0 ** -53


RAGGED = [(0, 0, 16), (0, 1, 1), (1, 0, 5), (1, 2, 2), (2, 1, 7)]
RAGGED_SMALL = [(0, 0, 13), (1, 1, 2), (2, 2, 1)]


def _ragged(spec):
    rng = np.random.default_rng(3)
    xyz = np.array([[0.0, 0.0, 0.0], [1.7, 0.3, -0.4], [-0.6, 2.1, 0.9]])
    shells = [(a, l, np.exp(rng.uniform(np.log(0.05), np.log(60.0), k)), rng.uniform(0.2, 1.0, k)) for a, l, k in spec]
    return _pack([6, 1, 8], xyz, shells, "ragged", -1)


@pytest.mark.parametrize("tau", [0.0, 1e-12])
@pytest.mark.parametrize("kw", [{}, {"df64": True}, {"fp32_bound": 1e-30}, {"deterministic": True}],
                         ids=["fp64", "df64", "split-empty", "deterministic"])
def test_ragged_contractions(hf, ctx, tau, kw):
    import torch
    mol = _ragged(RAGGED)
    ob, b = oracle.Basis(mol), hf.Basis(ctx, mol)
    rng = np.random.default_rng(5)
    C = rng.normal(size=(ob.nbf, 4)) / np.sqrt(ob.nbf)
    D = C @ C.T
    J0, K0, _ = ob.jk(D, tau=tau, nthreads=oracle.oracle_threads())
    J, K = b.fock_jk(torch.tensor(D, device="cuda:0"), opts=hf.jk_opts(tau, **kw))
    assert np.max(np.abs(J.cpu().numpy() - J0)) <= 1e-10
    assert np.max(np.abs(K.cpu().numpy() - K0)) <= 1e-10


def test_ragged_counts_and_tensor(hf, ctx):
    """Every unique quartet counted once although its ket is cut into units; the tensor whole."""
    mol = _ragged(RAGGED_SMALL)
    b = hf.Basis(ctx, mol)
    npair = mol.nshell * (mol.nshell + 1) // 2
    assert b.count_quartets(hf.jk_opts(0.0))[0] == npair * (npair + 1) // 2
    G = b.eri_tensor().cpu().numpy()
    assert np.max(np.abs(G - oracle.Basis(mol).eri_tensor())) <= 1e-12
