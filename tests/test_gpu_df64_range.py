"""The df64 tier over the exponents a basis may have: steep d and p shells (as
in all-electron bases of heavy elements), diffuse ones, and contractions that
hold both.  Floats carry 8 exponent bits, and the Hermite form of the L >= 5
classes goes through powers of the reduced exponent up to the eighth.

Scaling every exponent by 4^k and every length by 2^-k scales the integrals by
2^k exactly, so one molecule serves at all scales.  Tolerance: the tier's 1e-10
on J and K of order one, here relative to their largest element.
"""
import numpy as np
import pytest

import oracle
from synth.molecules import _pack

pytestmark = pytest.mark.gpu

XYZ = np.array([[0.0, 0.0, 0.0], [1.3, 0.2, -0.4], [-0.5, 1.6, 0.7]])
SHELLS = [(0, 2, [3.1], [1.0]), (0, 1, [30.0, 2.0], [0.4, 0.8]), (1, 2, [9.0, 0.7], [0.5, 0.7]), (1, 0, [1.1], [1.0]), (2, 2, [0.3], [1.0]),
          (2, 1, [0.9], [1.0])]
# steep and diffuse primitives side by side, on one centre and across centres
MIXED = [(0, 2, [8.0e4, 90.0, 0.2], [0.6, 0.5, 0.4]), (0, 2, [2500.0], [1.0]), (0, 1, [4.0e5, 0.5], [0.5, 0.6]), (1, 2, [1.0e4], [1.0]),
         (1, 1, [0.02], [1.0]), (2, 2, [0.006], [1.0]), (2, 0, [0.4], [1.0])]


def _scaled(k):
    return _pack([6, 1, 8], XYZ * 2.0 ** -k, [(a, l, np.array(e) * 4.0 ** k, c) for a, l, e, c in SHELLS], "scaled", -1)


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


CASES = {f"4^{k}": _scaled(k) for k in (-7, -5, -3, -2, 0, 2, 3, 4, 5, 7, 9)}
CASES["mixed"] = _pack([6, 1, 8], XYZ, MIXED, "mixed", -1)


@pytest.mark.parametrize("case", sorted(CASES))
def test_df64_over_the_range_of_exponents(hf, ctx, case):
    import torch
    mol = CASES[case]
    ob, b = oracle.Basis(mol), hf.Basis(ctx, mol)
    rng = np.random.default_rng(11)
    C = rng.normal(size=(ob.nbf, 4)) / np.sqrt(ob.nbf)
    D = C @ C.T
    J0, K0, _ = ob.jk(D, tau=0.0, nthreads=oracle.oracle_threads())
    for kw in ({}, {"df64": True}):
        J, K = b.fock_jk(torch.tensor(D, device="cuda:0"), opts=hf.jk_opts(0.0, **kw))
        for got, want in ((J.cpu().numpy(), J0), (K.cpu().numpy(), K0)):
            assert np.max(np.abs(got - want)) <= 1e-10 * np.max(np.abs(want)), kw
