"""Edges of small dispatch rules: the premise estimate (one cluster up to
n = 384, one launch per step beyond), the cyclic wavefronts at the smallest
orders and around a row chunk of 128, and calls before and after the library's
memory is given back.

Premise: 30 steps of the power iteration give a lower bound of ||E||_2 that
falls short by a factor 1 - 0.871 ln(n) / 29 on average over start vectors
(0.81 at n = 513), so at least half of it.  Cyclic: the bounds of the other
comparisons with the oracle's cyclic sweeps.
"""
import numpy as np
import pytest

import oracle
from paper_2509_00495_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def m():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_00495_gb300 import build, mpj
    build.build()
    return mpj


@pytest.mark.parametrize("n", [33, 383, 384, 385, 513])
def test_premise_estimate(m, n):
    A = torch.from_numpy(inputs.randn_sym(n, seed=n)).cuda()
    Q = m.stage1(A)[0]
    norm = torch.linalg.eigvalsh(Q.T @ Q - torch.eye(n, dtype=Q.dtype, device="cuda")).abs().max().item()
    e0 = m.syev_ex(A).info["ns_e0"]
    assert 0.5 * norm <= e0 <= norm * (1 + 1e-6)


@pytest.mark.parametrize("n", [2, 3, 4, 127, 128, 129])
def test_cyclic_wavefront_edges(m, n):
    A = inputs.randn_sym(n, seed=3 * n)
    tol = n * U * np.linalg.norm(A)
    a_ref, _, sw_ref, _, _, _ = oracle.jacobi(A, ordering=oracle.CYCLIC, tol=tol)
    a, v, sw, off, st = m.jacobi64(torch.from_numpy(A).cuda(), tol=tol, ordering="cyclic")
    a, v = a.cpu().numpy(), v.cpu().numpy()
    assert st == 0 and off <= tol and sw == sw_ref
    nA = np.linalg.norm(A, 2)
    assert np.abs(np.diag(a) - np.diag(a_ref)).max() <= 1e-13 * nA
    assert np.linalg.norm(A @ v - v * np.diag(a), 2) <= 1e-12 * nA


def test_results_survive_giving_memory_back(m):
    A = torch.from_numpy(inputs.randn_sym(150, seed=1)).cuda()
    B = torch.randn(150, 70, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    first, p = m.syev_ex(A), m.dgemm_tc("T", "N", 1.0, A, B)
    for _ in range(2):
        torch.cuda.synchronize()
        m.lib().mpj_release_plans()
        again, q = m.syev_ex(A), m.dgemm_tc("T", "N", 1.0, A, B)
        assert torch.equal(first.Q, again.Q) and torch.equal(first.W, again.W) and torch.equal(p, q)
