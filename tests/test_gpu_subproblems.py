"""The 32 x 32 subproblem kernels of the block orderings at the edges of their
ranges, through the C ABI.

FP64 sweeps: a subproblem runs in FP32 pairs when its couplings span at most
2^70 (2^100 with the diagonal) and in FP64 instructions otherwise; graded
matrices D B D with D = diag(2^-span .. 1) reach both.  Bounds as for the other
block-sweep tests: eigenvalues against the oracle's block ordering within
1e-12 ||A||, residual within tol + 4 n u ||A||, orthogonality within 4 n u.
Stage 1: sizes around one and two blocks; Q_l orthogonal and A Q_l - Q_l D
small to 8 n u_l, sweeps within one of the oracle's.
"""
import numpy as np
import pytest

import oracle
from paper_2509_00495_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = 2.0 ** -53
UL = 2.0 ** -24


@pytest.fixture(scope="module")
def m():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_00495_gb300 import build, mpj
    build.build()
    return mpj


@pytest.mark.parametrize("n", [32, 45])
@pytest.mark.parametrize("span", [0, 20, 34, 40, 80, 300])
def test_block_sweeps_on_graded_matrices(m, n, span):
    rng = np.random.default_rng(1000 * n + span)
    d = 2.0 ** rng.permutation(-np.linspace(0, span, n).round())
    A = inputs.randn_sym(n, seed=n + span) * d[:, None] * d[None, :]
    tol = n * U * np.linalg.norm(A)
    nA = np.linalg.norm(A, 2)
    a_ref = oracle.jacobi(A, ordering=oracle.BLOCK_ROUND_ROBIN, tol=tol)[0]
    a, v, _, off, st = m.jacobi64(torch.from_numpy(A).cuda(), tol=tol, ordering="block")
    a, v = a.cpu().numpy(), v.cpu().numpy()
    assert st == 0 and off <= tol
    assert np.abs(np.sort(np.diag(a)) - np.sort(np.diag(a_ref))).max() <= 1e-12 * nA
    assert np.linalg.norm(A @ v - v * np.diag(a)) <= tol + 4 * n * U * nA
    assert np.linalg.norm(v.T @ v - np.eye(n)) <= 4 * n * U


@pytest.mark.parametrize("scale", [2.0 ** -900, 1.0, 2.0 ** 480])
def test_block_sweeps_do_not_depend_on_the_scale(m, scale):
    """A power of two times A rotates the same way: the same vectors."""
    n = 64
    A = inputs.randn_sym(n, seed=64)
    _, v1, sw1, _, _ = m.jacobi64(torch.from_numpy(A).cuda(), tol=n * U * np.linalg.norm(A), ordering="block")
    _, v2, sw2, _, _ = m.jacobi64(torch.from_numpy(A * scale).cuda(), tol=n * U * np.linalg.norm(A) * scale,
                                  ordering="block")
    if scale > 2.0 ** -500:  # below, off(A)^2 underflows and the sweeps stop at once, as they always did
        assert sw1 == sw2 and torch.equal(v1, v2)
    else:
        assert sw2 == 0


@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 31, 32, 33, 64, 65])
def test_stage1_around_the_block_sizes(m, n):
    A = inputs.randn_sym(n, seed=7 * n)
    Ql, sw, off = m.stage1(torch.from_numpy(A).cuda())
    Ql = Ql.cpu().numpy()
    _, _, info = oracle.stage1(A, ordering32=oracle.BLOCK_ROUND_ROBIN)
    nA = np.linalg.norm(A, 2)
    assert abs(sw - info.sweeps32) <= 1 and off <= n * UL * np.linalg.norm(A)
    assert np.linalg.norm(Ql.T @ Ql - np.eye(n), 2) <= 8 * n * UL
    D = np.diag(Ql.T @ A @ Ql)
    assert np.linalg.norm(A @ Ql - Ql * D, 2) <= 8 * n * UL * nA
