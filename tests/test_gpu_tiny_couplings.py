"""Couplings whose square is below the FP64 range still rotate.

A pair of indices with diagonal 1e-170, 2e-170 and coupling 1e-165, beside an
ordinary pair that keeps off(A) above the stopping tolerance: the small pair
passes the skip test |a_pq| > 2^-53 sqrt|a_pp a_qq|, and one rotation gives its
eigenvalues 1.5e-170 +- 1e-165 sqrt(1 + 2.5e-11).  A rotation is some ten
roundings, so they have to agree to 2^-48.  The pairs of five indices lie first,
in the middle and in between in their wavefronts.
"""
import itertools

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def m():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_00495_gb300 import build, mpj
    build.build()
    return mpj


@pytest.mark.parametrize("p,q", list(itertools.combinations(range(5), 2)))
@pytest.mark.parametrize("ordering", ["cyclic", "round_robin", "block"])
def test_small_pair_rotates(m, ordering, p, q):
    i, j, k = (x for x in range(5) if x not in (p, q))
    A = np.zeros((5, 5))
    A[i, i], A[j, j], A[k, k], A[i, j], A[j, i] = 1.0, 2.0, 3.0, 0.1, 0.1
    A[p, p], A[q, q], A[p, q], A[q, p] = 1e-170, 2e-170, 1e-165, 1e-165
    a, v, _, _, st = m.jacobi64(torch.from_numpy(A).cuda(), ordering=ordering)
    a, v = a.cpu().numpy(), v.cpu().numpy()
    assert st == 0
    h = 1e-165 * np.sqrt(1 + 2.5e-11)
    got = np.sort([a[p, p], a[q, q]])
    assert np.abs(got - [1.5e-170 - h, 1.5e-170 + h]).max() <= 2.0 ** -48 * h
    assert np.abs(np.abs(v[[p, p, q, q], [p, q, p, q]]) - np.sqrt(0.5)).max() <= 1e-5
