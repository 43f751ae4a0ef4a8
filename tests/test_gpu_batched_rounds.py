"""The round-by-round batched solve at the edges of its size classes.

Matrices of every class boundary (n = 32 k, 32 k +- 1), equal and mixed sizes,
a single matrix, converged-at-once inputs next to hard ones, and new pointers on
a kept plan.  Bounds as for the other batched tests: eigenvalues within
1e-12 ||A|| of LAPACK, residual and orthogonality within 4 n u.
"""
import numpy as np
import pytest

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


def check(mats, Ws, Qs):
    for a, W, Q in zip(mats, Ws, Qs):
        n = a.shape[0]
        W, Q = W.cpu().numpy(), Q.cpu().numpy()
        nA = max(np.linalg.norm(a, 2), 1e-300)
        assert np.abs(W - np.linalg.eigvalsh(a)).max() <= 1e-12 * nA, n
        assert np.linalg.norm(a @ Q - Q * W) <= 4 * n * U * max(np.linalg.norm(a), 1e-300), n
        assert np.linalg.norm(Q.T @ Q - np.eye(n)) <= 4 * n * U, n


def goe(n, rng):
    g = rng.standard_normal((n, n)) / np.sqrt(n)
    return (g + g.T) / 2


@pytest.mark.parametrize("sizes", [[1], [256], [33] * 7, [1, 2, 31, 32, 33, 63, 64, 65, 95, 96, 97, 127, 128, 129],
                                   [159, 160, 161, 191, 192, 193, 223, 224, 225, 255, 256], [8, 256, 9, 255, 10, 254]])
def test_class_boundaries(m, sizes):
    rng = np.random.default_rng(sum(sizes))
    mats = [goe(n, rng) for n in sizes]
    Ws, Qs, sweeps, st = m.syev_batched([torch.from_numpy(a).cuda() for a in mats])
    assert st == 0 and all(0 <= s < 10 for s in sweeps)
    check(mats, Ws, Qs)


def test_converged_matrices_drop_out(m):
    rng = np.random.default_rng(5)
    mats = [np.diag(np.linspace(-1, 1, 70)), goe(70, rng), np.zeros((40, 40)), np.eye(40) * 3.0, goe(40, rng),
            np.diag([2.0]), 1e-200 * goe(50, rng)]
    Ws, Qs, sweeps, st = m.syev_batched([torch.from_numpy(a).cuda() for a in mats])
    assert st == 0
    assert sweeps[0] == sweeps[2] == sweeps[3] == sweeps[5] == 0 and sweeps[1] > 0
    check(mats[:6], Ws[:6], Qs[:6])


def test_new_buffers_on_a_kept_plan_and_a_nonfinite_neighbour(m):
    rng = np.random.default_rng(9)
    sizes = [100, 17, 64]
    keep = []
    for _ in range(3):  # other pointers each time
        mats = [goe(n, rng) for n in sizes]
        dm = [torch.from_numpy(a).cuda() for a in mats]
        keep.append(dm)
        Ws, Qs, _, st = m.syev_batched(dm)
        assert st == 0
        check(mats, Ws, Qs)
    solver = m.BatchedSolver(sizes)
    bad = [a.copy() for a in mats]
    bad[1][3, 4] = bad[1][4, 3] = np.nan
    with pytest.raises(m.MPJError) as e:
        solver.solve([torch.from_numpy(a).cuda() for a in bad])
    assert e.value.status == m.MPJ_ENONFINITE
    check([mats[0], mats[2]], [solver.W[0], solver.W[2]], [solver.Qt[0].T, solver.Qt[2].T])


@pytest.mark.parametrize("e", [-400, -126, -75, -30, 30, 60, 126, 400])
def test_scales(m, e):
    """2^e A rotates as A does, also where FP32 (or its squares) cannot hold 2^e: the
    same sweeps and the same vectors, the eigenvalues times 2^e."""
    rng = np.random.default_rng(11)
    mats = [goe(n, rng) for n in (40, 70, 130, 250)]
    W, Q, sweeps, st = m.syev_batched([torch.from_numpy(a).cuda() for a in mats])
    W2, Q2, sweeps2, st2 = m.syev_batched([torch.from_numpy(a * 2.0 ** e).cuda() for a in mats])
    assert st == 0 and st2 == 0 and sweeps == sweeps2
    assert all(torch.equal(a, b) for a, b in zip(Q, Q2))
    assert all(torch.equal(a * 2.0 ** e, b) for a, b in zip(W, W2))
