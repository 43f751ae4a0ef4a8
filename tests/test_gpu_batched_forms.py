"""Batches of small matrices are solved by one thread group each, in one launch,
where that is the faster form; the others go round by round.

Lists on both sides of the rule, ragged ones among them, against LAPACK with the
bounds of the other batched tests (eigenvalues within 1e-12 ||A||, residual and
orthogonality within 4 n u); the form shows in the number of launches.
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


def goe(n, rng):
    g = rng.standard_normal((n, n)) / np.sqrt(n)
    return (g + g.T) / 2


def check(mats, Ws, Qs):
    for a, W, Q in zip(mats, Ws, Qs):
        n = a.shape[0]
        W, Q = W.cpu().numpy(), Q.cpu().numpy()
        assert np.abs(W - np.linalg.eigvalsh(a)).max() <= 1e-12 * np.linalg.norm(a, 2), n
        assert np.linalg.norm(a @ Q - Q * W) <= 4 * n * U * np.linalg.norm(a), n
        assert np.linalg.norm(Q.T @ Q - np.eye(n)) <= 4 * n * U, n


@pytest.mark.parametrize("sizes,groups", [
    ([8], True), ([1, 2, 3, 20], True), ([8] * 608, True), ([24] * 153, True), ([40] * 700, True),
    ([5, 17, 32, 33, 40] * 100, True), ([48], False), ([48] * 40, False), ([64] * 20, False), ([8] * 600 + [65], False)])
def test_forms(m, sizes, groups):
    rng = np.random.default_rng(len(sizes) + sizes[-1])
    base = {n: [goe(n, rng) for _ in range(3)] for n in set(sizes)}
    dev = {n: [torch.from_numpy(a).cuda() for a in v] for n, v in base.items()}
    solver = m.BatchedSolver(sizes)
    for trial in range(2):  # the second call on the kept plan, with other data
        pick = [(i + trial) % 3 for i in range(len(sizes))]
        before = m.lib().mpj_kernel_launches()
        Ws, Qs, sweeps, st = solver.solve([dev[n][k] for n, k in zip(sizes, pick)])
        launches = m.lib().mpj_kernel_launches() - before
        assert st == 0 and (launches == 1) == groups, launches
        assert all(s < 10 for s in sweeps) and all((s > 0) == (n > 1) for s, n in zip(sweeps, sizes))
        check([base[n][k] for n, k in zip(sizes, pick)], Ws, Qs)


def test_groups_report_a_nonfinite_neighbour_and_take_a_tolerance(m):
    rng = np.random.default_rng(3)
    sizes = [20, 7, 24]
    mats = [goe(n, rng) for n in sizes]
    solver = m.BatchedSolver(sizes)
    bad = [a.copy() for a in mats]
    bad[1][2, 5] = bad[1][5, 2] = np.inf
    with pytest.raises(m.MPJError) as e:
        solver.solve([torch.from_numpy(a).cuda() for a in bad])
    assert e.value.status == m.MPJ_ENONFINITE
    check([mats[0], mats[2]], [solver.W[0], solver.W[2]], [solver.Qt[0].T, solver.Qt[2].T])
    Ws, _, sweeps, st = solver.solve([torch.from_numpy(a).cuda() for a in mats], tol=1.0)
    assert st == 0 and sweeps == [0, 0, 0]
    for a, W in zip(mats, Ws):  # stage 1 alone: off(A_cond) <= 1 bounds nothing, its own tolerance does
        assert np.abs(W.cpu().numpy() - np.linalg.eigvalsh(a)).max() <= a.shape[0] * 2.0 ** -23 * np.linalg.norm(a)
