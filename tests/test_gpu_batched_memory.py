"""The memory of the round-by-round batched solve.

A batch whose workspace cannot be had in one piece is solved in smaller chunks
(the arithmetic of a matrix does not depend on its chunk: the same bits), and
what stays between calls is one workspace, whatever lists of sizes came before.
The workspace of a 256 x 256 matrix is 3 x 512 KB of FP64 matrices and two
sliced operands of 1 MB: 3.5 MB, with some KB of subproblem data 3.7 MB at most.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module")
def m():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_00495_gb300 import build, mpj
    build.build()
    yield mpj
    mpj.lib().mpj_release_plans()


def goe(n, seed):
    g = np.random.default_rng(seed).standard_normal((n, n)) / np.sqrt(n)
    return torch.from_numpy((g + g.T) / 2).cuda()


def test_short_of_memory(m):
    base = {n: [goe(n, 10 * n + i) for i in range(3)] for n in (256, 200, 40)}
    sizes = [256] * 500 + [40] * 7 + [200] * 100 + [256] * 3
    mats = [base[n][i % 3] for i, n in enumerate(sizes)]
    m.syev_batched(mats[:2] + mats[500:502])  # load the kernels
    solver = m.BatchedSolver(sizes)
    m.lib().mpj_release_plans()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - 1500 * MB, dtype=torch.uint8, device="cuda")
    try:
        W, Q, sweeps, st = solver.solve(mats)
    finally:
        del fill
        torch.cuda.empty_cache()
    assert st == 0
    W, Q = [w.clone() for w in W], [q.clone() for q in Q]
    m.lib().mpj_release_plans()
    W2, Q2, sweeps2, st2 = solver.solve(mats)
    assert st2 == 0 and sweeps == sweeps2
    assert all(torch.equal(a, b) for a, b in zip(W, W2)) and all(torch.equal(a, b) for a, b in zip(Q, Q2))
    for i in (0, 499, 503, 550, 609):
        n, A = sizes[i], mats[i].cpu().numpy()
        assert np.abs(W[i].cpu().numpy() - np.linalg.eigvalsh(A)).max() <= 1e-12 * np.linalg.norm(A, 2), n


def test_changing_lists_keep_one_workspace(m):
    A = goe(256, 1)
    lists = [[A] * k for k in (300, 301, 302, 303, 304)]
    m.syev_batched(lists[0][:1])
    m.lib().mpj_release_plans()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    for x in lists[::-1]:
        m.syev_batched(x)
    grown = m.lib().mpj_device_allocations()
    for x in lists:
        assert m.syev_batched(x)[3] == 0
    assert m.lib().mpj_device_allocations() == grown
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    assert before - torch.cuda.mem_get_info()[0] <= 304 * 3.7 * MB + 64 * MB
    m.lib().mpj_release_plans()
    assert before - torch.cuda.mem_get_info()[0] <= 64 * MB
