"""The adjoint's grouped launches at the edges of their tiles and groups.

n around the 32-wide tiles and the 64 x 128 product tiles, batches that split
into several groups of matrices, leading dimensions larger than n, and missing
upstream gradients, against the oracle's adjoint to 1e-10 of its largest entry
(the bound of the other adjoint tests); the result is exactly symmetric.
"""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2509_00495_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def m():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_00495_gb300 import build, mpj
    build.build()
    return mpj


def problem(n, seed):
    rng = np.random.default_rng(seed)
    w = inputs.gapped_spectrum(n, rng, gap=min(1e-3, 1.0 / n))
    return w, inputs.haar_orthogonal(n, rng), rng.standard_normal(n), rng.standard_normal((n, n))


def check(got, ref):
    assert np.array_equal(got, got.T)
    assert np.abs(got - ref).max() <= 1e-10 * max(np.abs(ref).max(), 1e-300)


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 65, 127, 129, 200])
def test_sizes(m, n):
    ps = [problem(n, 10 * n + i) for i in range(3)]
    W, Q, dW, dQ = (torch.from_numpy(np.stack([p[k] for p in ps])).cuda() for k in range(4))
    dA = m.syev_backward(W, Q, dW, dQ).cpu().numpy()
    for i, (w, q, dw, dq) in enumerate(ps):
        check(dA[i], oracle.eigh_backward(w, q, dw, dq))
    check(m.syev_backward(W, Q, None, dQ).cpu().numpy()[1], oracle.eigh_backward(*ps[1][:2], np.zeros(n), ps[1][3]))
    check(m.syev_backward(W, Q, dW, None).cpu().numpy()[2], oracle.eigh_backward(*ps[2][:3], np.zeros((n, n))))


@pytest.mark.parametrize("n,batch", [(520, 50), (300, 70)])
def test_several_groups(m, n, batch):
    """The sliced operands of these batches exceed half a GB: two groups or more."""
    ps = [problem(n, i) for i in range(4)]
    W, Q, dW, dQ = (torch.from_numpy(np.stack([ps[b % 4][k] for b in range(batch)])).cuda() for k in range(4))
    dA = m.syev_backward(W, Q, dW, dQ)
    for b in range(batch):
        assert torch.equal(dA[b], dA[b % 4]), b
    for i in range(2):
        check(dA[i].cpu().numpy(), oracle.eigh_backward(*ps[i]))


def test_leading_dimensions(m):
    n, ld, batch = 70, 83, 2
    ps = [problem(n, 40 + i) for i in range(batch)]
    Q = torch.full((batch, n, ld), float("nan"), dtype=torch.float64, device="cuda")
    dQ, dA = Q.clone(), Q.clone()
    for b, p in enumerate(ps):  # column-major: row j of the buffer is column j
        Q[b, :, :n] = torch.from_numpy(np.ascontiguousarray(p[1].T))
        dQ[b, :, :n] = torch.from_numpy(np.ascontiguousarray(p[3].T))
    W = torch.from_numpy(np.stack([p[0] for p in ps])).cuda()
    dW = torch.from_numpy(np.stack([p[2] for p in ps])).cuda()
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    st = m.lib().mpj_syev_backward(batch, n, ptr(W), ptr(Q), ld, ptr(dW), ptr(dQ), ld, ptr(dA), ld,
                                   ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0
    got = dA.cpu().numpy()
    assert np.isnan(got[:, :, n:]).all()
    for b, p in enumerate(ps):
        check(got[b, :, :n].T, oracle.eigh_backward(*p))


def test_groups_of_a_ragged_size(m):
    """n = 300: an operand is padded to 384 x 512, 3.1 MB, so 85 matrices fit in half
    a GB and 91 split into two groups of unequal size."""
    n, batch = 300, 91
    ps = [problem(n, 70 + i) for i in range(4)]
    W, Q, dW, dQ = (torch.from_numpy(np.stack([ps[b % 4][k] for b in range(batch)])).cuda() for k in range(4))
    before = m.lib().mpj_kernel_launches()
    m.syev_backward(W[:4], Q[:4], dW[:4], dQ[:4])
    one = m.lib().mpj_kernel_launches() - before
    dA = m.syev_backward(W, Q, dW, dQ)
    assert m.lib().mpj_kernel_launches() - before == 3 * one  # one group, then two
    for b in range(batch):
        assert torch.equal(dA[b], dA[b % 4]), b
    for i in range(4):
        check(dA[i].cpu().numpy(), oracle.eigh_backward(*ps[i]))
