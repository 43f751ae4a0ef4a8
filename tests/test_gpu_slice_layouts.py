"""Operands of the tensor-core product whose k runs along memory: the 16-byte
loads and the 8-row x 32-k warps of the slicing at the edges of their ranges
(k and rows off every multiple, odd leading dimensions, a base that is only
8-byte aligned).

Bound per entry, u = 2^-53: the slicing rounds every factor to 2^-57 and drops
levels below 2^-54 of max|a_r| max|b_c| per term (2 k u max max in all), numpy's
product errs by at most k u (|A| |B|).
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


def _buffer(X, pad, off):
    """X column-major with leading dimension rows + pad, `off` doubles into an allocation."""
    r, c = X.shape
    ld = r + pad
    buf = torch.full((off + ld * c,), float("nan"), dtype=torch.float64)
    buf[off:].view(c, ld)[:, :r] = torch.from_numpy(np.ascontiguousarray(X.T))
    buf = buf.cuda()
    return buf, buf.data_ptr() + 8 * off, ld


@pytest.mark.parametrize("mm, nn, k", [(1, 1, 1), (65, 130, 7), (128, 64, 33), (3, 5, 40), (200, 70, 257)])
@pytest.mark.parametrize("pad, off", [(0, 0), (1, 0), (0, 1), (3, 1)])
@pytest.mark.parametrize("ta, tb", [("T", "N"), ("T", "T"), ("N", "N")])
def test_products_of_any_layout(m, mm, nn, k, pad, off, ta, tb):
    rng = np.random.default_rng(1000 * mm + 10 * k + pad + off)
    A, B = rng.standard_normal((mm, k)), rng.standard_normal((k, nn))
    a, pa, lda = _buffer(A.T if ta == "T" else A, pad, off)
    b, pb, ldb = _buffer(B.T if tb == "T" else B, pad, off)
    C = torch.zeros(nn, mm, dtype=torch.float64, device="cuda")
    st = m.lib().mpj_dgemm_tc(ta.encode(), tb.encode(), mm, nn, k, 1.0, pa, lda, pb, ldb, 0.0, C.data_ptr(), mm,
                              m._stream())
    assert st == 0
    bound = U * (k * (np.abs(A) @ np.abs(B)) +
                 2 * k * np.abs(A).max(1)[:, None] * np.abs(B).max(0)[None, :])
    assert (np.abs(C.T.cpu().numpy() - A @ B) <= bound).all()
