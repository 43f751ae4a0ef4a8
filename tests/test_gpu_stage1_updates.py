"""Stage 1 where the form of its updates changes: both matrices' tiles in one
launch (n <= 1024 on 152 SMs, also with a last row group of fewer than four
block pairs), one launch per matrix from 2945 on, separate kernels in between.

Bounds as for the small sizes: off(A) within the stage's tolerance
n u_l ||A||_F; Q_l orthogonal and A Q_l - Q_l D small to 8 n u_l (2-norms, from
the eigenvalues of the symmetric E = Q^T Q - I and of R^T R).
"""
import pytest

from paper_2509_00495_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

UL = 2.0 ** -24


@pytest.fixture(scope="module")
def m():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_00495_gb300 import build, mpj
    build.build()
    return mpj


@pytest.mark.parametrize("n", [129, 250, 1000, 1024, 1025, 2944, 2945, 2990])
def test_stage1_update_forms(m, n):
    A = torch.from_numpy(inputs.randn_sym(n, seed=7 * n)).cuda()
    Q, _, off = m.stage1(A)
    assert off <= n * UL * torch.linalg.matrix_norm(A).item()
    nA = torch.linalg.eigvalsh(A).abs().max().item()
    E = Q.T @ Q - torch.eye(n, dtype=A.dtype, device="cuda")
    assert torch.linalg.eigvalsh(E).abs().max().item() <= 8 * n * UL
    R = A @ Q - Q * torch.diag(Q.T @ A @ Q)
    assert torch.linalg.eigvalsh(R.T @ R).max().clamp(min=0).sqrt().item() <= 8 * n * UL * nA
