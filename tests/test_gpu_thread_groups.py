"""The batched solve with one thread group per matrix as MPJ_BATCHED_GROUP asks
for it: the group size is tuned on the first call, later calls on the same
buffers replay the captured launch with new data, and the choice is kept in (and
taken from) the file that MPJ_AUTOTUNE_CACHE names.  Bounds as for the other
batched tests: eigenvalues within 1e-12 ||A||, residual and orthogonality within
4 n u.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
U = 2.0 ** -53


@pytest.fixture(scope="module")
def m():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_00495_gb300 import build, mpj
    build.build()
    return mpj


def test_tuned_once_then_replayed(m, monkeypatch):
    monkeypatch.setenv("MPJ_BATCHED_GROUP", "auto")
    rng = np.random.default_rng(78)
    sizes = [int(n) for n in rng.integers(8, 257, size=23)]
    solver = m.BatchedSolver(sizes)
    for trial in range(3):
        mats = []
        for n in sizes:
            g = rng.standard_normal((n, n)) / np.sqrt(n)
            mats.append((g + g.T) / 2)
        before = m.lib().mpj_kernel_launches()
        Ws, Qs, sweeps, st = solver.solve([torch.from_numpy(a).cuda() for a in mats])
        launches = m.lib().mpj_kernel_launches() - before
        assert st == 0 and launches == (4 if trial == 0 else 1)  # three tuning runs, then the graph's kernel
        assert solver.group_size() in (256, 512, 1024)
        for a, W, Q in zip(mats, Ws, Qs):
            n, W, Q = a.shape[0], W.cpu().numpy(), Q.cpu().numpy()
            assert np.abs(W - np.linalg.eigvalsh(a)).max() <= 1e-12 * np.linalg.norm(a, 2)
            assert np.linalg.norm(a @ Q - Q * W) <= 4 * n * U * np.linalg.norm(a)
            assert np.linalg.norm(Q.T @ Q - np.eye(n)) <= 4 * n * U
    m.lib().mpj_release_plans()


SCRIPT = """
import sys
sys.path.insert(0, sys.argv[1])
import torch
from paper_2509_00495_gb300 import mpj
s = mpj.BatchedSolver([100, 40])
print(s.group_size())
before = mpj.lib().mpj_kernel_launches()
s.solve([torch.eye(100, dtype=torch.float64, device="cuda"), torch.eye(40, dtype=torch.float64, device="cuda")])
print(mpj.lib().mpj_kernel_launches() - before, s.group_size())
"""


def test_choices_are_kept_in_the_file(m, tmp_path):
    path = tmp_path / "groups.txt"

    def run():
        env = dict(os.environ, MPJ_BATCHED_GROUP="auto", MPJ_AUTOTUNE_CACHE=str(path))
        r = subprocess.run([sys.executable, "-c", SCRIPT, ROOT], env=env, capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr[-2000:]
        return [int(x) for x in r.stdout.split()]

    known, launches, chosen = run()
    assert known == 0 and launches == 4 and chosen in (256, 512, 1024)
    key, kept = path.read_text().split()
    assert int(kept) == chosen
    other = 512 if chosen != 512 else 1024
    path.write_text(f"{key} {other}\n")
    assert run() == [other, 1, other]
