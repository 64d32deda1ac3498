"""The blocked elimination of the dense inverse at the edges of its panels (16 steps), of the rows
that a block of the panel's cluster holds, and of the update's tiles."""
import hashlib
import os
import subprocess
import sys

import numpy as np
import pytest

from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    from paper_0907_4863_gb300 import build
    build.build()
    from paper_0907_4863_gb300 import saamg
    return saamg


@pytest.mark.parametrize("kind", ["dominant", "permuted", "ties"])
@pytest.mark.parametrize("n", [3, 15, 16, 17, 33, 48, 255, 257, 511, 545])
def test_inverse_at_panel_edges(S, n, kind):
    """dominant: every pivot on the diagonal; permuted: a pivot row elsewhere at almost every step;
    ties: integer entries, several rows share the largest.  Condition numbers stay below 1e2, so
    the oracle's LU with partial pivoting and the inverse agree to 1e-12."""
    import torch
    rng = np.random.default_rng(100 + n)
    if kind == "ties":
        m = rng.integers(-1, 2, (n, n)) / (2.0 * n)
        m[np.arange(n), np.arange(n)] = 2.0
        m[(np.arange(n) + 1) % n, np.arange(n)] += 1.0
    else:
        m = rng.uniform(-1.0, 1.0, (n, n)) / n
        m[np.arange(n), np.arange(n)] = 2.0 + rng.uniform(0.0, 1.0, n)
    if kind != "dominant":
        m = m[rng.permutation(n)]
    m = np.ascontiguousarray(m)
    a = torch.from_numpy(m).cuda()
    inv = torch.full_like(a, float("nan"))
    S.dense_inverse(a, inv)
    assert np.array_equal(a.cpu().numpy(), m)
    inv = inv.cpu().numpy()
    b = rng.standard_normal((n, 2))
    for c in range(2):
        x = O.dense_lu_solve(m, b[:, c])
        assert np.linalg.norm(inv @ b[:, c] - x) <= 1e-12 * np.linalg.norm(x)


SIZES = [17, 48, 545, 1250, 2050]


def _digests(S):
    import torch
    out = []
    for n in SIZES:
        rng = np.random.default_rng(n)
        m = rng.uniform(-1.0, 1.0, (n, n)) / n
        m[np.arange(n), np.arange(n)] = 2.0 + rng.uniform(0.0, 1.0, n)
        a = torch.from_numpy(m[rng.permutation(n)]).cuda()
        inv = torch.empty_like(a)
        for _ in range(3):  # the buffers of one call are the next call's
            S.dense_inverse(a, inv)
            out.append(hashlib.sha256(inv.cpu().numpy().tobytes()).hexdigest())
    return out


def test_panels_beside_updates_give_the_bits_of_launches_in_turn(S):
    """The update of a panel runs beside the factorisation of the next one; without dependent
    launches every kernel starts after the one before it has ended."""
    code = ("from tests.test_gpu_dense_inverse_panels import _digests\n"
            "from paper_0907_4863_gb300 import saamg\nprint(' '.join(_digests(saamg)))")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    p = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True,
                       timeout=300, env=dict(os.environ, SAAMG_PDL="0"))
    assert p.returncode == 0, p.stderr
    assert p.stdout.split() == _digests(S)
