"""The Schur decomposition where its kernels change form: window sizes up to and
past the number of bulges, sizes on both sides of what fits in a cluster's
shared memory (the reduction up to n = 654, the sweeps up to 448), and matrices
whose trailing blocks give poor shifts (graded, cyclic, orthogonal, symmetric, of
low rank).  The tolerance is that of the decomposition's other tests: about
2 n^2 rotations, each a few roundings, reach an entry in ~n steps of random
sign, well below 50 n eps normwise."""
import numpy as np
import pytest

from paper_1607_06303_gb300.inputs import make_A

pytestmark = pytest.mark.gpu


def _check(p, A):
    import torch
    Qt, Tt = p.schur(p.to_device(np.asfortranarray(A)))
    torch.cuda.synchronize()
    Q, T = p.to_numpy(Qt), p.to_numpy(Tt)
    n, eps = A.shape[0], np.finfo(float).eps
    assert np.all(np.tril(T, -1) == 0)
    assert np.linalg.norm(Q.conj().T @ Q - np.eye(n)) <= 50 * n * eps
    assert np.linalg.norm(Q @ T @ Q.conj().T - A) <= 50 * n * eps * np.linalg.norm(A)


@pytest.mark.parametrize("n", list(range(2, 14)) + [28, 29, 30, 31, 32, 33, 61, 65, 129, 448, 449, 654, 655])
def test_schur_sizes(gpu_lib, n):
    _check(gpu_lib, make_A(n, seed=n))


@pytest.mark.parametrize("n", [31, 120])
@pytest.mark.parametrize("kind", ["rows", "both", "huge", "tiny", "cyclic", "orthogonal", "symmetric", "rank", "band"])
def test_schur_hard_shifts(gpu_lib, n, kind):
    rng = np.random.Generator(np.random.PCG64(n))
    A = rng.standard_normal((n, n))
    if kind == "rows":
        A *= 10.0 ** rng.uniform(-8.0, 8.0, n)[:, None]
    elif kind == "both":
        g = np.logspace(6, -6, n)
        A *= g[:, None] * g[None, :]
    elif kind in ("huge", "tiny"):
        A = np.ldexp(A, 300 if kind == "huge" else -300)
    elif kind == "cyclic":
        A = np.roll(np.eye(n), 1, axis=0)
    elif kind == "orthogonal":
        A = np.linalg.qr(A)[0]
    elif kind == "symmetric":
        A = A + A.T
    elif kind == "rank":
        A = A[:, :5] @ A[:5, :]
    elif kind == "band":
        A = np.eye(n) + np.diag(np.ones(n - 1), 1) + 1e-3 * np.diag(np.ones(n - 1), -1)
    _check(gpu_lib, A)
