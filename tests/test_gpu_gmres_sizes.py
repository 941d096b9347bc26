"""The fused Arnoldi kernel at the edges of its launch shapes: one row, fewer rows than a warp, one
cluster (up to 1,024 rows) and just beyond, restarts of 1 and 256 vectors, a basis that only partly fits
in shared memory, rows longer than the entries a lane group holds at once, and a right-hand side whose
Krylov space is exhausted at once.

A = I + E with |E|_inf <= 1/2, so kappa(A) <= 3 and a residual of 1e-12 |b| leaves the solution within
3e-12 of the direct one; the bar is ten times that."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _system(n, row, seed):
    import scipy.sparse as sp

    rng = np.random.default_rng(seed)
    k = min(row, n)
    cols = np.stack([rng.permutation(n)[:k] if n < 5000 else rng.integers(0, n, k) for _ in range(n)])
    E = sp.csr_matrix((rng.uniform(-0.5 / k, 0.5 / k, n * k), cols.ravel(), np.arange(0, n * k + 1, k)), shape=(n, n))
    E.sum_duplicates()
    A = (sp.eye(n, format="csr") + E).tocsr()
    A.sort_indices()
    return A, rng.standard_normal(n)


@pytest.mark.parametrize("n,row,restart,transpose", [
    (1, 1, 64, False), (7, 3, 1, False), (33, 9, 256, True), (257, 20, 5, False), (1000, 70, 64, False),
    (1024, 12, 64, True), (1025, 12, 64, False), (40000, 33, 256, False)])
def test_gmres_shapes_against_direct(n, row, restart, transpose):
    import scipy.sparse.linalg as spl

    import paper_2311_08946_gb300 as pdd

    A, b = _system(n, row, n)
    dev = lambda a, dt: torch.tensor(a, dtype=dt, device="cuda")
    u, info = pdd.solve_csr(dev(A.indptr, torch.int32), dev(A.indices, torch.int32), dev(A.data, torch.float64),
                            dev(b, torch.float64), rtol=1e-12, restart=restart, transpose=transpose)
    assert info["converged"]
    M = A.T.tocsr() if transpose else A
    if n <= 2000:
        x = np.linalg.solve(M.toarray(), b)
    else:                                    # the Neumann series, to rounding
        x, d = b.copy(), b.copy()
        for _ in range(80):
            d = d - M @ d
            x += d
            if np.linalg.norm(d) < 1e-17 * np.linalg.norm(x):
                break
    assert np.linalg.norm(u.cpu().numpy() - x) <= 3e-11 * np.linalg.norm(x)


def test_gmres_breakdown_and_zero():
    """b an eigenvector: the second Gram-Schmidt pass leaves nothing; b = 0: u = 0 without an iteration."""
    import paper_2311_08946_gb300 as pdd

    n = 3000
    dev = lambda a, dt: torch.tensor(a, dtype=dt, device="cuda")
    rp, ci = dev(np.arange(n + 1), torch.int32), dev(np.arange(n), torch.int32)
    va = dev(np.full(n, 3.0), torch.float64)
    b = dev(np.random.default_rng(0).standard_normal(n), torch.float64)
    u, info = pdd.solve_csr(rp, ci, va, b, rtol=1e-13)
    assert info["converged"] and info["iters"] <= 2
    assert torch.allclose(u, b / 3.0, rtol=1e-12, atol=0.0)
    u, info = pdd.solve_csr(rp, ci, va, torch.zeros_like(b), rtol=1e-13)
    assert info["converged"] and info["iters"] == 0 and not u.any()
