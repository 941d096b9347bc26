"""A solve whose right-hand side or matrix holds a NaN or an infinity, or whose right-hand side's norm
overflows, has no residual to meet: it ends with PDD_ENOCONV after the first cycle (a cycle and its
residual are below 20 launches), never with PDD_OK.  (b = 0 has the solution 0 whatever C holds.)"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [40, 3000])
@pytest.mark.parametrize("noalloc", [False, True])
@pytest.mark.parametrize("where,value", [("b", float("nan")), ("b", float("inf")), ("b", 1e200),
                                         ("val", float("nan")), ("val", float("inf"))])
def test_not_reported_as_solved(n, noalloc, where, value):
    import paper_2311_08946_gb300 as pdd

    dev = lambda a, dt: torch.tensor(a, dtype=dt, device="cuda")
    col = (np.arange(n)[:, None] + np.array([0, 1, 5])) % n
    val = np.tile([2.0, 0.3, -0.4], (n, 1))
    b = np.random.default_rng(0).standard_normal(n)
    {"b": b, "val": val.reshape(-1)}[where][n // 2] = value
    args = (dev(3 * np.arange(n + 1), torch.int32), dev(col.ravel(), torch.int32), dev(val.ravel(), torch.float64),
            dev(b, torch.float64))
    before = pdd.launch_count()
    with pytest.raises(pdd.PddError) as e:
        if noalloc:
            pdd.solve_csr_noalloc(*args, torch.empty(n, dtype=torch.float64, device="cuda"))
        else:
            pdd.solve_csr(*args)
    assert e.value.code == "PDD_ENOCONV"
    assert pdd.launch_count() - before < 20


def test_zero_right_hand_side_needs_no_matrix():
    import paper_2311_08946_gb300 as pdd

    i = torch.arange(41, dtype=torch.int32, device="cuda")
    u, info = pdd.solve_csr(i, i[:40].clone(), torch.full((40,), float("nan"), dtype=torch.float64, device="cuda"),
                            torch.zeros(40, dtype=torch.float64, device="cuda"))
    assert info["converged"] and info["iters"] == 0 and not u.any()
