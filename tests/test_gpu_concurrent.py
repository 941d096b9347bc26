"""Two host threads on two streams, each with calls whose kernels take another amount of shared memory than
the other's: restarts 30 and 256 of the CSR solve, assemblies of few and of many disks and of small and large
grids, control variates of degree 1 and 4, gradients of few and of many parameters.  No call may fail, and
each must give what it gives alone (the sums of every kernel run in a fixed order; bar 1e-12)."""
import threading

import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu


def _solve(restart, diagonal):
    """A second difference of 3,000 rows with kappa = (diagonal + 2) / (diagonal - 2): several cycles."""
    import paper_2311_08946_gb300 as pdd

    n = 3000
    dev = lambda a, dt: torch.tensor(a, dtype=dt, device="cuda")
    col = np.sort((np.arange(n)[:, None] + np.array([-1, 0, 1])) % n, axis=1)
    val = np.where(col == np.arange(n)[:, None], diagonal, -1.0)
    args = (dev(3 * np.arange(n + 1), torch.int32), dev(col.ravel(), torch.int32), dev(val.ravel(), torch.float64),
            dev(np.random.default_rng(restart).standard_normal(n), torch.float64))
    return lambda: [pdd.solve_csr(*args, restart=restart)[0]]


def _assembly(precision, m, n_r, n_theta, n_knots, cv_degree=0):
    import paper_2311_08946_gb300 as pdd

    cfg = workloads.tiny(paths=64, h=1e-3)
    s = 1.0 / m
    cfg["domain"] = {"kind": "square", "p": [0.0, 0.0, 1.0, 1.0]}
    cfg["cover"] = {"kind": "square_lattice", "nx": m, "ny": m, "x_origin": 0.5 * s, "y_origin": 0.5 * s,
                    "spacing": s, "radius": 0.8 * s}
    cfg |= {"n_knots": n_knots, "n_r": n_r, "n_theta": n_theta}
    cfg["op"] = {"b": "sinx_cosy", "c": "quadratic", "f": "manufactured", "g": "sin_cos"}
    cfg["mc"] = dict(cfg["mc"], cv_degree=cv_degree)
    cov = pdd.Cover(cfg)
    return lambda: [pdd.System(cov, cfg, precision).csr()[k] for k in ("val", "b")]


def _gradient(n_c):
    import paper_2311_08946_gb300 as pdd

    cfg = workloads.grad(paths=64, h=1e-3)
    cfg["op"]["rbf"] = workloads.rbf_field(n_c, seed=5, sigma=0.2, negative=True, domain=cfg["domain"])
    sys_ = pdd.System(pdd.Cover(cfg), cfg, "fp64")
    u = sys_.solve()
    return lambda: [sys_.grad(u, u)]


PAIRS = {
    "restart": lambda: (_solve(30, 2.3), _solve(256, 2.005)),
    "fp64_disks": lambda: (_assembly("fp64", 4, 8, 16, 32), _assembly("fp64", 20, 8, 16, 32)),
    "mixed_disks": lambda: (_assembly("mixed", 4, 8, 16, 16), _assembly("mixed", 12, 20, 32, 24)),
    "control_variate": lambda: (_assembly("mixed", 4, 8, 16, 16, 1), _assembly("mixed", 4, 8, 16, 40, 4)),
    "gradient": lambda: (_gradient(3), _gradient(90)),
}


@pytest.mark.parametrize("pair,calls", [("restart", 100), ("fp64_disks", 40), ("mixed_disks", 40),
                                        ("control_variate", 40), ("gradient", 40)])
def test_two_threads(pair, calls):
    jobs = PAIRS[pair]()
    alone = [job() for job in jobs]
    torch.cuda.synchronize()
    errors, worst = [], [0.0, 0.0]
    start = threading.Barrier(2)

    def work(i):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                start.wait(60)
                for _ in range(calls):
                    out = jobs[i]()
                    for a, b in zip(out, alone[i]):
                        d = ((a - b).abs().max() / b.abs().max()).item()
                        worst[i] = max(worst[i], d) if d == d else float("inf")
        except Exception as e:                            # reported by the main thread
            errors.append(f"job {i}: {e}")

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    assert max(worst) <= 1e-12, worst
