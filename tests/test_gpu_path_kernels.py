"""Mixed-form paths at the sizes where their kernels change or run ragged, against the FP64 form on the
same Philox streams: paths long enough for the resident-warp kernel (r^2 / 4h >= 500) and short ones,
fewer paths than a warp, chunks of 256 records that cross rows, odd numbers of Gaussians in c and f, and
more of them than are kept in shared memory.

A mixed path follows its FP64 twin to FP32 rounding, about 2e-6 after a thousand steps, unless one of
the two leaves a step earlier because its end point lies that near the boundary (2e-6 / sqrt(h), below
1e-2 of the paths); then the scores differ by a step's displacement, sqrt(h) <= 1e-2, times a gradient
below 3.  A row's mean over P paths therefore differs by less than 2 max(1e-2, 1 / P) 3e-2 + 1e-4."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _check(cfg, paths):
    import paper_2311_08946_gb300 as pdd

    cov = pdd.Cover(cfg)
    ref, got = pdd.System(cov, cfg, "fp64"), pdd.System(cov, cfg, "mixed")
    s, t = ref.stats(), got.stats()
    assert t["paths_total"] == s["paths_total"] and t["capped_paths"] == 0
    assert abs(t["path_steps"] - s["path_steps"]) <= 0.02 * s["path_steps"] + 2000
    d = (got.mc()["bmean"] - ref.mc()["bmean"]).abs().max().item()
    assert d <= 2 * max(1e-2, 1.0 / paths) * 3e-2 + 1e-4


@pytest.mark.parametrize("paths,h", [(2, 1e-5), (33, 1e-5), (300, 1e-5), (2, 1e-4), (300, 1e-4)])
def test_path_counts(paths, h):
    _check(workloads.tiny(paths=paths, h=h), paths)


@pytest.mark.parametrize("n_c,n_f,h", [(1, 1, 1e-4), (7, 3, 1e-4), (64, 16, 1e-5), (1025, 255, 1e-4)])
def test_gaussian_counts(n_c, n_f, h):
    cfg = workloads.grad(paths=64, h=h)
    box = cfg["domain"]
    cfg["op"]["rbf"] = workloads.rbf_field(n_c, seed=5, sigma=0.2, negative=True, domain=box)
    cfg["op"]["rbf"]["w"] /= max(1.0, n_c / 8.0)
    cfg["op"]["frbf"] = workloads.rbf_field(n_f, seed=6, sigma=0.25, domain=box)
    cfg["op"]["frbf"]["w"] /= max(1.0, n_f / 4.0)
    _check(cfg, 64)
