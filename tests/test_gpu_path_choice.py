"""The mixed form's path kernel is chosen by the mean of r^2 / 4h over the Monte Carlo rows (resident warps,
three launches a wave, from 500 on; one CTA a row, one launch, below): a large floating circle, which walks
no path, does not count.  An 8 x 8 lattice of radius 0.1 and a circle of radius 0.3 inside it: r^2 / 4h is
2,500 h0/h on the lattice and 22,500 h0/h in the middle, h0 = 1e-6."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _launches(h):
    import paper_2311_08946_gb300 as pdd

    cfg = workloads.tiny(paths=32, h=h)
    x, y = (a.ravel() for a in np.meshgrid((np.arange(8) + 0.5) / 8, (np.arange(8) + 0.5) / 8))
    n = x.size + 1
    cfg["domain"] = {"kind": "square", "p": [0.0, 0.0, 1.0, 1.0]}
    cfg["cover"] = {"kind": "explicit", "cx": np.append(x, 0.507), "cy": np.append(y, 0.493),
                    "r": np.append(np.full(n - 1, 0.1), 0.3), "n_knots": np.full(n, 8, np.int32),
                    "n_r": np.full(n, 8, np.int32), "n_theta": np.full(n, 16, np.int32)}
    cfg |= {"n_knots": 0, "n_r": 0, "n_theta": 0}
    cov = pdd.Cover(cfg)
    a = cov.arrays()
    assert a["floating"][-1] and (a["row_sub"] == n - 1).any()
    pdd.System(cov, cfg, "mixed")                         # (first-use work is done)
    before = pdd.launch_count()
    pdd.System(cov, cfg, "mixed")
    return pdd.launch_count() - before


def test_floating_circles_do_not_choose():
    short = _launches(2e-4)                               # 12.5 steps; 112 in the middle
    assert _launches(1e-5) == short                       # 250; 2,250 in the middle
    assert _launches(1e-6) == short + 2                   # 2,500
