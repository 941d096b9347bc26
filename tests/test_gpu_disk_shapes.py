"""Disk grids at which the tiled disk kernels can go wrong, the mixed form against the FP64 form.

The two share neither the factorisation (pivot-free FP32 on the tensor cores / blocked FP64 with partial
pivoting, panels of 32, 16, 8 and 4 columns by n), nor the solves, nor the evaluation, nor the residuals
(angle pairs in tiles of 32 angles and 8 rings without drift; node by node with it).  Grids: fewer rings
than a tile and more, rings and angle halves that are no multiples, halves above 32, column counts that
leave ragged groups.  Bar: 1e-10 of each floating row, the one both forms meet against the oracle."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_r,n_theta,n_knots,drift", [
    (3, 4, 6, False), (13, 22, 10, False), (13, 22, 10, True), (20, 70, 16, False), (33, 50, 18, False),
    (32, 64, 20, True), (45, 64, 44, False), (48, 64, 16, True)])
def test_mixed_rows_match_fp64_rows(n_r, n_theta, n_knots, drift):
    import paper_2311_08946_gb300 as pdd

    cfg = workloads.tiny(paths=64)
    cfg["n_r"], cfg["n_theta"], cfg["n_knots"] = n_r, n_theta, n_knots
    if drift:
        cfg["op"] = {"b": "sinx_cosy", "c": "quadratic", "f": "manufactured", "g": "sin_cos"}
    cov = pdd.Cover(cfg)
    a = {k: v.cpu().numpy() for k, v in cov.arrays().items()}
    forms = [pdd.System(cov, cfg, p, path_precision="fp64") for p in ("fp64", "mixed")]
    ref, got = ({k: v.cpu().numpy() for k, v in s.csr().items()} for s in forms)
    assert forms[1].stats()["unconverged_disks"] == 0
    rows = [i for i in range(cov.N) if a["row_sub"][i] >= 0 and a["floating"][a["row_sub"][i]]]
    assert rows
    for i in rows:
        s = slice(a["rowptr"][i], a["rowptr"][i + 1])
        scale = np.linalg.norm(ref["val"][s])
        assert np.linalg.norm(got["val"][s] - ref["val"][s]) <= 1e-10 * scale, i
        assert abs(got["b"][i] - ref["b"][i]) <= 1e-10 * max(1.0, abs(ref["b"][i])), i


@pytest.mark.parametrize("n_knots", [6, 10, 16, 32])
def test_many_disks(n_knots):
    """More disks than SMs: the solves in groups of 8, 12 and 17 columns, two CTAs an SM."""
    import paper_2311_08946_gb300 as pdd

    m, s = 15, 0.25
    cfg = workloads.tiny(paths=32)
    cfg["domain"] = {"kind": "square", "p": [0.0, 0.0, m * s, m * s]}
    cfg["cover"] = {"kind": "square_lattice", "nx": m, "ny": m, "x_origin": s / 2, "y_origin": s / 2, "spacing": s,
                    "radius": 0.8 * s}
    cfg["n_r"], cfg["n_theta"], cfg["n_knots"] = 11, 20, n_knots
    cfg["op"] = {"b": "zero", "c": "quadratic", "f": "one", "g": "sin_cos"}
    cov = pdd.Cover(cfg)
    a = {k: v.cpu().numpy() for k, v in cov.arrays().items()}
    ref, got = (pdd.System(cov, cfg, p, path_precision="fp64") for p in ("fp64", "mixed"))
    assert got.stats()["floating_disks"] == (m - 2) ** 2 and got.stats()["unconverged_disks"] == 0
    g, r = ({k: v.cpu().numpy() for k, v in x.csr().items()} for x in (got, ref))
    for i in range(cov.N):
        if a["row_sub"][i] < 0 or not a["floating"][a["row_sub"][i]]:
            continue
        e = slice(a["rowptr"][i], a["rowptr"][i + 1])
        assert np.linalg.norm(g["val"][e] - r["val"][e]) <= 1e-10 * np.linalg.norm(r["val"][e]), i
        assert abs(g["b"][i] - r["b"][i]) <= 1e-10 * max(1.0, abs(r["b"][i])), i
