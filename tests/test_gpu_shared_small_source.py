"""Shared factors and a tiny source.

With g = 0 the floating rows' part of r is linear in f's weights, so weights 2^-100 times as
large must give a part 2^-100 times as large, to the mixed form's accuracy (refinement to 1e-12; bar 1e-11
of the largest entry), however few bits FP32 leaves for it."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _lattice(m, n_knots, n_r, n_theta, op):
    cfg = workloads.tiny(paths=32, h=1e-3)
    s = 1.0 / m
    cfg["domain"] = {"kind": "square", "p": [0.0, 0.0, 1.0, 1.0]}
    cfg["cover"] = {"kind": "square_lattice", "nx": m, "ny": m, "x_origin": 0.5 * s, "y_origin": 0.5 * s,
                    "spacing": s, "radius": 0.8 * s}
    cfg |= {"n_knots": n_knots, "n_r": n_r, "n_theta": n_theta, "op": op}
    return cfg


def _floating_b(cfg, precision):
    import paper_2311_08946_gb300 as pdd

    cov = pdd.Cover(cfg)
    a = {k: v.cpu().numpy() for k, v in cov.arrays().items()}
    s = pdd.System(cov, cfg, precision)
    assert s.stats()["unconverged_disks"] == 0
    sub = a["row_sub"]
    rows = np.flatnonzero((sub >= 0) & (a["floating"][np.maximum(sub, 0)] != 0))
    return cov, s, a, rows


def test_tiny_source():
    op = {"b": "zero", "c": "zero", "f": "rbf", "g": "zero"}
    field = workloads.rbf_field(6, seed=6, sigma=0.25, domain={"kind": "square", "p": [0.0, 0.0, 1.0, 1.0]})
    out = []
    for scale in (1.0, 2.0 ** -100):
        cfg = _lattice(9, 12, 10, 20, dict(op, frbf=dict(field, w=scale * np.asarray(field["w"]))))
        _, s, _, rows = _floating_b(cfg, "mixed")
        assert s.stats()["floating_disks"] > 34
        out.append(s.csr()["b"].cpu().numpy()[rows] / scale)
    assert np.abs(out[0]).max() > 0
    assert np.abs(out[1] - out[0]).max() <= 1e-11 * np.abs(out[0]).max()
