"""Row owners, rows by circle and the duplicate test where circles are uneven: a large circle among
small ones owns more rows than a sorting CTA has threads, and a far-away origin leaves FP32 few digits
for the distance test.  Integers, so equal."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _uneven(ox, oy):
    """Small circles on a lattice, and large ones over them with many more knots."""
    x, y = np.meshgrid((np.arange(20) + 0.5) * 0.1, (np.arange(20) + 0.5) * 0.1)
    big = np.array([[0.53, 0.57], [1.41, 0.63], [0.61, 1.37], [1.43, 1.47]])
    cx = np.concatenate([x.ravel(), big[:, 0]]) + ox
    cy = np.concatenate([y.ravel(), big[:, 1]]) + oy
    r = np.concatenate([np.full(400, 0.09), np.full(4, 0.52)])
    n = np.concatenate([np.full(400, 12), np.full(4, 40)]).astype(np.int32)
    return {"name": "uneven", "domain": {"kind": "square", "p": [ox, oy, ox + 2.0, oy + 2.0]},
            "cover": {"kind": "explicit", "cx": cx, "cy": cy, "r": r, "n_knots": n,
                      "n_r": np.full(404, 8, np.int32), "n_theta": np.full(404, 8, np.int32)},
            "n_knots": 0, "n_r": 0, "n_theta": 0, "op": {"b": "zero", "c": "zero", "f": "zero", "g": "exp_sin"},
            "mc": {"paths": 64, "h": 1e-4, "seed": 0}, "imq_c2": 1.5}


@pytest.mark.parametrize("ox,oy", [(0.0, 0.0), (-3.0e4, 7.0e3)])
def test_uneven_cover_matches_oracle(ox, oy):
    import paper_2311_08946_gb300 as pdd
    from oracle import cover as ocover

    cfg = _uneven(ox, oy)
    oc = ocover.full_cover(cfg)
    a = {k: v.cpu().numpy() for k, v in pdd.Cover(cfg).arrays().items()}
    for k in ("knot_ptr", "kowner", "row_sub", "rowptr", "col"):
        assert np.array_equal(a[k].astype(np.int64), getattr(oc, k).astype(np.int64)), k
    assert np.bincount(a["row_sub"][a["row_sub"] >= 0]).max() > 256


def test_coinciding_knots_are_refused():
    """Two equal circles: every knot coincides with another, at cells' edges and inside them."""
    import paper_2311_08946_gb300 as pdd

    cfg = _uneven(0.0, 0.0)
    c = cfg["cover"]
    for k in ("cx", "cy", "r", "n_knots", "n_r", "n_theta"):
        c[k] = np.concatenate([c[k], c[k][210:211]])
    with pytest.raises(pdd.PddError) as e:
        pdd.Cover(cfg)
    assert e.value.code == "PDD_EDUPLICATE_KNOT"
