"""Adjoint gradients at parameter and path counts that do not divide the replay kernel's groups
(four lanes per path, 128 threads, parts of a row), against the FP64 oracle.

Bar: 1e-8 of the largest entry, the one the full-size adjoint test meets (GMRES at 1e-14, kappa(C)
and the interpolation matrices' rounding)."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_c,n_f,n_g,paths", [(1, 1, 2, 2), (5, 3, 7, 65), (66, 17, 33, 300)])
def test_gradient_at_ragged_sizes(n_c, n_f, n_g, paths):
    import paper_2311_08946_gb300 as pdd
    from oracle import adjoint as oadj
    from oracle import cover as ocover
    from oracle import krylov as okrylov
    from oracle import system as osystem

    cfg = workloads.grad(paths=paths)
    box = cfg["domain"]
    cfg["op"]["rbf"] = workloads.rbf_field(n_c, seed=5, sigma=0.2, negative=True, domain=box)
    cfg["op"]["frbf"] = workloads.rbf_field(n_f, seed=6, sigma=0.25, domain=box)
    cfg["op"]["g_coef"] = np.random.default_rng(7).standard_normal(n_g)
    oc = ocover.full_cover(cfg)
    S = pdd.System(pdd.Cover(cfg), cfg, "fp64")
    u = S.solve(rtol=1e-14)
    u_obs = np.cos(oc.kx + oc.ky)
    g = S.grad(u, 2.0 * (u - torch.tensor(u_obs, device="cuda"))).cpu().numpy()
    ref = osystem.assemble(cfg, oc, with_grad=True)
    uo = okrylov.solve(ref.csr(), ref.b)
    gw, ga, _, gf = oadj.gradient(cfg, ref, uo, 2.0 * (uo - u_obs))
    want = np.concatenate([gw, gf, ga])
    assert g.shape == want.shape
    assert np.abs(g - want).max() <= 1e-8 * np.abs(want).max()
