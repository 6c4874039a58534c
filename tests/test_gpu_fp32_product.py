"""The FP32 Jacobian action of the cycle against the FP64 one, directly.

A two-level cycle of one pre-smoothing sweep from zero hands the coarse level d = I (g - G x1), x1 = omega D^-1 g,
formed by one FP32 product; dg_record_coarse gives d, and the same sweep of a one-level handle x1 itself.
The levels are k and k - 1, so that d holds every mode of degree <= k - 1. Against g - G x1 with the FP64 product.

Bound, per mode over the elements: an entry goes through at most about 60 FP32 operations one after
another (scaling, traces or gradients, interpolation, flux, projection, derivatives), 6e-8 each, and its terms may
exceed the result by a factor of 10: 4e-5, taken relative to the mode's own |G x1| + |g|.
Meshes that fill groups of 2, 4 and 8 elements only partly, with and without walls.
"""
import numpy as np
import pytest

import synthetic as S
from _gpu_common import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,walls", [((3, 3, 3), False), ((11, 11, 11), True), ((13, 14, 15), False)])
@pytest.mark.parametrize("k", [2, 3, 4])
def test_fp32_product_per_mode(k, dims, walls):
    import torch
    import paper_1809_00866_gb300 as P
    xs = [S.perturbed_nodes(n, seed=s) for n, s in zip(dims, (1, 2, 3))]
    two = P.DG(*xs, [k, k - 1], S.NU_TGV, S.AC_C, S.ETA, walls=walls)
    one = P.DG(*xs, [k], S.NU_TGV, S.AC_C, S.ETA, walls=walls)
    w, x1, z, Gx = (two.empty() for _ in range(4))
    two.dg_project_tgv(w)
    w += dev(S.perturbation(two.ne, k, 0.02, 4))
    g = dev(S.direction(two.ne, k, 5).astype(np.float32))
    opts = P.solve_opts(pre_sweeps=1, post_sweeps=0, coarse_sweeps=1, omega=0.5, precision=P.DG_PRECOND_FP32)
    for dg in (two, one):
        dg.dg_set_linearization(w, 0.7)
        dg.dg_assemble(precision=P.DG_PRECOND_FP32)
    one.pmg_vcycle(g, x1, opts)
    d = two.empty(1)
    two.dg_record_coarse(d)
    two.pmg_vcycle(g, z, opts)
    assert two.dg_recorded() == 1
    two.dg_jvp(x1, Gx)
    nc = d.shape[-1]
    got, gx, gg = (host(t)[..., :nc] for t in (d, Gx, g))
    err = np.sqrt(((got - (gg - gx)) ** 2).sum(0))
    scale = np.sqrt((gx ** 2).sum(0)) + np.sqrt((gg ** 2).sum(0))
    assert (err / scale).max() < 4e-5
    assert np.linalg.norm(gx) > 0.05 * np.linalg.norm(gg) and two.dg_get_status() == 0
    torch.cuda.synchronize()
