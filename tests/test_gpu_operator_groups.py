"""Operator passes on meshes that fill their element and face groups only partly.

Both passes take groups of 8 (small meshes: 2) elements, or faces of one direction, per CTA. 1331
elements leave 3 of 8 in the last group, 121 wall faces 1 of 8, 27 elements 1 of 2; k = 1..4 run every
pencil length. Against the oracle in FP64 at the bound of the other operator tests, 1e-12 relative:
the sums have at most a few hundred terms of comparable size, rounding 1e-16 each.
"""
import numpy as np
import pytest

import oracle as O
import synthetic as S
from _gpu_common import dev, host, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,walls", [(11, False), (11, True), (3, True)])
@pytest.mark.parametrize("k", [1, 2, 3, 4])
def test_partly_filled_groups(k, n, walls):
    import paper_1809_00866_gb300 as P
    xs = [S.perturbed_nodes(n, seed=s) for s in (1, 2, 3)]
    dg = P.DG(*xs, [k], S.NU_TGV, S.AC_C, S.ETA, walls=walls)
    m = O.Mesh(*xs, k, S.NU_TGV, S.AC_C, S.ETA, walls=walls)
    w = O.project_tgv(m) + S.perturbation(m.ne, k, 0.02, 4)
    v = S.direction(m.ne, k, 5)
    out = dg.empty()
    dg.dg_residual(dev(w), out)
    assert rel(host(out), O.residual(m, w)) < 1e-12
    dg.dg_set_linearization(dev(w), 0.7)
    dg.dg_jvp(dev(v), out)
    assert rel(host(out), O.jvp(m, w, v, 0.7)) < 1e-12
    assert np.isfinite(host(out)).all() and dg.dg_get_status() == 0
