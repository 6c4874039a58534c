"""Operator passes on meshes that fill their element and face groups only partly.

Both passes take groups of 8 (small meshes: 2 or 4) elements, or faces of one direction, per CTA. 1331
elements leave 3 of 8 in the last group (FP32: 3 of 4), 121 wall faces 1 of 8, 27 elements 1 of 2, 441
elements 1 of 4; k = 1..4 run every pencil length. Against the oracle in FP64 at the bound of the other operator tests, 1e-12 relative:
the sums have at most a few hundred terms of comparable size, rounding 1e-16 each.
"""
import numpy as np
import pytest

import oracle as O
import synthetic as S
from _gpu_common import dev, host, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,walls", [((11, 11, 11), False), ((11, 11, 11), True), ((3, 3, 3), True),
                                        ((7, 7, 9), True)])
@pytest.mark.parametrize("k", [1, 2, 3, 4])
def test_partly_filled_groups(k, dims, walls):
    import paper_1809_00866_gb300 as P
    xs = [S.perturbed_nodes(n, seed=s) for n, s in zip(dims, (1, 2, 3))]
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


@pytest.mark.parametrize("dims", [(3, 3, 3), (11, 11, 11), (13, 14, 15)])
@pytest.mark.parametrize("k", [2, 4])
def test_fp32_passes_in_groups(k, dims):
    """The FP32 passes (groups of 2, 4 and 8 elements) through a cycle, against the FP64 cycle: FP32
    roundoff 6e-8 times a condition number of 1e4 of the blocks, with a factor of three."""
    import paper_1809_00866_gb300 as P
    xs = [S.perturbed_nodes(n, seed=s) for n, s in zip(dims, (1, 2, 3))]
    dg = P.DG(*xs, [k, 1], S.NU_TGV, S.AC_C, S.ETA)
    w, a, b = dg.empty(), dg.empty(), dg.empty()
    dg.dg_project_tgv(w)
    w += dev(S.perturbation(dg.ne, k, 0.02, 4))
    dg.dg_set_linearization(w, 0.7)
    g = dev(S.direction(dg.ne, k, 5))
    for out, prec in ((a, P.DG_PRECOND_FP64), (b, P.DG_PRECOND_FP32)):
        dg.dg_assemble(precision=prec)
        dg.pmg_vcycle(g, out, P.solve_opts(pre_sweeps=1, post_sweeps=1, coarse_sweeps=1, omega=0.5, precision=prec))
    assert rel(host(b), host(a)) < 2e-3
    assert dg.dg_get_status() == 0
