"""The assembled blocks against the operator they come from, at every degree.

Diagonal blocks: for x with support on one element e, the rows e of G x are D_e x_e, and one
block-Jacobi sweep from zero must return x_e; the bound 1e-8 leaves a condition number of 1e6 for
the LU solution in FP64. Level-1 block rows: they are the restriction of G, so that on coarse
vectors I G I^T and the block-sparse product agree to rounding, 1e-12 as in the other operator tests.
FP32 assembly: a cycle of one block-Jacobi sweep per level, with explicit inverses, against the same
cycle in FP64 at 2e-3, the bound of a condition number of 1e4 times the FP32 roundoff 6e-8 with a
factor of three. Two-element boxes have one neighbour across two faces, walls a one-sided Jacobian.
"""
import numpy as np
import pytest

import synthetic as S
from _gpu_common import dev, host, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,walls", [((2, 3, 3), False), ((3, 2, 4), True), ((3, 3, 2), False)])
@pytest.mark.parametrize("levels", [[1], [2, 1], [3, 1], [3, 2, 1], [4, 3], [4, 2, 1]])
def test_blocks_match_operator(levels, dims, walls):
    import paper_1809_00866_gb300 as P
    xs = [S.perturbed_nodes(n, seed=s) for n, s in zip(dims, (1, 2, 3))]
    k = levels[0]
    dg = P.DG(*xs, levels, S.NU_TGV, S.AC_C, S.ETA, walls=walls)
    w, t = dg.empty(), dg.empty()
    dg.dg_project_tgv(w)
    w += dev(S.perturbation(dg.ne, k, 0.02, 4))
    dg.dg_set_linearization(w, 0.7)
    dg.dg_assemble()
    v = S.direction(dg.ne, k, 5)
    for e in range(0, dg.ne, 5):
        x = np.zeros_like(v)
        x[e] = v[e]
        dg.dg_jvp(dev(x), t)
        g = np.zeros_like(v)
        g[e] = host(t)[e]
        y = dg.empty()
        y.zero_()
        dg.block_jacobi_smooth(0, dev(g), y, 1, 1.0)
        assert rel(host(y)[e], v[e]) < 1e-8
    if len(levels) > 1:
        xc = dev(S.direction(dg.ne, levels[1], 6))
        f, yc, zc = dg.empty(), dg.empty(1), dg.empty(1)
        f.zero_()
        dg.pmg_prolong(0, xc, f)
        dg.dg_jvp(f, t)
        dg.pmg_restrict(0, t, yc)
        dg.bsr_spmv(1, 1.0, xc, 0.0, zc)
        assert rel(host(zc), host(yc)) < 1e-12
    o64 = P.solve_opts(pre_sweeps=1, post_sweeps=1, coarse_sweeps=1, omega=0.5)
    o32 = P.solve_opts(pre_sweeps=1, post_sweeps=1, coarse_sweeps=1, omega=0.5, precision=P.DG_PRECOND_FP32)
    a, b = dg.empty(), dg.empty()
    dg.pmg_vcycle(dev(v), a, o64)
    dg.dg_assemble(precision=P.DG_PRECOND_FP32)
    dg.pmg_vcycle(dev(v), b, o32)
    assert rel(host(b), host(a)) < 2e-3
    assert dg.dg_get_status() == 0
