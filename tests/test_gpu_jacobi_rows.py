"""The block-Jacobi apply straight from memory against the ring of bulk copies.

Blocks of k <= 3 take the first unless a cap on the ring's CTAs is set; both multiply the same stored
inverses and differ by the order of FP32 sums of at most 80 terms, in each of about ten sweeps of the
cycle: 1e-4 leaves a condition number of ten for the difference to grow. Element counts that fill the
last CTA partly, one CTA, and several elements per CTA.
"""
import pytest

import synthetic as S
from _gpu_common import dev, host, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 3, 3), (5, 5, 5), (11, 11, 13)])
@pytest.mark.parametrize("storage", ["FP32", "FP32_H16", "FP32_BF16"])
def test_rows_match_ring(dims, storage):
    import paper_1809_00866_gb300 as P
    xs = [S.perturbed_nodes(n, seed=s) for n, s in zip(dims, (1, 2, 3))]
    dg = P.DG(*xs, [3, 2, 1], S.NU_TGV, S.AC_C, S.ETA)
    w, a, b = dg.empty(), dg.empty(), dg.empty()
    dg.dg_project_tgv(w)
    w += dev(S.perturbation(dg.ne, 3, 0.02, 4))
    dg.dg_set_linearization(w, 0.7)
    prec = getattr(P, "DG_PRECOND_" + storage)
    dg.dg_assemble(precision=prec)
    g = dev(S.direction(dg.ne, 3, 5))
    opts = P.solve_opts(precision=prec, omega=0.5, pre_sweeps=2, post_sweeps=1, coarse_sweeps=2)
    dg.pmg_vcycle(g, a, opts)
    dg.dg_set_tuning(P.DG_TUNE_FP32, jacobi_max_ctas=64)
    dg.pmg_vcycle(g, b, opts)
    assert rel(host(a), host(b)) < 1e-4
    assert dg.dg_get_status() == 0
