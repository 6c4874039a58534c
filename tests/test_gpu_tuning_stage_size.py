"""The autotuner and jacobi_stage_kb, the bytes per stage of the block-Jacobi apply's ring.

Only the ring reads it: FP32 blocks of k = 4, and blocks of k <= 3 under a cap on its CTAs. Elsewhere the
tuner leaves the field as it is set and reports the one time it measured; a result taken from the cache
leaves the cap and, there, the field as they are set, too.
"""
import pytest

import synthetic as S
from _gpu_common import dev

pytestmark = pytest.mark.gpu


def handle(k, storage, n=3):
    import paper_1809_00866_gb300 as P
    prec = getattr(P, "DG_PRECOND_" + storage)
    xs = [S.perturbed_nodes(n, seed=s) for s in (1, 2, 3)]
    dg = P.DG(*xs, [k, 1], S.NU_TGV, S.AC_C, S.ETA)
    w, g = dg.empty(), dg.empty()
    dg.dg_project_tgv(w)
    dg.dg_set_linearization(w, 0.7)
    dg.dg_assemble(precision=prec)
    dg.pmg_vcycle(dev(S.direction(dg.ne, k, 5)), g, P.solve_opts(precision=prec, omega=0.5))
    return P, dg


@pytest.mark.parametrize("k,storage,cap,read", [(2, "FP32", 0, False), (3, "FP32_H16", 0, False),
                                                (4, "FP32_H16", 0, False), (4, "FP32_BF16", 16, False),
                                                (4, "FP32", 0, True), (3, "FP32", 16, True), (2, "FP32_H16", 16, True)])
def test_stage_size_is_tuned_only_where_it_is_read(k, storage, cap, read):
    P, dg = handle(k, storage)
    dg.dg_set_tuning(P.DG_TUNE_FP32, jacobi_stage_kb=17, jacobi_max_ctas=cap)
    rep = dg.dg_autotune(P.DG_TUNE_FP32, use_cache=False)
    t = dg.dg_get_tuning(P.DG_TUNE_FP32).as_dict()
    assert t["jacobi_max_ctas"] == cap and rep["jacobi_chosen_ms"] > 0
    if read:
        assert t["jacobi_stage_kb"] in (48, 96, 144, 200)
    else:
        assert t["jacobi_stage_kb"] == 17 and rep["jacobi_chosen_ms"] == rep["jacobi_default_ms"]
    # another handle of the same shape, with its own field and cap, reuses the result
    _, d2 = handle(k, storage)
    d2.dg_set_tuning(P.DG_TUNE_FP32, jacobi_stage_kb=33, jacobi_max_ctas=cap)
    assert not any(d2.dg_autotune(P.DG_TUNE_FP32, use_cache=True).values())
    t2 = d2.dg_get_tuning(P.DG_TUNE_FP32).as_dict()
    assert t2 == dict(t, jacobi_stage_kb=t["jacobi_stage_kb"] if read else 33)
    # one under another cap does not take it over
    d2.dg_set_tuning(P.DG_TUNE_FP32, jacobi_max_ctas=cap + 5)
    d2.dg_autotune(P.DG_TUNE_FP32, use_cache=True)
    assert d2.dg_get_tuning(P.DG_TUNE_FP32).as_dict()["jacobi_max_ctas"] == cap + 5
