"""Which organisation a subtracted-real call runs is a rule on its arguments (CPU; no GPU
needed): the automatic choice takes the per-term queues for mixed-precision batches between 2^19
points and the queues' limit of 2^29 - 1, for e+e- -> u ubar g only with cuts; above the limit the masked
evaluation takes the call."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def rule():
    from paper_2503_07439_gb300 import build
    import paper_2503_07439_gb300 as me
    f = ctypes.CDLL(build.build()).me_internal_term_queues
    f.restype, f.argtypes = ctypes.c_int, [ctypes.c_char_p, ctypes.c_void_p, ctypes.c_int64]

    def run(name, n, **kw):
        p = me.default_params(**{"precision": me.ME_PREC_MIXED, **kw})
        return f(name.encode(), ctypes.byref(p), n)

    run.me = me
    return run


CUTS = {"ee_uug": [dict(cut_abs_cos_axis_max=0.8), dict(cut_thrust_max=0.9)], "gg_ttg": [{}, dict(cut_pt_min=50.0)],
        "uu_ttg": [{}, dict(cut_abs_y_max=2.0)]}


@pytest.mark.parametrize("name,cuts", [(k, c) for k, v in CUTS.items() for c in v])
def test_automatic_range(rule, name, cuts):
    lo, hi = 1 << 19, 1 << 29
    assert [rule(name, n, **cuts) for n in (1, lo - 1, lo, hi - 1, hi, (1 << 31) - 1)] == [0, 0, 1, 1, 0, 0]
    me = rule.me
    for kw in (dict(precision=me.ME_PREC_FP64), dict(queued_rescue=1), dict(rescue=me.ME_RESCUE_POINTS)):
        assert rule(name, lo, **cuts, **kw) == 0


def test_without_cuts_and_fixed_choices(rule):
    me = rule.me
    for n in (1 << 19, 1 << 24):
        assert rule("ee_uug", n) == 0
        assert rule("ee_uug", n, cut_pt_min=50.0) == 0  # a cut of the other processes
    for name in CUTS:
        for n in (1, 1 << 20, 1 << 29):
            assert rule(name, n, term_queues=me.ME_TERMS_QUEUED) == 1
            assert rule(name, n, term_queues=me.ME_TERMS_MASKED) == 0
    assert rule("gg_tt", 1 << 20) == -1 and rule("none", 1) == -1
