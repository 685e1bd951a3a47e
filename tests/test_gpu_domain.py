"""Points without a direction have no subtracted weight (GPU).

A three-momentum with a NaN, or one whose square underflows, has no direction: like the other
points outside the FKS domain it gets weight 0, in every precision and organisation, whatever the
sign bit of the NaN, and the points around it and the accumulators keep their values."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def me():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2503_07439_gb300 as m
    return m


# the legs whose directions define the sectors: the gluon and its partners, or the beams
LEGS = {"ee_uug": (4, 2, 3), "gg_ttg": (4, 0, 1), "uu_ttg": (4, 0, 1)}


@pytest.mark.parametrize("queues", [0, 1])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("name", list(LEGS))
def test_points_without_a_direction(me, name, prec, queues):
    p = synth.flat_points(name, 64, 61).p
    kw = dict(precision=me.ME_PREC_FP64 if prec == "fp64" else me.ME_PREC_MIXED, lanes_per_event=1, term_queues=queues)
    ref = me.Handle(name, **kw).real_subtracted(torch.from_numpy(p).cuda()).cpu().numpy()
    assert np.all(np.isfinite(ref)) and np.all(ref != 0.0)
    bad = np.zeros(64, bool)
    nans = np.array([0x7FF8000000000000, 0xFFF8000000000000], np.uint64).view(np.float64)
    i = 1
    for leg in LEGS[name]:
        for c in (1, 2, 3):
            for x in nans:
                p[c, leg, i], bad[i] = x, True
                i += 2
        p[1:, leg, i], bad[i] = [1e-170, -2e-170, 3e-170], True  # the square is 0
        i += 2
    h = me.Handle(name, **kw)
    got = h.real_subtracted(torch.from_numpy(p).cuda()).cpu().numpy()
    np.testing.assert_array_equal(got[bad], 0.0)
    np.testing.assert_array_equal(got[~bad], ref[~bad])
    np.testing.assert_allclose(h.accumulators()[:2], [ref[~bad].sum(), (ref[~bad] ** 2).sum()], rtol=1e-12)
